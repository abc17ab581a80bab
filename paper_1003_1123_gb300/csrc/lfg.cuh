// Additive Lagged Fibonacci generator shared by all threads (Algorithm 3):
//   x_p = x_{p-ll} + x_{p-D}  mod 2^32,   D = ll - sl.
//
// Fan.  Since ll = D + sl, the values D apart that a fan holds,
//   x_p, x_{p+D}, ..., x_{p+(K-1)D},
// follow from the K + 1 words b_i = x_{p-D-i sl} (i = 0 .. K) alone: with
// a_i <- a_i + a_{i+1} applied to the row, a_0 is x_p after one application,
// x_{p+D} after two, and so on (a_i after k + 1 applications is x_{p+kD-i sl}:
// the recurrence at that index).  So one thread turns K + 1 loads into K values
// with K (K + 1) / 2 additions, and the K D positions from U on are the fans at
// p = U + o, o < D, which read only positions below U.  Against computing each
// value from the leap form x_p = sum_j C(k, j) x_{p-(k-j)ll-jD} this is (K + 1) / K
// instead of k + 1 loads a value at the same distance from the nearest
// dependency.
//
// The fans of a round read back to U - H, H = D + K sl, and rely on the
// recurrence from U - (K - 1) sl on.  The seeds x_{-ll..-1} are extended
// backwards with the recurrence run in reverse, x_q = x_{q+ll} - x_{q+sl}, down
// to x_{-H}, which makes it hold there from position 0 on.
//
// Ring.  Position p lives in slot p mod R; slot arithmetic is 32-bit: an offset
// below R is added with one conditional subtraction of R.  R is a multiple of 32
// and at least 3 K D (and K D + H): while a round's values are used, the next
// round's are written and the one after that may have been begun.
//
// Rounds.  A launch walks its positions in rounds of W <= K D.  A persistent
// cooperative grid, one CTA a SM, generates round r + 1 while it uses round r
// (the Langevin steps), with warps of its own for each; a grid barrier separates
// the rounds.  The CTA arrives at it as soon as its share of round r + 1 is stored,
// so the barrier's latency (1.3 us) passes behind the use of round r.  An extra
// warp does the waiting, bounded by %globaltimer; a wait that runs out records
// GBRNG_ETIMEOUT and every CTA returns.
//
// K goes by the Table I row, the deepest of 2, 4, 8, 16 with K D <= 4.1e6 (the
// last row 2, rows 0 to 6 16): small rows get the most positions, and so steps, a
// round.
#pragma once

#include <algorithm>
#include <type_traits>

#include "device.cuh"
#include "internal.cuh"

namespace gb {

struct LfgArgs {
    uint32_t* ring;        // R words
    uint32_t R;            // ring slots
    uint32_t D, sl;        // ll - sl, sl
    uint32_t back[17];     // (D + i sl) mod R: from x_p's slot back to its fan's b_i
    uint32_t ahead[16];    // k D mod R: to the fan's k-th value
    uint32_t base_slot;    // slot of position `base`
    int64_t n_pos;         // positions of this launch
    int w;                 // round width (positions)
    int64_t N;             // oscillators (particles)
    int64_t n_steps;       // steps (equilibrium start: 2)
    void* out;
    float* x;
    float* v;
    const float* Kper;
    LdCoef c;
    uint64_t* arrive;      // grid-barrier arrival counter (zeroed before launch; 64-bit, never wraps)
    int* status;           // beside it: set when a wait has run out
    int* host_status;      // the same for the host (mapped)
    uint64_t wait_ns;
    StatsSink sink;
    int stall_cta;         // test hook: this CTA never arrives (-1: none)
    bool vec;              // every quad of words that is read together starts on a multiple of 4
};

// s + o mod R and s - o mod R for s, o < R (R < 2^31): of the sum and the sum less
// R (the difference and the difference plus R), the one that has not wrapped below
// zero is the smaller.
__host__ __device__ __forceinline__ uint32_t slot_add(uint32_t s, uint32_t o, uint32_t R)
{
    const uint32_t r = s + o, q = r - R;
    return q < r ? q : r;
}
__host__ __device__ __forceinline__ uint32_t slot_sub(uint32_t s, uint32_t o, uint32_t R)
{
    const uint32_t r = s - o, q = r + R;
    return q < r ? q : r;
}

// Slot of position p (p >= -R).
inline uint32_t slot_of(int64_t p, uint32_t R)
{
    const int64_t r = p % (int64_t)R;
    return (uint32_t)(r < 0 ? r + R : r);
}

// ---------------------------------------------------------------- barriers
// One thread's part of the grid barrier: adds the CTA's arrival with release
// semantics (the CTA's threads have met before, so it publishes all their writes)
// and polls the counter until `target` CTAs have arrived.  Every arrival is an
// atomic add to the counter, so the acquire read that ends the poll lies in each
// arrival's release sequence and synchronises with all of them.  The poll is
// bounded by a %globaltimer deadline and stops early when another CTA has
// recorded a failure.
__device__ inline bool barrier_thread(const LfgArgs& a, uint64_t target, bool arrive_here)
{
    if (arrive_here) red_release_add_u64(a.arrive, 1ull);
    const uint64_t deadline = global_ns() + a.wait_ns;
    for (uint32_t n = 1; ld_acquire_u64(a.arrive) < target; ++n) {
        if ((n & 15u) == 0) {
            if (ld_volatile_i32(a.status) != DEV_OK) return false;
            if (global_ns() > deadline) {
                if (atomicCAS(a.status, DEV_OK, DEV_TIMEOUT) == DEV_OK) {
                    *(volatile int*)a.host_status = DEV_TIMEOUT;
                    __threadfence_system();
                }
                return false;
            }
        }
    }
    return true;
}

// The warps of a CTA.  Generating warps arrive at BAR_STORED when the CTA's share
// of round r is stored; the waiting warp meets them there, takes the CTA through
// the grid barrier and meets every warp at BAR_GO: the using warps, which then use
// round r, and the generating ones, which then generate round r + 1.  A using warp
// comes to BAR_GO with round r - 1 used, so the arrival that follows says that the
// CTA is done with it: R >= 3 W keeps it until then.
//
// A wait that ran out is told by its round (kNoRound: none did).  Past BAR_GO of
// round r the waiting warp needs only the generating warps to be in round r + 1, and
// to fail there; a using warp that looks late must not leave for that before BAR_GO of
// round r + 1, which counts on it.  So warps leave by round_failed(r), the same for all.
constexpr int64_t kNoRound = INT64_MAX;
__device__ __forceinline__ bool round_failed(const int64_t* failed, int64_t r)
{
    return *(volatile const int64_t*)failed <= r;
}
enum { BAR_STORED = 1, BAR_GO = 2 };

// The waiting warp: one barrier for each of `count` rounds, `stored` threads at
// BAR_STORED and `threads` at BAR_GO.
__device__ __forceinline__ void wait_warp(const LfgArgs& a, int64_t count, int stored, int threads, int64_t* failed)
{
    const bool arrive_here = (int)blockIdx.x != a.stall_cta;
    for (int64_t r = 0; r < count; ++r) {
        bar_sync(BAR_STORED, stored);
        int ok = 1;
        if ((threadIdx.x & 31) == 0) {
            ok = barrier_thread(a, (uint64_t)gridDim.x * (uint64_t)(r + 1), arrive_here);
            if (!ok) *(volatile int64_t*)failed = r;
        }
        ok = __shfl_sync(0xffffffffu, ok, 0);
        bar_sync(BAR_GO, threads);
        if (!ok) return;
    }
}

// -------------------------------------------------------------------- fans
// A warp's unit: the fans of 32 J consecutive offsets o of a round; lane l holds
// those of o = o0 + 32 j + l.  J has 15 to 18 loads in flight, and the slots' arithmetic
// shared by as many values as the registers of 1024 threads take (1e6 oscillators, K = 2:
// 7.08 us a step; J = 4 with the next unit's loads issued before a unit's stores 7.40,
// without 7.16; J = 8 7.07, but uniform fills 462 us against 432; J = 12 7.29).
template <int K>
__host__ __device__ constexpr int fan_j() { return K <= 2 ? 6 : K == 4 ? 3 : K == 8 ? 2 : 1; }
template <int K>
__host__ __device__ constexpr int fan_offsets() { return 32 * fan_j<K>(); }

template <int K>
struct Fan {
    uint32_t b[fan_j<K>()][K + 1];
    uint32_t s;   // slot of x_{U + o0}; J = 1: of x_{U + o0 + lane}
    int o0;
    bool plain;   // no window and no store crosses the ring's end
};

// Issue the loads of the unit at offset o0 whose first value goes to slot s; kept:
// this lane's b_0 (32 words apart) where they are still on chip, or null.  With J =
// 1 every lane wraps its own slots; else the unit's windows are contiguous unless
// one crosses the ring's end.
template <int K>
__device__ __forceinline__ void fan_load(const LfgArgs& a, uint32_t s, int o0, Fan<K>& f,
                                         const uint32_t* kept = nullptr)
{
    constexpr int J = fan_j<K>();
    const int lane = threadIdx.x & 31;
    f.o0 = o0;
    if constexpr (J == 1) {
        f.s = slot_add(s, lane, a.R);
#pragma unroll
        for (int i = 0; i <= K; ++i)
            if (i > 0 || !kept) f.b[0][i] = __ldcg(a.ring + slot_sub(f.s, a.back[i], a.R));
    } else {
        f.s = s;
        uint32_t w[K + 1], most = s;
#pragma unroll
        for (int i = 0; i <= K; ++i) w[i] = slot_sub(s, a.back[i], a.R), most = max(most, w[i]);
#pragma unroll
        for (int k = 1; k < K; ++k) most = max(most, slot_add(s, a.ahead[k], a.R));
        f.plain = most <= a.R - 32 * J;
        if (f.plain) {
#pragma unroll
            for (int i = 0; i <= K; ++i) {
                if (i == 0 && kept) continue;
                const uint32_t* p = a.ring + w[i] + lane;
#pragma unroll
                for (int j = 0; j < J; ++j) f.b[j][i] = __ldcg(p + 32 * j);
            }
        } else {
#pragma unroll
            for (int i = 0; i <= K; ++i) {
                if (i == 0 && kept) continue;
#pragma unroll
                for (int j = 0; j < J; ++j) f.b[j][i] = __ldcg(a.ring + slot_add(w[i], 32 * j + lane, a.R));
            }
        }
    }
    if (kept)
#pragma unroll
        for (int j = 0; j < J; ++j) f.b[j][0] = kept[32 * j];
}

// The unit's values to the ring, those of offsets below n_off and positions below
// n (of the round); each also to use(k, j, value).
template <int K, class F>
__device__ __forceinline__ void fan_store(const LfgArgs& a, int n_off, int n, Fan<K>& f, F&& use)
{
    constexpr int J = fan_j<K>();
    const int lane = threadIdx.x & 31;
    const bool whole = (J == 1 || f.plain) && f.o0 + 32 * J <= n_off && f.o0 + 32 * J + (K - 1) * (int)a.D <= n;
#pragma unroll
    for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int j = 0; j < J; ++j) {
#pragma unroll
            for (int i = 0; i < K - k; ++i) f.b[j][i] += f.b[j][i + 1];
            use(k, j, f.b[j][0]);
        }
        const uint32_t s = slot_add(f.s, a.ahead[k], a.R);
        if (whole) {
            uint32_t* p = a.ring + s + (J == 1 ? 0 : lane);
#pragma unroll
            for (int j = 0; j < J; ++j) __stcg(p + 32 * j, f.b[j][0]);
        } else {
            const int at = f.o0 + k * (int)a.D;   // the fan's position in the round
#pragma unroll
            for (int j = 0; j < J; ++j) {
                const int e = 32 * j + lane;
                if (f.o0 + e < n_off && at + e < n)
                    __stcg(a.ring + slot_add(s, J == 1 ? 0 : e, a.R), f.b[j][0]);
            }
        }
    }
}

// The generating warps (0 .. GW - 1 of them): every round's fans, each CTA a
// contiguous share, a warp every GW-th unit of it.
template <int K, int GW>
__device__ __forceinline__ void gen_warps(const LfgArgs& a, int warp, int64_t n_rounds, int threads,
                                          const int64_t* failed)
{
    constexpr int FO = fan_offsets<K>();
    uint32_t s_round = a.base_slot;
    const int64_t last = n_rounds - 1;
    int g0 = 0, g1 = 0, n = 0, n_off = 0;
    for (int64_t r = 0; r < n_rounds; ++r) {
        if (r == 0 || r == last) {
            n = r == last ? (int)(a.n_pos - r * a.w) : a.w;
            n_off = min((int)a.D, n);
            const unsigned units = (unsigned)(n_off + FO - 1) / FO;   // units x CTAs < 2^31
            g0 = (int)(blockIdx.x * units / gridDim.x);
            g1 = (int)((blockIdx.x + 1) * units / gridDim.x);
        }
        Fan<K> f;
#pragma unroll 1
        for (int g = g0 + warp; g < g1; g += GW) {
            fan_load<K>(a, slot_add(s_round, (uint32_t)(g * FO), a.R), g * FO, f);
            fan_store<K>(a, n_off, n, f, [](int, int, uint32_t) {});
        }
        bar_arrive(BAR_STORED, 32 * (GW + 1));
        s_round = slot_add(s_round, (uint32_t)n, a.R);
        bar_sync(BAR_GO, threads);
        if (round_failed(failed, r)) return;
    }
}

// ----------------------------------------------------------- rounds in use
// Words s .. s + 3 and s, s + 1 (s < R).  a.vec: the caller's s are multiples of 4
// (of 2 for a pair), so that the words lie together and never cross the ring's end.
__device__ __forceinline__ uint4 ring_quad(const LfgArgs& a, uint32_t s)
{
    if (a.vec) return __ldcg(reinterpret_cast<const uint4*>(a.ring + s));
    return make_uint4(__ldcg(a.ring + s), __ldcg(a.ring + slot_add(s, 1, a.R)), __ldcg(a.ring + slot_add(s, 2, a.R)),
                      __ldcg(a.ring + slot_add(s, 3, a.R)));
}
__device__ __forceinline__ uint2 ring_two(const LfgArgs& a, uint32_t s)
{
    if (a.vec) return __ldcg(reinterpret_cast<const uint2*>(a.ring + s));
    return make_uint2(__ldcg(a.ring + s), __ldcg(a.ring + slot_add(s, 1, a.R)));
}
// Lane's eight words s + 8 lane .. + 7 of the 256 from slot s on.
__device__ __forceinline__ void ring_octet(const LfgArgs& a, uint32_t s, uint4& q0, uint4& q1)
{
    const int lane = threadIdx.x & 31;
    if (a.vec && s <= a.R - 256) {
        const uint4* p = reinterpret_cast<const uint4*>(a.ring + s) + 2 * lane;
        q0 = __ldcg(p), q1 = __ldcg(p + 1);
    } else {
        const uint32_t t = slot_add(s, (uint32_t)(8 * lane), a.R);
        q0 = ring_quad(a, t), q1 = ring_quad(a, slot_add(t, 4, a.R));
    }
}

// Two compensated binary32 sums, in the lanes of the paired instructions.
struct Kahan2 {
    float2 s = {0.f, 0.f}, c = {0.f, 0.f};
    __device__ __forceinline__ void add(float2 e)
    {
        const float2 y = __fadd2_rn(e, make_float2(-c.x, -c.y));
        const float2 t = __fadd2_rn(s, y);
        c = __fadd2_rn(__fadd2_rn(t, make_float2(-s.x, -s.y)), make_float2(-y.x, -y.y));
        s = t;
    }
    __device__ __forceinline__ double value() const
    {
        return ((double)s.x - (double)c.x) + ((double)s.y - (double)c.y);
    }
};

// ------------------------------------------------------------- host side
// Arguments of a launch that starts at the handle's position.
LfgArgs lfg_args(const Handle* h);
// Fan depth of a launch: the process-wide setting, else the ring's own.
int lfg_depth(const Handle* h);
// Order and width (positions) of the widest step of the paper form and the overdamped run.
int lfg_step_order(const Handle* h);
int64_t lfg_step_width(const Handle* h);
// Barrier counter, status words, wait limit and test hook of a launch of G CTAs.
int lfg_begin(Handle* h, LfgArgs& a, int64_t G, cudaStream_t st);
// Wait for the launch and read its status.
int lfg_end(Handle* h, const LfgArgs& a, cudaStream_t st);
int lfg_cooperative(const void* fn, int64_t G, int T, void** args, size_t smem, cudaStream_t st);
enum { LFG_U32 = 0, LFG_UNIFORM = 1, LFG_NORMAL = 2, LFG_LD = 3, LFG_LD_INIT = 4 };
// Small systems (lfg_team.cu): 1 and launched (a.w set), 0 where they do not fit, or
// an error.  a: of the run, x = R for the overdamped one; R0: R(0); n_rec: its
// records, one slot a CTA (h->partials), or 0.
int lfg_team_ld(Handle* h, LfgArgs& a, int k, int64_t n_steps, cudaStream_t st);
int lfg_team_ou(Handle* h, LfgArgs& a, int k, OuCoef c, const float* R0, int64_t n_steps, int64_t every,
                int64_t n_rec, cudaStream_t st);

// f(integral constant K) for a depth k.
template <class F>
static int with_depth(int k, F&& f)
{
    switch (k) {
        case 1: return f(std::integral_constant<int, 1>{});
        case 2: return f(std::integral_constant<int, 2>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 8: return f(std::integral_constant<int, 8>{});
        default: return f(std::integral_constant<int, 16>{});
    }
}

}  // namespace gb
