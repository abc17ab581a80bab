// The launches that use the Lagged Fibonacci sequence as it is generated (lfg.cuh):
// Langevin runs, the equilibrium start and normal fills.
#include <algorithm>
#include <climits>

#include "lfg.cuh"

namespace gb {

// Two oscillators' step in the lanes of the paired instructions, from their raw
// words; each lane em_component's and energy3's operations.
__device__ __forceinline__ float2 pair_step(const LdCoef& c, float2 nckx, float2 hK, uint4 w0, uint4 w1,
                                            float2 (&X)[3], float2 (&V)[3])
{
    const uint32_t r[2][4] = {{w0.x, w0.y, w0.z, w0.w}, {w1.x, w1.y, w1.z, w1.w}};
    float2 g[3];
    normals3x2_u32(r, g);
#pragma unroll
    for (int q = 0; q < 3; ++q) em_component2(splat2(c.cdt), splat2(c.cva), nckx, splat2(c.cs), g[q], X[q], V[q]);
    return __ffma2_rn(hK, EnergySum2::norm2x2(X), __fmul2_rn(splat2(c.hm), EnergySum2::norm2x2(V)));
}

__device__ __forceinline__ void final_sums(const float2 (&X)[3], const float2 (&V)[3], bool live0, bool live1,
                                           double (&acc)[4])
{
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (live0) {
            acc[0] += (double)X[q].x * X[q].x;
            acc[1] += (double)V[q].x * V[q].x;
            acc[2] += (double)X[q].x * V[q].x;
        }
        if (live1) {
            acc[0] += (double)X[q].y * X[q].y;
            acc[1] += (double)V[q].y * V[q].y;
            acc[2] += (double)X[q].y * V[q].y;
        }
    }
}

// The Langevin run with x and v on chip: CTA c owns the oscillators [c n_c, c n_c +
// n_c) for the whole launch, their x and v in shared memory, and a round holds
// whole steps (W = 4 N S).  A worker warp takes units of 64 oscillators, two a
// lane, through all steps of the round.
constexpr int kUnitWords = 6 * 64;   // a unit's x and v: [x, v][component][oscillator]

template <int K, int CW, int GW>
__global__ void __launch_bounds__(32 * (CW + GW + 1), 1) lfg_resident_kernel(LfgArgs a, int n_c)
{
    extern __shared__ __align__(16) float res_sm[];   // [unit][kUnitWords]
    __shared__ int64_t s_failed;
    __shared__ double red[4 * 32];
    constexpr int T = 32 * (CW + GW + 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * n_c;
    const int nc = (int)max((int64_t)0, min(a.N - j0, (int64_t)n_c));
    const int n_units = (nc + 63) >> 6;
    const int64_t n_rounds = (a.n_pos + a.w - 1) / a.w;
    if (threadIdx.x == 0) s_failed = kNoRound;
    // word q of oscillator j of the CTA (q: x, then v)
    auto at = [](int j, int q) { return (j >> 6) * kUnitWords + 64 * q + (j & 63); };
    for (int i = threadIdx.x; i < 3 * nc; i += T) {
        const int j = i / 3, q = i - 3 * j;
        res_sm[at(j, q)] = a.x[3 * j0 + i];
        res_sm[at(j, 3 + q)] = a.v[3 * j0 + i];
    }
    __syncthreads();
    Kahan2 e;
    if (warp >= CW + GW) {
        wait_warp(a, n_rounds, 32 * (GW + 1), T, &s_failed);
    } else if (warp >= CW) {
        gen_warps<K, GW>(a, warp - CW, n_rounds, T, &s_failed);
    } else {
        // slot of this warp's first unit in the round's first step
        uint32_t s_first = slot_add(slot_add(a.base_slot, (uint32_t)(4 * min(j0, a.N)), a.R), (uint32_t)(256 * min(warp, n_units)), a.R);
        const uint32_t step_slots = (uint32_t)(4 * a.N);
        const int S = a.w / (int)(4 * a.N);   // steps a round
        int64_t left = a.n_steps;
        for (int64_t p = 0; p < n_rounds; ++p) {
            const int steps = (int)min((int64_t)S, left);
            left -= steps;
            bar_sync(BAR_GO, T);
            if (round_failed(&s_failed, p)) break;
            // raw words are loaded one item (a unit's step) ahead
            uint4 w0, w1;
            uint32_t su = s_first;
            if (warp < n_units) ring_octet(a, su, w0, w1);
#pragma unroll 1
            for (int u = warp; u < n_units; u += CW) {
                const int j = 64 * u + 2 * lane;
                float* xs = res_sm + u * kUnitWords + 2 * lane;
                float2 X[3], V[3];
                float k0 = a.c.K, k1 = a.c.K;
                if (a.Kper) {
                    if (j < nc) k0 = __ldg(a.Kper + j0 + j);
                    if (j + 1 < nc) k1 = __ldg(a.Kper + j0 + j + 1);
                }
                const float2 nckx = make_float2(-__fmul_rn(a.c.ckm, k0), -__fmul_rn(a.c.ckm, k1));
                const float2 hK = make_float2(0.5f * k0, 0.5f * k1);
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    X[q] = *reinterpret_cast<const float2*>(xs + 64 * q);
                    V[q] = *reinterpret_cast<const float2*>(xs + 64 * (3 + q));
                }
                uint32_t ss = su;
                su = u + CW < n_units ? slot_add(su, 256u * CW, a.R) : su;
#pragma unroll 1
                for (int s = 1; s <= steps; ++s) {
                    ss = s < steps ? slot_add(ss, step_slots, a.R) : su;
                    uint4 n0, n1;
                    ring_octet(a, ss, n0, n1);
                    float2 en = pair_step(a.c, nckx, hK, w0, w1, X, V);
                    if (j + 1 >= nc) {   // a unit's dead oscillators
                        en.y = 0.f;
                        if (j >= nc) en.x = 0.f;
                    }
                    e.add(en);
                    w0 = n0, w1 = n1;
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    *reinterpret_cast<float2*>(xs + 64 * q) = X[q];
                    *reinterpret_cast<float2*>(xs + 64 * (3 + q)) = V[q];
                }
            }
            s_first = slot_add(s_first, (uint32_t)a.w, a.R);
        }
    }
    __syncthreads();
    if (s_failed != kNoRound) return;
    double acc[4] = {0, 0, 0, 0};
    for (int i = threadIdx.x; i < 3 * nc; i += T) {
        const int j = i / 3, q = i - 3 * j;
        const float x = res_sm[at(j, q)], v = res_sm[at(j, 3 + q)];
        a.x[3 * j0 + i] = x;
        a.v[3 * j0 + i] = v;
        acc[0] += (double)x * x;
        acc[1] += (double)v * v;
        acc[2] += (double)x * v;
    }
    if (a.sink.partials) {
        acc[3] = e.value();
        const double sums = block_sums(acc, red);
        if (warp == 0) store_stats(a.sink, sums);
    }
}

// The runs whose data streams through global memory: Langevin steps of systems beyond the
// resident kernel and the equilibrium start.  A round is shared out in units of 64 quads
// of words (oscillator-steps, two a lane); a Langevin round holds at most half a step (W <=
// 2 N), so that an oscillator's next step comes two phases later at the earliest, after
// the barrier that its last update's stores precede.
//
// A unit's x, v and K pass through shared memory, copied in (cp.async) while the warp works
// on the unit before, and out again, side by side over the warp: 16, 8 or 4 bytes a lane as
// the unit's first words are aligned, which for an odd N changes from step to step.  A lane's
// six words taken straight from x and v are strided, three accesses from an 8-byte boundary
// and up to six elsewhere, and K was waited for at its use: us a step before / so, even N,
// odd N, odd N with K_per: 2e6 26.1 / 22.7, 43.5 / 23.7, 46.2 / 26.7; 1e7 139 / 129, 231 /
// 138, 230 / 146.  (4 bytes a lane always 151 at 1e7, at most 8 139; three stages instead
// of two 1 to 2% slower.)
constexpr int kStreamStages = 2, kStageWords = 7 * 64;   // of a warp: x, v [64][3], K [64]
template <int CW>
constexpr size_t stream_smem() { return sizeof(float) * kStageWords * kStreamStages * CW; }

template <int BYTES>
using Width = std::integral_constant<int, BYTES>;
template <int BYTES>
using Words = typename std::conditional<BYTES == 4, float, typename std::conditional<BYTES == 8, float2, float4>::type>::type;

template <int BYTES>
__device__ __forceinline__ void copy_words(float* to, const float* from, Width<BYTES>)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from),
                 "n"(BYTES)
                 : "memory");
}
template <int BYTES>
__device__ __forceinline__ void store_words(float* to, const float* from, Width<BYTES>)
{
    *reinterpret_cast<Words<BYTES>*>(to) = *reinterpret_cast<const Words<BYTES>*>(from);
}

template <int MODE, int K, int CW, int GW>
__global__ void __launch_bounds__(32 * (CW + GW + 1), 1) lfg_stream_kernel(LfgArgs a)
{
    extern __shared__ __align__(16) float str_sm[];   // LD: [using warp][stage][kStageWords]
    __shared__ int64_t s_failed;
    __shared__ double red[4 * 32];
    constexpr int T = 32 * (CW + GW + 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_rounds = (a.n_pos + a.w - 1) / a.w;
    if (threadIdx.x == 0) s_failed = kNoRound;
    __syncthreads();
    Kahan2 e;
    double acc[4] = {0, 0, 0, 0};
    if (warp >= CW + GW) {
        wait_warp(a, n_rounds, 32 * (GW + 1), T, &s_failed);
    } else if (warp >= CW) {
        gen_warps<K, GW>(a, warp - CW, n_rounds, T, &s_failed);
    } else {
        uint32_t s_round = a.base_slot;
        int64_t j_round = 0, t_round = 0;   // oscillator and step of the round's first quad
        int n = 0, quads = 0, u0 = 0, u1 = 0;
        float* const stages = str_sm + warp * kStreamStages * kStageWords;
        for (int64_t p = 0; p < n_rounds; ++p) {
            const int64_t U = p * a.w;   // launch offset of the round
            if (p == 0 || p == n_rounds - 1) {
                n = (int)min((int64_t)a.w, a.n_pos - U);
                quads = (n + 3) >> 2;
                const unsigned units = (unsigned)(quads + 63) >> 6;
                u0 = (int)(blockIdx.x * units / gridDim.x) + warp;
                u1 = (int)((blockIdx.x + 1) * units / gridDim.x);
            }
            // the quads from `wrap` on belong to the next step
            const int wrap = (int)min(a.N - j_round, (int64_t)INT_MAX);
            auto index = [&](int qd) { return j_round + qd - (qd >= wrap ? a.N : 0); };
            // f(k, i, width): this lane passes `width` bytes of unit uu's words from the k-th of
            // 64 x 3 on, which is word i of x and of v
            auto words = [&](int uu, auto&& f) {
                const int q0 = 64 * uu;
                if (q0 + 64 <= quads && (q0 >= wrap || q0 + 64 <= wrap)) {
                    const int64_t i = 3 * index(q0);
                    const uint32_t low = (uint32_t)(uintptr_t)(a.x + i) | (uint32_t)(uintptr_t)(a.v + i);
                    if (low % 16 == 0) {
                        f(4 * lane, i + 4 * lane, Width<16>{});
                        if (lane < 16) f(128 + 4 * lane, i + 128 + 4 * lane, Width<16>{});
                    } else if (low % 8 == 0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) f(64 * c + 2 * lane, i + 64 * c + 2 * lane, Width<8>{});
                    } else {
#pragma unroll
                        for (int c = 0; c < 6; ++c) f(32 * c + lane, i + 32 * c + lane, Width<4>{});
                    }
                } else {
#pragma unroll 1
                    for (int k = lane; k < 192; k += 32)
                        if (q0 + k / 3 < quads) f(k, 3 * index(q0 + k / 3) + k % 3, Width<4>{});
                }
            };
            auto copy_in = [&](int uu, float* st) {
                if (uu < u1) {
                    words(uu, [&](int k, int64_t i, auto w) {
                        copy_words(st + k, a.x + i, w);
                        copy_words(st + 192 + k, a.v + i, w);
                    });
                    if (a.Kper)
#pragma unroll
                        for (int k = lane; k < 64; k += 32)
                            if (64 * uu + k < quads) copy_words(st + 384 + k, a.Kper + index(64 * uu + k), Width<4>{});
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            bar_sync(BAR_GO, T);
            if (round_failed(&s_failed, p)) break;
            uint4 w0, w1;
            if (u0 < u1) ring_octet(a, slot_add(s_round, (uint32_t)(256 * u0), a.R), w0, w1);
            int stage = 0;
            if (MODE == LFG_LD) copy_in(u0, stages);
#pragma unroll 1
            for (int u = u0; u < u1; u += CW) {
                const int qd = 64 * u + 2 * lane;   // first quad of this lane
                const bool live0 = qd < quads, live1 = qd + 1 < quads;
                uint4 n0, n1;
                if (u + CW < u1) ring_octet(a, slot_add(s_round, (uint32_t)(256 * (u + CW)), a.R), n0, n1);
                if (MODE == LFG_LD) {
                    float* const st = stages + stage * kStageWords;
                    stage ^= 1;
                    __syncwarp();   // the warp has left the unit before's stage
                    copy_in(u + CW, stages + stage * kStageWords);
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    __syncwarp();
                    float2* const xs = reinterpret_cast<float2*>(st) + 3 * lane;
                    float2* const vs = xs + 96;
                    const float2 k = a.Kper ? reinterpret_cast<const float2*>(st + 384)[lane] : splat2(a.c.K);
                    const float2 x0 = xs[0], x1 = xs[1], x2 = xs[2], v0 = vs[0], v1 = vs[1], v2 = vs[2];
                    float2 x[3] = {make_float2(x0.x, x1.y), make_float2(x0.y, x2.x), make_float2(x1.x, x2.y)};
                    float2 v[3] = {make_float2(v0.x, v1.y), make_float2(v0.y, v2.x), make_float2(v1.x, v2.y)};
                    float2 en = pair_step(a.c, make_float2(-__fmul_rn(a.c.ckm, k.x), -__fmul_rn(a.c.ckm, k.y)),
                                          make_float2(0.5f * k.x, 0.5f * k.y), w0, w1, x, v);
                    if (!live0) en.x = 0.f;
                    if (!live1) en.y = 0.f;
                    e.add(en);
                    const bool la = t_round + (qd >= wrap) == a.n_steps - 1;
                    const bool lb = t_round + (qd + 1 >= wrap) == a.n_steps - 1;
                    if (la || lb) final_sums(x, v, live0 && la, live1 && lb, acc);
                    xs[0] = make_float2(x[0].x, x[1].x), xs[1] = make_float2(x[2].x, x[0].y), xs[2] = make_float2(x[1].y, x[2].y);
                    vs[0] = make_float2(v[0].x, v[1].x), vs[1] = make_float2(v[2].x, v[0].y), vs[2] = make_float2(v[1].y, v[2].y);
                    __syncwarp();
                    words(u, [&](int k, int64_t i, auto w) {
                        store_words(a.x + i, st + k, w);
                        store_words(a.v + i, st + 192 + k, w);
                    });
                } else {
                    // draw-step 0 -> x = sqrt(kT/K_i) g, draw-step 1 -> v = sqrt(kT/m) g
                    const int64_t ja = index(live0 ? qd : 0), jb = index(live1 ? qd + 1 : 0);
                    const float k0 = a.Kper ? __ldg(a.Kper + ja) : a.c.K, k1 = a.Kper ? __ldg(a.Kper + jb) : a.c.K;
                    float g[2][3];
                    box_muller3_u32(w0.x, w0.y, w0.z, w0.w, g[0][0], g[0][1], g[0][2]);
                    box_muller3_u32(w1.x, w1.y, w1.z, w1.w, g[1][0], g[1][1], g[1][2]);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (!(h ? live1 : live0)) continue;
                        const int64_t j = h ? jb : ja;
                        const bool pos = t_round + (qd + h >= wrap) == 0;
                        const float f = pos ? __fsqrt_rn(__fdiv_rn(a.c.kT, h ? k1 : k0)) : a.c.sv;
#pragma unroll
                        for (int q = 0; q < 3; ++q) (pos ? a.x : a.v)[3 * j + q] = __fmul_rn(f, g[h][q]);
                    }
                }
                w0 = n0, w1 = n1;
            }
            if (MODE == LFG_LD) __syncwarp();   // the stages are left before the next round's copies
            s_round = slot_add(s_round, (uint32_t)n, a.R);
            j_round += n >> 2;
            if (j_round >= a.N) j_round -= a.N, ++t_round;
        }
    }
    if (MODE == LFG_LD && a.sink.partials) {
        __syncthreads();
        if (s_failed != kNoRound) return;
        acc[3] = e.value();
        const double sums = block_sums(acc, red);
        if (warp == 0) store_stats(a.sink, sums);
    }
}

// ------------------------------------------------------------- host side
// Using and generating warps, whose sum also sets the registers a thread has.  The
// resident kernel: 15 and 12, per step of 1e6 oscillators 6.80 us (7.08 with 15 and 16,
// 7.04 with 14 and 13, 7.12 with 13 and 14, 7.3 with 15 or 16 and 11, 7.8 with 15 and 8:
// the generating warps' loads in flight and the using warps' arithmetic share a round).
// The streamed one (us a step at 1.1e6, 1.2e6, 1500001, 2e6, 1e7 oscillators): 11 and 12
// 15.6, 15.4, 20.2, 24.6, 134; 12 and 10 16.5, 16.9, 18.6, 22.7, 129; 13 and 10 ., ., ., 24.5,
// 130; 10 and 13 15.0, 16.2, 19.8, 25.6, 139.  A round holds at most 2 N of its k D
// positions, so the narrow ones leave less time to generate: 11 and 12 up to 3 N = k D.
constexpr int kResWarps = 15, kResGen = 12;

template <int MODE, int CW, int GW>
static int launch_stream(Handle* h, LfgArgs& a, int k, cudaStream_t st)
{
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int64_t G = di.sms;
    GB_CHECK(lfg_begin(h, a, G, st));
    void* args[] = {&a};
    return with_depth(k, [&](auto kk) {
        constexpr int K = decltype(kk)::value;
        return lfg_cooperative((const void*)lfg_stream_kernel<MODE, K, CW, GW>, G, 32 * (CW + GW + 1), args,
                               MODE == LFG_LD ? stream_smem<CW>() : 0, st);
    });
}

// Final-state statistics when no step is taken.
__global__ void snapshot_kernel(const float* x, const float* v, int64_t n, StatsSink sink)
{
    __shared__ double red[4 * 32];
    double acc[4] = {0, 0, 0, 0};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 3 * n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const double xi = x[i], vi = v[i];
        acc[0] += xi * xi;
        acc[1] += vi * vi;
        acc[2] += xi * vi;
    }
    const double sums = block_sums(acc, red);
    if (threadIdx.x < 32) store_stats(sink, sums);
}

// The resident kernel takes a system whose step fits a round (4 N <= k D) and
// whose share of x and v fits a CTA's shared memory.
static bool resident_fits(const Handle* h, int64_t n, int k, const DevInfo& di, int* n_c, size_t* smem)
{
    if (4 * n > (int64_t)k * (h->ll - h->sl)) return false;
    const int64_t c = ((n + di.sms - 1) / di.sms + 1) & ~(int64_t)1;
    *n_c = (int)c;
    *smem = sizeof(float) * kUnitWords * (size_t)((c + 63) / 64);
    return *smem + 2048 <= di.smem_optin;
}

int lfg_ld(const ld_system* s, int64_t n_steps, int init, ld_stats* out, cudaStream_t st)
{
    Handle* h = s->rng;
    if (s->n == 0 || (!init && n_steps == 0)) {
        if (!out) return GBRNG_OK;
        if (s->n == 0) {
            *out = ld_stats{0, 0, 0, 0, n_steps};
            return GBRNG_OK;
        }
        StatsSink sink;
        GB_CHECK(make_sink(h, 256, true, &sink));
        snapshot_kernel<<<256, 256, 0, st>>>(s->x, s->v, s->n, sink);
        GB_CUDA(cudaGetLastError());
        return finish_stats(h, sink, 256, 0, out, st);
    }
    const int k = lfg_depth(h);
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int64_t G = di.sms;
    LfgArgs a = lfg_args(h);
    a.N = s->n;
    a.n_steps = init ? 2 : n_steps;
    a.n_pos = 4 * s->n * a.n_steps;
    a.x = s->x;
    a.v = s->v;
    a.Kper = s->K_per;
    a.c = make_coef(s);
    GB_CHECK(make_sink(h, G, out != nullptr, &a.sink));
    int n_c = 0;
    size_t smem = 0;
    if (init) {
        a.w = (int)((int64_t)k * a.D & ~(int64_t)3);
        GB_CHECK((launch_stream<LFG_LD_INIT, 15, 8>(h, a, k, st)));
    } else if (const int rc = lfg_team_ld(h, a, k, n_steps, st)) {
        if (rc < 0) return rc;
    } else if (resident_fits(h, s->n, k, di, &n_c, &smem)) {
        a.w = (int)(4 * s->n * std::min<int64_t>((int64_t)k * a.D / (4 * s->n), n_steps));
        GB_CHECK(lfg_begin(h, a, G, st));
        void* args[] = {&a, &n_c};
        GB_CHECK(with_depth(k, [&](auto kk) {
            constexpr int K = decltype(kk)::value;
            return lfg_cooperative((const void*)lfg_resident_kernel<K, kResWarps, kResGen>, G,
                                   32 * (kResWarps + kResGen + 1), args,
                                   smem, st);
        }));
    } else {
        // whole groups of four oscillators, whose x and v start on 16 bytes
        a.w = (int)(std::min<int64_t>((int64_t)k * a.D, 2 * s->n) & ~(int64_t)15);
        if (3 * s->n < (int64_t)k * a.D)
            GB_CHECK((launch_stream<LFG_LD, 11, 12>(h, a, k, st)));
        else
            GB_CHECK((launch_stream<LFG_LD, 12, 10>(h, a, k, st)));
    }
    GB_CHECK(lfg_end(h, a, st));
    h->pos += a.n_pos;
    return finish_stats(h, a.sink, G, n_steps, out, st);
}

}  // namespace gb
