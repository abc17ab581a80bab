// Lagged Fibonacci handles, uniform fills and the paper-form step (the sequence, its
// ring and rounds: lfg.cuh).
#include <algorithm>
#include <atomic>

#include "lfg.cuh"

namespace gb {

// ------------------------------------------------------------------ fills
// Each CTA owns a contiguous share of every round's offsets, a warp the same units
// of it round after round.  A round's values go to the ring and to shared memory,
// from where, after the CTA's arrival at the barrier, the warps write them out (as
// words, uniforms or normals), so that the output is formed while the barrier
// completes.  b_0 of a full round is the last fan of the round before at the same
// offset: it comes from shared memory.  L2 traffic a value: K / K loads, the ring and
// the output store, 12 B, against 20 with a value from three lag loads; 2^28
// uniforms of the last row 572 -> 444 us (7.3 TB/s of L2 traffic, about the
// L2-resident copy rate), of row 6 3820 -> 776.
//
// Normals: a pair's words lie together in one fan's plane, or, where k D is odd,
// across the end of the CTA's share: the next word is then generated here too
// (`over`), from its own K + 1 loads.  K is even, so a round is whole pairs.
constexpr int kFillWarps = 23, BAR_SHARE = 3;

template <int MODE, int K>
__global__ void __launch_bounds__(32 * (kFillWarps + 1), 1) lfg_fill_kernel(LfgArgs a)
{
    extern __shared__ __align__(16) uint32_t fill_sm[];   // [K][units of the CTA][offsets of a unit]
    __shared__ int64_t s_failed;
    __shared__ uint32_t over[K];
    constexpr int J = fan_j<K>(), FO = 32 * J, T = 32 * (kFillWarps + 1), WORK = 32 * kFillWarps;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_rounds = (a.n_pos + a.w - 1) / a.w;
    if (threadIdx.x == 0) s_failed = kNoRound;
    __syncthreads();
    if (warp == kFillWarps) {
        wait_warp(a, n_rounds - 1, T, T, &s_failed);
        return;
    }
    const int n_off = (int)min((int64_t)min((int)a.D, a.w), a.n_pos);
    const int units = (n_off + FO - 1) / FO;
    const int g0 = (int)((int64_t)blockIdx.x * units / gridDim.x);
    const int g1 = (int)((int64_t)(blockIdx.x + 1) * units / gridDim.x);
    const int plane = (units / (int)gridDim.x + 1) * FO;
    const int o_lo = g0 * FO, o_hi = min(g1 * FO, n_off);   // the share's offsets
    uint32_t sU = a.base_slot;
    for (int64_t r = 0; r < n_rounds; ++r) {
        const int n = (int)min((int64_t)a.w, a.n_pos - r * a.w);
        for (int g = g0 + warp; g < g1; g += kFillWarps) {
            Fan<K> f;
            uint32_t* keep = fill_sm + (g - g0) * FO + lane;
            fan_load<K>(a, slot_add(sU, (uint32_t)(g * FO), a.R), g * FO, f, r ? keep + (K - 1) * plane : nullptr);
            fan_store<K>(a, n_off, n, f, [&](int k, int j, uint32_t v) { keep[k * plane + 32 * j] = v; });
        }
        if (MODE == LFG_NORMAL && threadIdx.x == WORK - 1) {
            // the fan at the share's end; past the last offset, position k D + D is
            // the next fan's first
            const bool end = o_hi == (int)a.D;
            const uint32_t s = slot_add(sU, end ? 0u : (uint32_t)o_hi, a.R);
            uint32_t b[K + 1];
#pragma unroll
            for (int i = 0; i <= K; ++i) b[i] = __ldcg(a.ring + slot_sub(s, a.back[i], a.R));
#pragma unroll
            for (int k = 0; k < K; ++k) {
#pragma unroll
                for (int i = 0; i < K - k; ++i) b[i] += b[i + 1];
                if (!end)
                    over[k] = b[0];
                else if (k > 0)
                    over[k - 1] = b[0];
            }
        }
        if (r + 1 < n_rounds) {
            bar_arrive(BAR_STORED, T);
        }
        if (MODE == LFG_NORMAL) {
            bar_sync(BAR_SHARE, WORK);   // pairs cross units, and so warps
#pragma unroll 1
            for (int k = 0; k < K; ++k) {
                const int at = k * (int)a.D;
                const int first = o_lo + ((at + o_lo) & 1);   // the first even position's offset
                const int pairs = (min(o_hi, n - at) - first + 1) >> 1;
                const uint32_t* row = fill_sm + k * plane - o_lo;
                float2* out = (float2*)((float*)a.out + r * a.w + at + first);
                auto words = [&](int e, uint32_t& x, uint32_t& y) {
                    const int o = first + 2 * e;
                    x = row[o];
                    y = o + 1 < o_hi ? row[o + 1] : over[k];
                };
                for (int e = threadIdx.x; e < pairs; e += 2 * WORK) {
                    const int e1 = e + WORK;
                    uint32_t x0, y0, x1, y1;
                    words(e, x0, y0);
                    words(e1 < pairs ? e1 : e, x1, y1);
                    float2 p0, p1;
                    box_muller_2pairs_u32(x0, y0, x1, y1, p0, p1);
                    __stcs(out + e, p0);
                    if (e1 < pairs) __stcs(out + e1, p1);
                }
            }
        } else {
            for (int g = g0 + warp; g < g1; g += kFillWarps) {
                const uint32_t* keep = fill_sm + (g - g0) * FO + lane;
#pragma unroll
                for (int k = 0; k < K; ++k)
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const int o = g * FO + 32 * j + lane;
                        const int at = o + k * (int)a.D;
                        if (o < n_off && at < n) {
                            const uint32_t v = keep[k * plane + 32 * j];
                            if (MODE == LFG_U32)
                                __stcs((uint32_t*)a.out + r * a.w + at, v);
                            else
                                __stcs((float*)a.out + r * a.w + at, u01_from_u32(v));
                        }
                    }
            }
        }
        sU = slot_add(sU, (uint32_t)n, a.R);
        if (r + 1 < n_rounds) {
            bar_sync(BAR_GO, T);
            if (round_failed(&s_failed, r)) return;
        }
    }
}

// -------------------------------------------------------- single positions
// The value of the position in slot s that lies p < 4 D after the first position not in the
// ring, computed by itself: n = p div D + 1 applications of the recurrence, x_q = sum_i C(n,
// i) x_{q - n D - i sl}, its n + 1 loads side by side.
__device__ __forceinline__ uint32_t lag_value(const LfgArgs& a, uint32_t s, int64_t p)
{
    const int n = 1 + (p >= a.D) + (p >= 2ll * a.D) + (p >= 3ll * a.D);
    const uint32_t binom = n == 1 ? 0x11u : n == 2 ? 0x121u : n == 3 ? 0x1331u : 0x14641u;   // C(n, i), a digit each
    uint32_t t = s, sum = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) t = i < n ? slot_sub(t, a.D, a.R) : t;
#pragma unroll
    for (int i = 0; i <= 4; ++i) {
        if (i <= n) sum += (binom >> (4 * i) & 15u) * __ldcg(a.ring + t);
        t = slot_sub(t, a.sl, a.R);
    }
    return sum;
}

// ----------------------------------------------------------- paper form
// One launch per step (Algorithm 3 with Sec. III.C's one-step-per-launch
// scheme): thread j computes positions P + 4j .. P + 4j + 3 (slots from sP)
// from the ring, stores them, and takes oscillator j's step with x, v and its
// energy sum in global memory.  The launch boundary is the only
// synchronisation, so every position of the step must be dependency-free
// (checked on the host).
__global__ void __launch_bounds__(256) lfg_step_kernel(LfgArgs a, uint32_t sP, float2* eacc)
{
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= a.N) return;
    const uint32_t s = slot_add(sP, (uint32_t)(4 * j), a.R);   // 4j < 4N < R
    uint32_t w[4];
    // all four by one application of the recurrence, or each by one or two, as nearly
    // everywhere: the loads then stand side by side (one after another 1e4 oscillators take 6.2
    // us a step instead of a launch's 4.1, 1e6 26.7 instead of 20.9).  The quad across D is
    // among the latter: by itself its words' loops kept a step of any small row at 6.3 us.
    if (4 * j + 3 < a.D) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const uint32_t t = slot_sub(slot_add(s, r, a.R), a.D, a.R);
            w[r] = __ldcg(a.ring + t) + __ldcg(a.ring + slot_sub(t, a.sl, a.R));
        }
    } else if (4 * j + 3 < 2ll * a.D) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const bool two = 4 * j + r >= a.D;
            uint32_t t = slot_sub(slot_add(s, r, a.R), a.D, a.R);
            if (two) t = slot_sub(t, a.D, a.R);
            const uint32_t b0 = __ldcg(a.ring + t);
            t = slot_sub(t, a.sl, a.R);
            const uint32_t b1 = __ldcg(a.ring + t), b2 = two ? __ldcg(a.ring + slot_sub(t, a.sl, a.R)) : 0u;
            w[r] = b0 + b1 + (two ? b1 + b2 : 0u);
        }
    } else {
#pragma unroll
        for (int r = 0; r < 4; ++r) w[r] = lag_value(a, slot_add(s, r, a.R), 4 * j + r);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) __stcg(a.ring + slot_add(s, r, a.R), w[r]);
    float g0, g1, g2;
    box_muller3_u32(w[0], w[1], w[2], w[3], g0, g1, g2);
    const float Ki = a.Kper ? a.Kper[j] : a.c.K;
    float* xp = a.x + 3 * j;
    float* vp = a.v + 3 * j;
    float x0 = xp[0], x1 = xp[1], x2 = xp[2];
    float v0 = vp[0], v1 = vp[1], v2 = vp[2];
    const float ckx = __fmul_rn(a.c.ckm, Ki);
    em_component(a.c.cdt, a.c.cva, ckx, a.c.cs, g0, x0, v0);
    em_component(a.c.cdt, a.c.cva, ckx, a.c.cs, g1, x1, v1);
    em_component(a.c.cdt, a.c.cva, ckx, a.c.cs, g2, x2, v2);
    xp[0] = x0, xp[1] = x1, xp[2] = x2;
    vp[0] = v0, vp[1] = v1, vp[2] = v2;
    Kahan e;
    const float2 ec = eacc[j];
    e.s = ec.x;
    e.c = ec.y;
    e.add(energy3(0.5f * Ki, a.c.hm, x0, x1, x2, v0, v1, v2));
    eacc[j] = make_float2(e.s, e.c);
}

// Seeds: the value at position w - ll (w = 0..ll-1) is the low half of
// SplitMix64 at counter w, and x_{-ll} is forced odd.  Position q < 0 lives in
// slot q + R.
__global__ void lfg_seed_kernel(uint64_t seed, int32_t ll, LfgArgs a)
{
    const int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (w >= ll) return;
    uint32_t v = (uint32_t)splitmix64_at(seed, (uint64_t)w);
    if (w == 0) v |= 1u;
    a.ring[a.R - (uint32_t)ll + (uint32_t)w] = v;
}

// The recurrence run backwards, x_q = x_{q+ll} - x_{q+sl}, for q in
// [q_hi - count, q_hi): every read lies at q_hi or above (count <= sl).
__global__ void lfg_extend_kernel(LfgArgs a, int64_t q_hi, int64_t count)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= count) return;
    const int64_t q = q_hi - count + i;
    const uint32_t R = a.R;
    a.ring[(uint32_t)(q + R)] = a.ring[(uint32_t)(q + a.D + a.sl + R)] - a.ring[(uint32_t)(q + a.sl + R)];
}

// The whole extension of a small row in one launch, by one cluster of blocks with its
// barrier between the pieces (other blocks' values come from L2).  n applications of the
// reverse, x_q = sum_i (-1)^i C(n, i) x_{q + (n-i) ll + i sl}, give pieces of n sl positions once
// every read lies below 0, from q = -n ll on: a fan of depth 16 takes 7 or 8 pieces with n up to
// 4 where it takes 15 with one (handle of row 0, 3, 6 made in 32, 37, 60 us with one; 28, 32, 55
// with two; 26, 30, 56 with four; a launch each 81 for row 2).
constexpr int kExtBlocks = 8, kExtThreads = 1024;
template <int N>
__device__ __forceinline__ void extend_piece(const LfgArgs& a, int64_t q, int64_t cnt)
{
    constexpr uint32_t binom = N == 1 ? 0x11u : N == 2 ? 0x121u : 0x14641u;   // C(N, i), a digit each
    const uint32_t s0 = (uint32_t)(q + a.R), ll = a.D + a.sl;
#pragma unroll 4
    for (uint32_t i = blockIdx.x * kExtThreads + threadIdx.x; i < (uint32_t)cnt; i += kExtBlocks * kExtThreads) {
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k <= N; ++k) {
            const uint32_t v = (binom >> (4 * k) & 15u) * __ldcg(a.ring + s0 + i + (N - k) * ll + k * a.sl);
            sum += k & 1 ? 0u - v : v;
        }
        __stcg(a.ring + s0 + i, sum);
    }
}

__global__ void __cluster_dims__(kExtBlocks, 1, 1) __launch_bounds__(kExtThreads)
    lfg_extend_all_kernel(LfgArgs a, int64_t q_hi, int64_t q_end)
{
    const int64_t ll = (int64_t)a.D + a.sl;
    while (q_hi > q_end) {
        const int n = q_hi <= -4 * ll ? 4 : q_hi <= -2 * ll ? 2 : 1;
        const int64_t cnt = min((int64_t)n * a.sl, q_hi - q_end);
        q_hi -= cnt;
        if (n == 4) extend_piece<4>(a, q_hi, cnt);
        else if (n == 2) extend_piece<2>(a, q_hi, cnt);
        else extend_piece<1>(a, q_hi, cnt);
        cluster_sync();
    }
}

// ------------------------------------------------------------- host side
LfgArgs lfg_args(const Handle* h)
{
    LfgArgs a{};
    a.ring = h->ring;
    a.R = h->ring_size;
    a.D = (uint32_t)(h->ll - h->sl);
    a.sl = (uint32_t)h->sl;
    for (int64_t i = 0; i <= 16; ++i) a.back[i] = (uint32_t)((a.D + i * a.sl) % a.R);
    for (int64_t k = 0; k < 16; ++k) a.ahead[k] = (uint32_t)(k * a.D % a.R);
    a.base_slot = slot_of(h->pos, h->ring_size);
    a.vec = a.base_slot % 4 == 0;
    return a;
}

int lfg_seed(Handle* h, cudaStream_t st)
{
    h->pos = 0;
    const int T = 256;
    const LfgArgs a = lfg_args(h);
    lfg_seed_kernel<<<(unsigned)((h->ll + T - 1) / T), T, 0, st>>>(h->seed, h->ll, a);
    GB_CUDA(cudaGetLastError());
    // x_{-H} .. x_{-ll-1}, in pieces of sl positions from -ll downwards: in one launch where
    // a piece is at most eight words a thread of the cluster, else in one each
    const int64_t q_end = -lfg_history(h);
    if (h->sl <= 8 * kExtBlocks * kExtThreads) {
        lfg_extend_all_kernel<<<kExtBlocks, kExtThreads, 0, st>>>(a, -(int64_t)h->ll, q_end);
    } else {
        for (int64_t q_hi = -(int64_t)h->ll; q_hi > q_end;) {
            const int64_t cnt = std::min<int64_t>(h->sl, q_hi - q_end);
            lfg_extend_kernel<<<(unsigned)((cnt + T - 1) / T), T, 0, st>>>(a, q_hi, cnt);
            q_hi -= cnt;
        }
    }
    GB_CUDA(cudaGetLastError());
    return GBRNG_OK;
}

// Fan depth: the process-wide setting, else the ring's own, at most the ring's.
static std::atomic<int> g_lfg_order{0};

void lfg_new_handle(Handle* h)
{
    const int64_t D = (int64_t)h->ll - h->sl;
    h->order_max = g_lfg_order.load() == 4 ? 4 : 2;
    int k = 16;
    while (k > 2 && k * D > 4100000) k /= 2;
    h->depth = std::max(k, h->order_max);
    const int64_t R = std::max(3 * h->depth * D, h->depth * D + lfg_history(h));
    h->ring_size = (uint32_t)((R + 31) & ~(int64_t)31);
}

int lfg_depth(const Handle* h)
{
    const int o = g_lfg_order.load();
    return o ? std::min(o, h->depth) : h->depth;
}

// The order set, at most the handle's, or 2.
int lfg_step_order(const Handle* h)
{
    const int o = g_lfg_order.load();
    return o ? std::min(o, h->order_max) : 2;
}

// k D positions of that order k (whole quads).
int64_t lfg_step_width(const Handle* h)
{
    return (lfg_step_order(h) * ((int64_t)h->ll - h->sl)) & ~(int64_t)3;
}

// Barrier counter, status words, wait limit and test hook of one launch.
int lfg_begin(Handle* h, LfgArgs& a, int64_t G, cudaStream_t st)
{
    GB_CHECK(ensure_progress(h, 2));
    a.arrive = h->progress;
    a.status = reinterpret_cast<int*>(h->progress + 1);
    char* host = (char*)host_block();
    if (!host) return fail(GBRNG_ENOMEM, "cannot allocate pinned host memory");
    a.host_status = reinterpret_cast<int*>(host + kHostBlock - 64);
    *a.host_status = DEV_OK;
    a.wait_ns = wait_limit_ns();
    const int64_t stall = test_stall_chunk();
    a.stall_cta = stall < 0 ? -1 : (int)(stall % G);
    GB_CUDA(cudaMemsetAsync(h->progress, 0, 2 * sizeof(uint64_t), st));
    return GBRNG_OK;
}

int lfg_end(Handle* h, const LfgArgs& a, cudaStream_t st)
{
    GB_CHECK(sync_results(st));
    if (*(volatile int*)a.host_status == DEV_TIMEOUT) {
        // some CTAs may have counted themselves into the statistics
        GB_CUDA(cudaMemsetAsync(h->ticket, 0, sizeof(unsigned), st));
        return fail(GBRNG_ETIMEOUT, "Lagged Fibonacci grid barrier wait exceeded %llu ns",
                    (unsigned long long)wait_limit_ns());
    }
    return GBRNG_OK;
}

int lfg_cooperative(const void* fn, int64_t G, int T, void** args, size_t smem, cudaStream_t st)
{
    // beyond 48 KB with the kernel's own, at most 2 KB, the limit has to be raised: to one
    // value, as another thread may launch the same kernel with more in between
    if (smem > 46 * 1024) {
        int device = 0;
        DevInfo di;
        GB_CUDA(cudaGetDevice(&device));
        GB_CHECK(dev_info(device, &di));
        GB_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)di.smem_optin - 2048));
    }
    GB_CUDA(cudaLaunchCooperativeKernel(fn, dim3((unsigned)G), dim3(T), args, smem, st));
    return GBRNG_OK;
}

int lfg_fill(Handle* h, void* dst, int64_t n, int mode, cudaStream_t st)
{
    // normals: whole pairs a round, so an even depth
    const int k = mode == LFG_NORMAL ? std::max(lfg_depth(h), 2) : lfg_depth(h);
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    LfgArgs a = lfg_args(h);
    a.n_pos = n;
    a.out = dst;
    a.w = (int)((int64_t)k * a.D);
    // no more CTAs than a round has units: the barrier is cheaper (1000 uniforms of row 9 27.2 ->
    // 24.6 us; row 0 with order 2 forced, 6 CTAs, 1e7 uniforms 8.93 -> 7.60 ms)
    const int FO = with_depth(k, [](auto kk) { return fan_offsets<decltype(kk)::value>(); });
    const int64_t units = (std::min<int64_t>(a.D, n) + FO - 1) / FO, G = std::min<int64_t>(di.sms, units);
    GB_CHECK(lfg_begin(h, a, G, st));
    void* args[] = {&a};
    GB_CHECK(with_depth(k, [&](auto kk) {
        constexpr int K = decltype(kk)::value;
        const size_t smem = sizeof(uint32_t) * K * (size_t)(units / G + 1) * FO;
        const void* fn = mode == LFG_U32       ? (const void*)lfg_fill_kernel<LFG_U32, K>
                         : mode == LFG_UNIFORM ? (const void*)lfg_fill_kernel<LFG_UNIFORM, K>
                                               : (const void*)lfg_fill_kernel<LFG_NORMAL, K == 1 ? 2 : K>;
        return lfg_cooperative(fn, G, 32 * (kFillWarps + 1), args, smem, st);
    }));
    GB_CHECK(lfg_end(h, a, st));
    h->pos += n;
    return GBRNG_OK;
}

int lfg_ld_stepwise(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    Handle* h = s->rng;
    if (s->n == 0) {
        if (out) *out = ld_stats{0, 0, 0, 0, n_steps};
        return GBRNG_OK;
    }
    const int64_t four_n = 4 * s->n;
    if (four_n > lfg_step_width(h))
        return fail(GBRNG_ELAGS,
                    "one launch per step needs 4N = %lld within %d times the lag distance "
                    "(ll - sl = %lld)",
                    (long long)four_n, lfg_step_order(h), (long long)(h->ll - h->sl));
    GB_CHECK(ensure_eacc(h, s->n));
    GB_CUDA(cudaMemsetAsync(h->eacc, 0, sizeof(float2) * s->n, st));
    LfgArgs a = lfg_args(h);
    a.N = s->n;
    a.x = s->x;
    a.v = s->v;
    a.Kper = s->K_per;
    a.c = make_coef(s);
    const unsigned blocks = (unsigned)((s->n + 255) / 256);
    uint32_t sP = a.base_slot;
    for (int64_t t = 0; t < n_steps; ++t) {
        lfg_step_kernel<<<blocks, 256, 0, st>>>(a, sP, h->eacc);
        sP = slot_add(sP, (uint32_t)four_n, a.R);
    }
    GB_CUDA(cudaGetLastError());
    h->pos += four_n * n_steps;
    return stepwise_stats(h, s, n_steps, out, st);
}

}  // namespace gb

using namespace gb;

extern "C" int gbrng_set_lfg_order(int k)
{
    if (k != 0 && k != 1 && k != 2 && k != 4)
        return fail(GBRNG_EINVAL, "Lagged Fibonacci leap order must be 0 (automatic), 1, 2 or 4");
    g_lfg_order.store(k);
    return GBRNG_OK;
}
