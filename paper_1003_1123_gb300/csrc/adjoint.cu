// Reverse-time adjoint of the trajectory-averaged energy
//   L = (1/S) sum_{t=1..S} sum_i ( m |v_i(t)|^2 + K_i |x_i(t)|^2 ) / 2
// under fixed noise, for the per-thread generators.
//
// Oscillators are independent, so one thread carries one oscillator through
//  A) the forward run, writing a checkpoint (x, v, generator state) at the
//     start of every segment of P steps, accumulating L and the direct part
//     of dL/dK_i, and finally the end state;
//  B) the reverse sweep, segment by segment from the last: the segment's
//     normals (3 floats per step) are either read from the history A wrote
//     when the whole run's noise fits the history limit, or regenerated
//     bit-exactly into a scratch buffer from the segment's checkpointed
//     generator state; then,
//     walking the segment backwards from its exact end state (the next
//     checkpoint, or the final state), each step is inverted,
//        v_t = (v_{t+1} + b x_{t+1} - c g_t) / (a + b dt),  x_t = x_{t+1} - dt v_t,
//     and the discrete adjoint recursion is applied:
//        lx_t = lx_{t+1} - b lv_{t+1} + [t>=1] K x_t / S,
//        lv_t = dt lx_{t+1} + a lv_{t+1} + [t>=1] m v_t / S,
//     with a = 1 - gamma dt/m, b = dt K_i/m, c = sqrt(2 gamma kT dt)/m, and
//        dL/dK_i   += -(dt/m) lv_{t+1}.x_t,
//        dL/dgamma += lv_{t+1}.(-(dt/m) v_t + c/(2 gamma) g_t),
//        dL/dkT    += lv_{t+1}.(c/(2 kT) g_t).
// Inversion only runs inside one segment (at most P steps from an exact
// state), where it is stable.  Sums over steps are Kahan-compensated binary32,
// sums over oscillators fixed-order doubles.
#include <algorithm>
#include <atomic>

#include "device.cuh"
#include "internal.cuh"

namespace gb {

struct AdjArgs {
    int64_t n, S, P, nseg;
    float* x;
    float* v;
    const float* Kper;
    LdCoef c;
    float c_over_2g, c_over_2kT, invS, m;
    uint4* taus;
    int32_t* r2;
    int64_t streams;
    float* ckpt;        // [nseg][6 + state words][n]
    float* gbuf;        // [S][3][n] the run's noise, or [P][3][n] a segment's
    float* dK;          // [n] or null
    StatsSink sink;     // loss, dgamma, dkT, unused
};

// Two compensated binary32 sums in the lanes of the paired instructions.
struct KahanPair {
    float2 s = {0.f, 0.f}, c = {0.f, 0.f};
    __device__ __forceinline__ void add(float a, float b)
    {
        const float2 y = __fadd2_rn(make_float2(a, b), make_float2(-c.x, -c.y));
        const float2 t = __fadd2_rn(s, y);
        c = __fadd2_rn(__fadd2_rn(t, make_float2(-s.x, -s.y)), make_float2(-y.x, -y.y));
        s = t;
    }
    __device__ __forceinline__ double first() const { return (double)s.x - (double)c.x; }
    __device__ __forceinline__ double second() const { return (double)s.y - (double)c.y; }
};

// Where the reverse sweep's normals come from: regenerated segment by segment, or
// kept by the forward run.
enum { NOISE_REGEN = 0, NOISE_KEPT = 1 };

// The reverse sweep is bound by the latency of its loads where the noise is kept
// (one step's three normals at a time, 12 B from memory): with the next eight
// steps' loads in flight and up to 128 registers, 64-thread blocks, eight a SM, 1e5
// oscillators x 1000 steps take 1.09 ms for Hybrid Taus (1.55 with no load ahead;
// twelve blocks at 85 registers: 1.48 with one step ahead, 1.25 with three, 1.13
// with four, 1.17 with eight), 1.20 for Ran2 (1.75); 1e4 x 1000 0.27 (0.62).
// Regenerated noise comes back from L2 and needs two.  Components 0 and 2 and the
// compensated sums run in the lanes of the paired instructions.
template <int KIND, int NOISE>
__global__ void __launch_bounds__(64, 8) adjoint_kernel(AdjArgs a)
{
    constexpr int kAhead = NOISE == NOISE_REGEN ? 2 : 8;   // steps whose normals are loaded ahead
    extern __shared__ int32_t tab[];   // Ran2: [32][blockDim.x]
    __shared__ double red[4 * 32];
    constexpr int SW = KIND == GBRNG_TAUS ? 4 : 35;   // state words
    constexpr int CW = 6 + SW;                         // checkpoint words
    const int64_t W = (int64_t)gridDim.x * blockDim.x;
    const LdCoef c = a.c;
    const int64_t n = a.n;
    double acc[4] = {0, 0, 0, 0};
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += W) {
        const float Ki = a.Kper ? a.Kper[i] : c.K;
        const float ckx = __fmul_rn(c.ckm, Ki);
        const float hK = 0.5f * Ki;
        float x[3] = {a.x[3 * i], a.x[3 * i + 1], a.x[3 * i + 2]};
        float v[3] = {a.v[3 * i], a.v[3 * i + 1], a.v[3 * i + 2]};
        TausDraw td;
        Ran2Draw rd;
        auto load_state = [&](const float* src, int64_t stride) {
            // src == nullptr: from the generator itself
            if (KIND == GBRNG_TAUS) {
                if (!src) {
                    td.y = taus_load(a.taus[i]);
                } else {
                    td.y.x = __float_as_uint(src[0]);
                    td.y.y = __float_as_uint(src[stride]);
                    td.y.z = __float_as_uint(src[2 * stride]);
                    td.y.w = __float_as_uint(src[3 * stride]);
                }
            } else if (!src) {
                rd.load<16>(a.r2 + i, a.streams, tab, blockDim.x);
            } else {
                rd.load<16>(src, stride, tab, blockDim.x);
            }
        };
        auto save_state = [&](float* dst, int64_t stride) {
            if (KIND == GBRNG_TAUS) {
                dst[0] = __uint_as_float(td.y.x);
                dst[stride] = __uint_as_float(td.y.y);
                dst[2 * stride] = __uint_as_float(td.y.z);
                dst[3 * stride] = __uint_as_float(td.y.w);
            } else {
                rd.store<16>(dst, stride);
            }
        };
        // ---------------- A: forward with checkpoints
        // components 0 and 2 in the lanes of the paired instructions (as the transform
        // leaves their normals), component 1 by itself
        load_state(nullptr, 0);
        KahanPair lx2;   // loss, |x|^2
        float2 xp = make_float2(x[0], x[2]), vp = make_float2(v[0], v[2]);
        float xo = x[1], vo = v[1];
        const float2 cdt2 = splat2(c.cdt), cva2 = splat2(c.cva), nck2 = splat2(-ckx), cs2 = splat2(c.cs);
        for (int64_t seg = 0; seg < a.nseg; ++seg) {
            float* ck = a.ckpt + seg * CW * n + i;
            ck[0] = xp.x, ck[n] = xo, ck[2 * n] = xp.y;
            ck[3 * n] = vp.x, ck[4 * n] = vo, ck[5 * n] = vp.y;
            if (NOISE == NOISE_REGEN) save_state(ck + 6 * n, n);
            const int64_t len = min(a.P, a.S - seg * a.P);
            float* gp = a.gbuf + seg * a.P * 3 * n + i;
            for (int64_t t = 0; t < len; ++t, gp += 3 * n) {
                float g[3];
                if (KIND == GBRNG_TAUS) td.normals3(g[0], g[1], g[2]); else rd.normals3(g[0], g[1], g[2]);
                if (NOISE == NOISE_KEPT) gp[0] = g[0], gp[n] = g[1], gp[2 * n] = g[2];
                em_component2(cdt2, cva2, nck2, cs2, make_float2(g[0], g[2]), xp, vp);
                em_component(c.cdt, c.cva, ckx, c.cs, g[1], xo, vo);
                const float xx = norm2(xp.x, xo, xp.y);
                lx2.add(__fmaf_rn(hK, xx, __fmul_rn(c.hm, norm2(vp.x, vo, vp.y))), xx);
            }
        }
        // end state: the system advances exactly as ld_run would
        a.x[3 * i] = xp.x, a.x[3 * i + 1] = xo, a.x[3 * i + 2] = xp.y;
        a.v[3 * i] = vp.x, a.v[3 * i + 1] = vo, a.v[3 * i + 2] = vp.y;
        if (KIND == GBRNG_TAUS) {
            a.taus[i] = td.y;
        } else {
            rd.store<16>(a.r2 + i, a.streams);
        }
        // ---------------- B: reverse sweep
        const float inv_ab = __frcp_rn(__fmaf_rn(ckx, c.cdt, c.cva));
        const float wK = a.invS * Ki, wm = a.invS * a.m;
        const float2 ck2 = splat2(ckx), ncs2 = splat2(-c.cs), inv2 = splat2(inv_ab), ncdt2 = splat2(-c.cdt);
        const float2 c2g2 = splat2(a.c_over_2g), nckm2 = splat2(-c.ckm);
        float2 lxp = make_float2(wK * xp.x, wK * xp.y), lvp = make_float2(wm * vp.x, wm * vp.y);
        float lxo = wK * xo, lvo = wm * vo;
        KahanPair dkg;   // dK, dgamma
        Kahan dT;
        // the adjoint of the step from (xt, vt) with the normals g; its loss terms w
        auto adjoint = [&](float2 xt, float xu, float2 vt, float vu, float2 g, float gu, float k, float m) {
            const float2 pk = __fmul2_rn(lvp, xt);
            const float2 pg = __fmul2_rn(lvp, __ffma2_rn(nckm2, vt, __fmul2_rn(c2g2, g)));
            const float2 pT = __fmul2_rn(lvp, g);
            const float ddk = __fmaf_rn(lvo, xu, pk.x) + pk.y;
            const float ddg = __fmaf_rn(lvo, __fmaf_rn(-c.ckm, vu, a.c_over_2g * gu), pg.x) + pg.y;
            const float ddT = __fmaf_rn(lvo, gu, pT.x) + pT.y;
            const float2 lxn = __ffma2_rn(splat2(k), xt, __ffma2_rn(nck2, lvp, lxp));
            const float2 lvn = __ffma2_rn(splat2(m), vt, __ffma2_rn(cva2, lvp, __fmul2_rn(cdt2, lxp)));
            const float lxq = __fmaf_rn(k, xu, __fmaf_rn(-ckx, lvo, lxo));
            const float lvq = __fmaf_rn(m, vu, __fmaf_rn(c.cva, lvo, c.cdt * lxo));
            lxp = lxn, lvp = lvn, lxo = lxq, lvo = lvq;
            dkg.add(-c.ckm * ddk, ddg);
            dT.add(a.c_over_2kT * ddT);
        };
        for (int64_t seg = a.nseg - 1; seg >= 0; --seg) {
            const float* ck = a.ckpt + seg * CW * n + i;
            const int64_t len = min(a.P, a.S - seg * a.P);
            if (NOISE == NOISE_REGEN) {
                load_state(ck + 6 * n, n);
                float* gp = a.gbuf + i;
                for (int64_t t = 0; t < len; ++t, gp += 3 * n) {
                    float g[3];
                    if (KIND == GBRNG_TAUS) td.normals3(g[0], g[1], g[2]); else rd.normals3(g[0], g[1], g[2]);
                    gp[0] = g[0], gp[n] = g[1], gp[2 * n] = g[2];
                }
            }
            // x, v: the state after step t; the normals of the kAhead steps below are
            // loaded while this one is taken back
            const float* gp = a.gbuf + ((NOISE == NOISE_REGEN ? 0 : seg * a.P) + len - 1) * 3 * n + i;   // of step t
            float2 g, ga[kAhead];
            float gu, gb[kAhead];
            auto fetch = [&](int64_t d, float2& f, float& fu) {
                const float* p = gp - d * 3 * n;
                f = make_float2(p[0], p[2 * n]), fu = p[n];
            };
#pragma unroll
            for (int d = 0; d < kAhead; ++d)
                if (d < len) fetch(d, ga[d], gb[d]);
            auto back = [&](int d) {
                g = ga[d], gu = gb[d];
                vp = __fmul2_rn(__ffma2_rn(ncs2, g, __ffma2_rn(ck2, xp, vp)), inv2);
                vo = __fmaf_rn(-c.cs, gu, __fmaf_rn(ckx, xo, vo)) * inv_ab;
                xp = __ffma2_rn(ncdt2, vp, xp);
                xo = __fmaf_rn(-c.cdt, vo, xo);
            };
            int64_t t = len - 1;
            for (; t > kAhead; t -= kAhead, gp -= kAhead * 3 * n) {
#pragma unroll
                for (int d = 0; d < kAhead; ++d) {
                    back(d);
                    if (t - d >= kAhead) fetch(kAhead + d, ga[d], gb[d]);
                    adjoint(xp, xo, vp, vo, g, gu, wK, wm);
                }
            }
#pragma unroll
            for (int d = 0; d < kAhead; ++d) {
                if (t - d <= 0) break;
                back(d);
                if (t - d >= kAhead) fetch(kAhead + d, ga[d], gb[d]);
                adjoint(xp, xo, vp, vo, g, gu, wK, wm);
            }
            // step 0's normals: the t-th of those at hand
            const int d0 = t < kAhead ? (int)t : 0;
#pragma unroll
            for (int d = 0; d < kAhead; ++d)
                if (d == d0) g = ga[d], gu = gb[d];
            // the segment's start: the checkpoint holds the exact state
            xp = make_float2(ck[0], ck[2 * n]), xo = ck[n];
            vp = make_float2(ck[3 * n], ck[5 * n]), vo = ck[4 * n];
            adjoint(xp, xo, vp, vo, g, gu, seg > 0 ? wK : 0.f, seg > 0 ? wm : 0.f);
        }
        if (a.dK) a.dK[i] = (float)(dkg.first() + 0.5 * (double)a.invS * lx2.second());
        acc[0] += lx2.first() * (double)a.invS;
        acc[1] += dkg.second();
        acc[2] += dT.value();
    }
    const double sums = block_sums(acc, red);
    if (threadIdx.x < 32) store_stats(a.sink, sums);
}

// Largest noise history (bytes) ld_backward keeps; -1: half the free device
// memory at the call.
static std::atomic<int64_t> g_hist_limit{-1};

}  // namespace gb

using namespace gb;

extern "C" int ld_set_adjoint_history_limit(int64_t bytes)
{
    if (bytes < -1) return fail(GBRNG_EINVAL, "history limit must be >= -1, got %lld", (long long)bytes);
    g_hist_limit.store(bytes);
    return GBRNG_OK;
}

extern "C" int ld_backward(ld_system* sys, int64_t n_steps, int ckpt_every, float* dK_per,
                           double* dgamma, double* dkT, double* loss, void* stream)
{
    NvtxRange range("ld_backward");
    GB_CHECK(check_system(sys, true));
    Handle* h = sys->rng;
    if (h->kind != GBRNG_TAUS && h->kind != GBRNG_RAN2)
        return fail(GBRNG_EINVAL, "ld_backward needs a per-thread generator (Taus or Ran2)");
    if (n_steps < 1 || ckpt_every < 1) return fail(GBRNG_EINVAL, "need n_steps >= 1, ckpt_every >= 1");
    if (!(sys->gamma > 0) || !(sys->kT > 0)) return fail(GBRNG_EINVAL, "need gamma > 0 and kT > 0");
    cudaStream_t st = (cudaStream_t)stream;
    const int64_t n = sys->n;
    if (n == 0) {
        if (dgamma) *dgamma = 0;
        if (dkT) *dkT = 0;
        if (loss) *loss = 0;
        return GBRNG_OK;
    }
    const int64_t P = std::min<int64_t>(ckpt_every, n_steps);
    const int64_t nseg = (n_steps + P - 1) / P;
    const int SW = h->kind == GBRNG_TAUS ? 4 : 35;
    const size_t ck_bytes = sizeof(float) * (size_t)nseg * (6 + SW) * (size_t)n;
    // Noise buffer: the whole run's (12 B per oscillator-step) when it fits
    // the limit, else one segment's.  The scratch stays with the handle for
    // the next call (this call synchronises its stream before returning), and
    // the automatic limit counts what the handle already holds as free.
    const size_t hist_bytes = sizeof(float) * 3 * (size_t)n_steps * (size_t)n;
    const size_t seg_bytes = sizeof(float) * (size_t)P * 3 * (size_t)n;
    int64_t limit = g_hist_limit.load();
    if (limit < 0) {
        size_t free_b = 0, total_b = 0;
        limit = cudaMemGetInfo(&free_b, &total_b) == cudaSuccess
                    ? (int64_t)((free_b + h->adj_bytes) / 2) : 0;
        cudaGetLastError();
    }
    bool hist = n_steps > P && (int64_t)hist_bytes <= limit;
    if (hist && ensure_adj(h, ck_bytes + hist_bytes) != GBRNG_OK) hist = false;
    if (!hist) GB_CHECK(ensure_adj(h, ck_bytes + seg_bytes));
    float* scratch = h->adj;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int T = 64;
    const size_t smem = h->kind == GBRNG_RAN2 ? sizeof(int32_t) * 32 * T : 0;
    void (*fn)(AdjArgs) = h->kind == GBRNG_RAN2
        ? (hist ? adjoint_kernel<GBRNG_RAN2, NOISE_KEPT> : adjoint_kernel<GBRNG_RAN2, NOISE_REGEN>)
        : (hist ? adjoint_kernel<GBRNG_TAUS, NOISE_KEPT> : adjoint_kernel<GBRNG_TAUS, NOISE_REGEN>);
    int occ = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, T, smem);
    if (e != cudaSuccess || occ < 1) occ = 1;
    // one full resident wave at most; oscillators i, i + W, ... per thread
    const int64_t blocks = std::min<int64_t>((int64_t)di.sms * occ, (n + T - 1) / T);
    AdjArgs a;
    GB_CHECK(make_sink(h, blocks, true, &a.sink));
    a.n = n;
    a.S = n_steps;
    a.P = P;
    a.nseg = nseg;
    a.x = sys->x;
    a.v = sys->v;
    a.Kper = sys->K_per;
    a.c = make_coef(sys);
    const double cval = sqrt(2.0 * sys->gamma * sys->kT * sys->dt) / sys->m;
    a.c_over_2g = (float)(cval / (2.0 * sys->gamma));
    a.c_over_2kT = (float)(cval / (2.0 * sys->kT));
    a.invS = (float)(1.0 / (double)n_steps);
    a.m = (float)sys->m;
    a.taus = h->taus;
    a.r2 = h->r2;
    a.streams = h->n;
    a.ckpt = scratch;
    a.gbuf = scratch + ck_bytes / sizeof(float);
    a.dK = dK_per;
    fn<<<(unsigned)blocks, T, smem, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(GBRNG_ECUDA, "adjoint launch failed: %s", cudaGetErrorString(e));
    ld_stats tmp;
    GB_CHECK(finish_stats(h, a.sink, blocks, 1, &tmp, st));
    if (loss) *loss = tmp.sum_x2;
    if (dgamma) *dgamma = tmp.sum_v2;
    if (dkT) *dkT = tmp.sum_xv;
    return GBRNG_OK;
}
