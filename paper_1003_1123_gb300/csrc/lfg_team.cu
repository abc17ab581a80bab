// Langevin runs of small systems driven by the shared Lagged Fibonacci sequence
// (lfg.cuh): ld_run's oscillators and ou_run's particles.
//
// A round holds many steps of a small system, and one oscillator's draws and
// transforms of all of them are independent; only the updates follow one another.
// So a CTA's using warps first form the normals of its oscillators for every step
// of the round, spread over all lanes, into shared memory, and then a lane per
// oscillator and component (LD) or particle (OU) walks the steps, x, v (R) in
// registers for the whole launch: about 18 cycles a step (LD: the compensated
// energy sums' chain) instead of the 300 and more of a step in one thread.  The
// next round is generated meanwhile, and that and the grid barrier bound a phase:
// about 3 us (1.3 the barrier, 0.7 the loads and stores around it, the rest the
// fans' instructions).  1e4 oscillators x 1000 steps: 1513 us with a lane an
// oscillator and a barrier every third step, 338 with a lane two oscillators (the
// resident kernel) and 31 steps a round, 155 here; overdamped 1e4 particles x 1000
// steps 1250 -> 120.
#include <algorithm>

#include "lfg.cuh"

namespace gb {

enum { LFG_TEAM_LD = 0, LFG_TEAM_OU = 1 };

struct LfgTeamArgs {
    LfgArgs l;
    OuCoef oc;
    const float* R0;   // OU: R(0)
    int64_t every;     // OU: steps between records
    double* records;   // OU: [record][CTA][2] or null
    int n_c;           // oscillators of a CTA, even
};

constexpr int kTeamUse = 15, kTeamGen = 16, kTeamThreads = 32 * (kTeamUse + kTeamGen + 1);
constexpr int BAR_NORMALS = 3;

// Sums of N doubles over the using warps, sum k in lane k of the first; sm: N kTeamUse
// doubles.
template <int N>
__device__ __forceinline__ double use_sums(const double (&v)[N], double* sm)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double t = warp_sums(v);
    if (lane < N) sm[warp * N + lane] = t;
    bar_sync(BAR_NORMALS, 32 * kTeamUse);
    if (warp == 0) {
        t = 0.0;
        for (int i = lane; i < N * kTeamUse; i += 32) t += sm[i];
        t = warp_sums_strided<N>(t);
    }
    bar_sync(BAR_NORMALS, 32 * kTeamUse);
    return t;
}

template <int MODEL, int K>
__global__ void __launch_bounds__(kTeamThreads, 1) lfg_team_kernel(LfgTeamArgs o)
{
    extern __shared__ __align__(16) float team_sm[];   // [steps][normal][n_c]
    __shared__ int64_t s_failed;
    __shared__ double red[4 * kTeamUse];
    constexpr int Q = MODEL == LFG_TEAM_LD ? 3 : 1, WORDS = MODEL == LFG_TEAM_LD ? 4 : 2;   // a step's normals, draws
    constexpr int USE = 32 * kTeamUse, T = kTeamThreads;
    const LfgArgs& a = o.l;
    const int warp = threadIdx.x >> 5, n2 = o.n_c;
    const int64_t j0 = (int64_t)blockIdx.x * n2;
    const int nc = (int)max((int64_t)0, min(a.N - j0, (int64_t)n2));
    const int64_t n_rounds = (a.n_pos + a.w - 1) / a.w;
    if (threadIdx.x == 0) s_failed = kNoRound;
    __syncthreads();
    if (warp >= kTeamUse + kTeamGen) {
        wait_warp(a, n_rounds, 32 * (kTeamGen + 1), T, &s_failed);
        return;
    }
    if (warp >= kTeamUse) {
        gen_warps<K, kTeamGen>(a, warp - kTeamUse, n_rounds, T, &s_failed);
        return;
    }
    const int tid = threadIdx.x;
    // ---- the walk's lane: component q of oscillator j
    const int q = tid / n2, j = tid - q * n2;
    const bool live = q < Q && j < nc;
    const int64_t at = MODEL == LFG_TEAM_LD ? 3 * (j0 + j) + q : j0 + j;
    float x = live ? a.x[at] : 0.f, v = 0.f, nck = 0.f, hK = 0.f;
    if (MODEL == LFG_TEAM_LD && live) {
        const float k = a.Kper ? a.Kper[j0 + j] : a.c.K;
        v = a.v[at];
        nck = -__fmul_rn(a.c.ckm, k);
        hK = 0.5f * k;
    }
    const float R0 = MODEL == LFG_TEAM_OU && live ? o.R0[at] : 0.f;
    Kahan2 e;   // LD: sums of x^2 and v^2
    int64_t t = 0, rec = 0, next_rec = 0;
    auto record = [&](float Rt) {
        const double v[2] = {live ? (double)Rt : 0.0, live ? (double)Rt * (double)R0 : 0.0};
        const double sum = use_sums(v, red);
        if (tid < 2) o.records[2 * (rec * gridDim.x + blockIdx.x) + tid] = sum;
        ++rec;
        next_rec += o.every;
    };
    if (MODEL == LFG_TEAM_OU) {
        if (o.records) record(x);
        else next_rec = INT64_MAX;
    }
    // ---- the normals' lane: pairs (2i, 2i + 1) of the CTA's oscillators, from (i, s)
    // on, every USE-th of the round's pairs
    const int np = max(1, (nc + 1) >> 1);
    const int i0 = tid % np, s0 = tid / np, di = USE % np, ds = USE / np;
    const uint32_t step_slots = (uint32_t)(WORDS * a.N);
    uint32_t s_cta = slot_add(a.base_slot, (uint32_t)(WORDS * min(j0, a.N)), a.R);
    const int S = a.w / (int)step_slots;
    for (int64_t p = 0; p < n_rounds; ++p) {
        const int steps = (int)min((int64_t)S, a.n_steps - p * S);
        bar_sync(BAR_GO, T);
        if (round_failed(&s_failed, p)) return;
        if (nc > 0) {
            auto fetch = [&](int i, int s, uint4& w0, uint4& w1) {
                const uint32_t sl = slot_add(slot_add(s_cta, (uint32_t)s * step_slots, a.R), (uint32_t)(2 * WORDS * i), a.R);
                w0 = ring_quad(a, sl);
                if (MODEL == LFG_TEAM_LD) w1 = ring_quad(a, slot_add(sl, 4, a.R));
            };
            auto next = [&](int& i, int& s) {
                i += di, s += ds;
                if (i >= np) i -= np, ++s;
            };
            int i = i0, s = s0, ni = i0, ns = s0;
            uint4 w0, w1, m0, m1;
            if (s < steps) fetch(i, s, w0, w1);
            next(ni, ns);
            while (s < steps) {
                if (ns < steps) fetch(ni, ns, m0, m1);
                float* g_out = team_sm + s * Q * n2 + 2 * i;
                if constexpr (MODEL == LFG_TEAM_LD) {
                    const uint32_t r[2][4] = {{w0.x, w0.y, w0.z, w0.w}, {w1.x, w1.y, w1.z, w1.w}};
                    float2 g[3];
                    normals3x2_u32(r, g);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        *reinterpret_cast<float2*>(g_out + k * n2) = __fmul2_rn(splat2(a.c.cs), g[k]);
                } else {
                    const float2 u = make_float2(open01_from_u32(w0.x), open01_from_u32(w0.z));
                    const float2 x4 = __ffma2_rn(splat2(4.0f), make_float2(mant_from_u32(w0.y), mant_from_u32(w0.w)),
                                                 splat2(-0x1.fffffep+1f));
                    *reinterpret_cast<float2*>(g_out) = box_muller_cos2(neg2log2(u), x4);
                }
                i = ni, s = ns, w0 = m0, w1 = m1;
                next(ni, ns);
            }
        }
        bar_sync(BAR_NORMALS, USE);
        const float* g = team_sm + q * n2 + j;
        if (MODEL == LFG_TEAM_LD) {
            if (live) {
#pragma unroll 4
                for (int s = 0; s < steps; ++s) {
                    const float vn = __fmaf_rn(a.c.cva, v, __fmaf_rn(nck, x, g[s * Q * n2]));
                    x = __fmaf_rn(a.c.cdt, v, x);
                    v = vn;
                    e.add(make_float2(__fmul_rn(x, x), __fmul_rn(v, v)));
                }
            }
        } else {
            int s = 0;
            while (s < steps) {   // up to the next record, or the round's end
                const int end = (int)min((int64_t)steps, next_rec == INT64_MAX ? (int64_t)steps : s + (next_rec - t));
                const int from = s;
                if (live) {
#pragma unroll 8
                    for (; s < end; ++s) x = __fmaf_rn(o.oc.cs, g[s * n2], __fmaf_rn(-o.oc.c1, x, x));
                }
                s = end;
                t += end - from;
                if (t == next_rec) record(x);
            }
        }
        s_cta = slot_add(s_cta, (uint32_t)a.w, a.R);
    }
    if (live) {
        a.x[at] = x;
        if (MODEL == LFG_TEAM_LD) a.v[at] = v;
    }
    if (MODEL == LFG_TEAM_LD && a.sink.partials) {
        double acc[4] = {0, 0, 0, 0};
        if (live) {
            acc[0] = (double)x * x;
            acc[1] = (double)v * v;
            acc[2] = (double)x * v;
            acc[3] = (double)hK * ((double)e.s.x - (double)e.c.x) + (double)a.c.hm * ((double)e.s.y - (double)e.c.y);
        }
        const double sums = use_sums(acc, red);
        if (warp == 0) store_stats(a.sink, sums);
    }
}

// A CTA's share must give every component a lane, and several steps fit a round.
// On success a.w is set and *smem the normals' buffer.
static bool team_fits(int model, LfgArgs& a, int k, int64_t n_steps, const DevInfo& di, int* n_c, size_t* smem)
{
    const int words = model == LFG_TEAM_LD ? 4 : 2, normals = model == LFG_TEAM_LD ? 3 : 1;
    const int64_t c = ((a.N + di.sms - 1) / di.sms + 1) & ~(int64_t)1;
    if (normals * c > 32 * kTeamUse) return false;
    const int64_t step = words * a.N;
    const int64_t buffer = 160 * 1024 / (int64_t)sizeof(float) / (normals * c);   // steps that fit
    const int64_t S = std::min(std::min<int64_t>((int64_t)k * a.D / step, buffer), n_steps);
    if (S < 2) return false;
    *n_c = (int)c;
    *smem = sizeof(float) * (size_t)(S * normals * c);
    a.w = (int)(S * step);
    return true;
}

int lfg_team_ld(Handle* h, LfgArgs& a, int k, int64_t n_steps, cudaStream_t st)
{
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    LfgTeamArgs o{};
    size_t smem = 0;
    if (!team_fits(LFG_TEAM_LD, a, k, n_steps, di, &o.n_c, &smem)) return 0;
    GB_CHECK(lfg_begin(h, a, di.sms, st));
    o.l = a;
    void* args[] = {&o};
    GB_CHECK(with_depth(k, [&](auto kk) {
        return lfg_cooperative((const void*)lfg_team_kernel<LFG_TEAM_LD, decltype(kk)::value>, di.sms, kTeamThreads,
                               args, smem, st);
    }));
    return 1;
}

int lfg_team_ou(Handle* h, LfgArgs& a, int k, OuCoef c, const float* R0, int64_t n_steps, int64_t every,
                int64_t n_rec, cudaStream_t st)
{
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    LfgTeamArgs o{};
    size_t smem = 0;
    if (!team_fits(LFG_TEAM_OU, a, k, n_steps, di, &o.n_c, &smem)) return 0;
    o.oc = c;
    o.R0 = R0;
    o.every = every;
    if (n_rec) {
        GB_CHECK(ensure_partials(h, (2 * n_rec * di.sms + 2 * n_rec + 3) / 4));
        o.records = h->partials;
    }
    GB_CHECK(lfg_begin(h, a, di.sms, st));
    o.l = a;
    void* args[] = {&o};
    GB_CHECK(with_depth(k, [&](auto kk) {
        return lfg_cooperative((const void*)lfg_team_kernel<LFG_TEAM_OU, decltype(kk)::value>, di.sms, kTeamThreads,
                               args, smem, st);
    }));
    return 1;
}

}  // namespace gb
