// Fused Langevin dynamics for the per-thread generators (Hybrid Taus, Ran2):
// one persistent launch runs every step of every oscillator.  A thread owns
// oscillators i = g, g + W, g + 2W, ... (W = threads in the grid) and, for
// each, keeps x, v, K_i and the generator state in registers (Ran2's shuffle
// table in a shared-memory column) for all n_steps; per step it draws four
// uniforms, forms three Box-Muller normals, applies the Euler-Maruyama update
// and accumulates |x|^2 and |v|^2 for the time-summed energy.  State goes back to global memory once.
#include <algorithm>

#include "device.cuh"
#include "internal.cuh"

namespace gb {

struct LdArgs {
    int64_t n, n_steps;
    float* x;
    float* v;
    const float* Kper;
    LdCoef c;
    uint4* taus;       // Taus state [streams]
    int32_t* r2;       // Ran2 state [35][streams]
    uint32_t* lcg;     // LCG state [streams]
    int64_t S;         // streams of the generator (row stride of r2)
    StatsSink sink;
};

// Register budget (128-thread blocks per SM, measured at 1e6 oscillators):
// Hybrid Taus and Ran2 six (up to 85 registers, no spills; Taus 1% and Ran2 5%
// faster than ten and nine blocks at 48 and 56 registers, which spilled), the
// LCG seven (5% faster than ten).
template <int KIND, bool INIT>
__global__ void __launch_bounds__(128, KIND == GBRNG_LCG ? 7 : 6) ld_pt_kernel(LdArgs a)
{
    extern __shared__ int32_t tab[];   // Ran2: [32][blockDim.x]
    __shared__ double red[4 * 32];
    const int64_t W = (int64_t)gridDim.x * blockDim.x;
    const LdCoef c = a.c;
    double acc[4] = {0, 0, 0, 0};      // sum x^2, v^2, x.v, energy
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < a.n; i += W) {
        const float Ki = a.Kper ? a.Kper[i] : c.K;
        float x0, x1, x2, v0, v1, v2;
        if (!INIT) {
            x0 = a.x[3 * i], x1 = a.x[3 * i + 1], x2 = a.x[3 * i + 2];
            v0 = a.v[3 * i], v1 = a.v[3 * i + 1], v2 = a.v[3 * i + 2];
        }
        TausDraw td;
        LcgDraw lc;
        Ran2Draw rd;
        if (KIND == GBRNG_TAUS) {
            td.y = taus_load(a.taus[i]);
        } else if (KIND == GBRNG_LCG) {
            lc.x = a.lcg[i];
        } else {
            rd.load(a.r2 + i, a.S, tab, 32);
        }
        EnergySum es;
        float hK = 0.f;
        if (INIT) {
            // draw-step 0 -> x = sqrt(kT/K_i) g, draw-step 1 -> v = sqrt(kT/m) g
            float g0, g1, g2;
            draw3<KIND>(td, lc, rd, g0, g1, g2);
            const float sx = __fsqrt_rn(__fdiv_rn(c.kT, Ki));
            x0 = __fmul_rn(sx, g0), x1 = __fmul_rn(sx, g1), x2 = __fmul_rn(sx, g2);
            draw3<KIND>(td, lc, rd, g0, g1, g2);
            v0 = __fmul_rn(c.sv, g0), v1 = __fmul_rn(c.sv, g1), v2 = __fmul_rn(c.sv, g2);
        } else {
            const float ckx = __fmul_rn(c.ckm, Ki);
            hK = 0.5f * Ki;
            for (int64_t t0 = 0; t0 < a.n_steps; t0 += kEnergyBlock) {
                const int nb = (int)min((int64_t)kEnergyBlock, a.n_steps - t0);
                // steps an iteration: the LCG 3% faster with two; Ran2, whose next
                // draws' chain then runs beside a step's transforms, with eight (1000
                // oscillators x 1000 steps 195 -> 191 us, 5e4 365 -> 351); Taus loses 1-2%
#pragma unroll(KIND == GBRNG_LCG ? 2 : KIND == GBRNG_RAN2 ? 8 : 1)
                for (int k = 0; k < nb; ++k) {
                    float g0, g1, g2;
                    draw3<KIND>(td, lc, rd, g0, g1, g2);
                    em_component(c.cdt, c.cva, ckx, c.cs, g0, x0, v0);
                    em_component(c.cdt, c.cva, ckx, c.cs, g1, x1, v1);
                    em_component(c.cdt, c.cva, ckx, c.cs, g2, x2, v2);
                    es.add(x0, x1, x2, v0, v1, v2);
                }
                es.flush();
            }
        }
        a.x[3 * i] = x0, a.x[3 * i + 1] = x1, a.x[3 * i + 2] = x2;
        a.v[3 * i] = v0, a.v[3 * i + 1] = v1, a.v[3 * i + 2] = v2;
        if (!INIT && a.n_steps == 0) {
            // nothing drawn: the state as it stands
        } else if (KIND == GBRNG_TAUS) {
            a.taus[i] = td.y;
        } else if (KIND == GBRNG_LCG) {
            a.lcg[i] = lc.x;
        } else {
            rd.store(a.r2 + i, a.S);
        }
        acc[0] += (double)x0 * x0 + (double)x1 * x1 + (double)x2 * x2;
        acc[1] += (double)v0 * v0 + (double)v1 * v1 + (double)v2 * v2;
        acc[2] += (double)x0 * v0 + (double)x1 * v1 + (double)x2 * v2;
        acc[3] += es.value(hK, c.hm);
    }
    if (a.sink.partials) {
        const double sums = block_sums(acc, red);
        if (threadIdx.x < 32) store_stats(a.sink, sums);
    }
}

// Two oscillators a thread (Hybrid Taus, the LCG, Ran2): thread g takes the
// adjacent pairs (2p, 2p + 1) for p = g, g + W, ..., and advances both in the
// same loop, several steps an iteration, so each thread carries two independent
// generator chains, and the two oscillators' floating-point work (transforms,
// update, energy sums) runs in the two lanes of the paired binary32
// instructions.  One-warp blocks, one full resident wave; Ran2's two tables in
// shared-memory columns.  Per oscillator the draws, operations and state are
// those of ld_pt_kernel, bit for bit; only the order of the final sums over
// oscillators differs.
template <int KIND>
__global__ void __launch_bounds__(32) ld_pair_kernel(LdArgs a, int64_t n_pairs)
{
    extern __shared__ int32_t tab[];   // Ran2: [2][32][blockDim.x], one table per lane oscillator
    __shared__ double red[4 * 32];
    const int64_t W = (int64_t)gridDim.x * blockDim.x;
    const LdCoef c = a.c;
    double acc[4] = {0, 0, 0, 0};
    const float2 cdt = splat2(c.cdt), cva = splat2(c.cva), cs = splat2(c.cs);
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n_pairs; p += W) {
        int64_t idx[2];
        bool live[2];
        // lane j of every pair below is oscillator 2p + j
        float2 X[3], V[3], nckx;
        float hK[2];
        TausDraw td[2];
        LcgDraw lc[2];
        Ran2Draw rd[2];
        EnergySum2 es;
        float xs[2][3], vs[2][3], ck[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            idx[j] = 2 * p + j;
            live[j] = idx[j] < a.n;
            const int64_t i = live[j] ? idx[j] : 2 * p;   // a dead second lane shadows the first
            const float Ki = a.Kper ? a.Kper[i] : c.K;
            ck[j] = -__fmul_rn(c.ckm, Ki);
            hK[j] = 0.5f * Ki;
#pragma unroll
            for (int q = 0; q < 3; ++q) xs[j][q] = a.x[3 * i + q], vs[j][q] = a.v[3 * i + q];
            if (KIND == GBRNG_TAUS) {
                td[j].y = taus_load(a.taus[i]);
            } else if (KIND == GBRNG_LCG) {
                lc[j].x = a.lcg[i];
            } else {
                rd[j].load<16>(a.r2 + i, a.S, tab + j * 32 * blockDim.x, 32);
            }
        }
        nckx = make_float2(ck[0], ck[1]);
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            X[q] = make_float2(xs[0][q], xs[1][q]);
            V[q] = make_float2(vs[0][q], vs[1][q]);
        }
        for (int64_t t0 = 0; t0 < a.n_steps; t0 += kEnergyBlock) {
            const int nb = (int)min((int64_t)kEnergyBlock, a.n_steps - t0);
            // steps an iteration: Hybrid Taus 4.33 ms with two and converted exponents,
            // 4.09 with two, 4.05 with eight (1e6 x 1000); the LCG 3.15 and Ran2 6.04 with
            // two, 3.11 and 5.96 with four, 3.11 and 6.13 with eight; since its two
            // oscillators draw side by side Ran2 takes 5.23, 5.19 and 5.26
#pragma unroll(KIND == GBRNG_TAUS ? 8 : 4)
            for (int k = 0; k < nb; ++k) {
                float2 g[3];
                draw3x2<KIND>(td, lc, rd, g);
#pragma unroll
                for (int q = 0; q < 3; ++q) em_component2(cdt, cva, nckx, cs, g[q], X[q], V[q]);
                es.add(X, V);
            }
            es.flush();
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (!live[j]) continue;
            const int64_t i = idx[j];
            const float x0 = j ? X[0].y : X[0].x, x1 = j ? X[1].y : X[1].x, x2 = j ? X[2].y : X[2].x;
            const float v0 = j ? V[0].y : V[0].x, v1 = j ? V[1].y : V[1].x, v2 = j ? V[2].y : V[2].x;
            a.x[3 * i] = x0, a.x[3 * i + 1] = x1, a.x[3 * i + 2] = x2;
            a.v[3 * i] = v0, a.v[3 * i + 1] = v1, a.v[3 * i + 2] = v2;
            if (a.n_steps == 0) {
                // nothing drawn: the state as it stands
            } else if (KIND == GBRNG_TAUS) {
                a.taus[i] = td[j].y;
            } else if (KIND == GBRNG_LCG) {
                a.lcg[i] = lc[j].x;
            } else {
                rd[j].store<16>(a.r2 + i, a.S);
            }
            acc[0] += (double)x0 * x0 + (double)x1 * x1 + (double)x2 * x2;
            acc[1] += (double)v0 * v0 + (double)v1 * v1 + (double)v2 * v2;
            acc[2] += (double)x0 * v0 + (double)x1 * v1 + (double)x2 * v2;
            acc[3] += es.value(j, hK[j], c.hm);
        }
    }
    if (a.sink.partials) {
        const double sums = block_sums(acc, red);
        if (threadIdx.x < 32) store_stats(a.sink, sums);
    }
}

// Pair-kernel grid: one full resident wave of one-warp blocks (16 a SM for
// Taus, 20 for Ran2 at 1e6 oscillators), fewer where the pairs do not fill it.
// Measured at 1e6 oscillators x 1000 steps (scalar arithmetic): 5.90 ms for
// Hybrid Taus against 6.13 ms for one oscillator a thread; 64-, 128- and
// 256-thread blocks 6.06-6.60 ms; a grid trimmed so that every thread gets the
// same number of pairs (fewer warps a SM) 6.36 ms.  With the paired
// instructions: Taus 4.05 ms, Ran2 5.19 ms.
template <int KIND>
static int launch_pairs(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    Handle* h = s->rng;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int T = 32;
    const size_t smem = KIND == GBRNG_RAN2 ? sizeof(int32_t) * 2 * 32 * T : 0;
    int occ = 0;
    GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ld_pair_kernel<KIND>, T, smem));
    if (occ < 1) occ = 1;
    const int64_t pairs = (s->n + 1) / 2;
    const int64_t blocks = std::min<int64_t>((int64_t)di.sms * occ, (pairs + T - 1) / T);
    LdArgs a;
    a.n = s->n;
    a.n_steps = n_steps;
    a.x = s->x;
    a.v = s->v;
    a.Kper = s->K_per;
    a.c = make_coef(s);
    a.taus = h->taus;
    a.r2 = h->r2;
    a.lcg = h->lcg;
    a.S = h->n;
    GB_CHECK(make_sink(h, blocks, out != nullptr, &a.sink));
    ld_pair_kernel<KIND><<<(unsigned)blocks, T, smem, st>>>(a, pairs);
    GB_CUDA(cudaGetLastError());
    return finish_stats(h, a.sink, blocks, n_steps, out, st);
}

// Grid shape: threads per block T and one full resident wave (SMs x blocks
// per SM, fewer only when the system has fewer oscillators than that wave has
// threads).  Thread g takes oscillators g, g + W, ...; the last, partial round
// then falls on the lowest blocks, which the block scheduler spreads over all
// SMs, so every SM carries the same work to within one block's round.  (A grid
// cut to ceil(n / (oscillators per thread x T)) blocks leaves some SMs a block
// short and others a block over, about 9% apart at 1e6 oscillators.)
template <int KIND, bool INIT>
static int launch_ld(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    Handle* h = s->rng;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    int T = 128;
    // one-warp blocks spread small systems over all SMs, and are 1% faster for
    // Ran2 at any size (25 warps a SM at 79 registers)
    if (s->n < (int64_t)di.sms * 128 * 2 || KIND == GBRNG_RAN2) T = 32;
    const size_t smem = KIND == GBRNG_RAN2 ? sizeof(int32_t) * 32 * T : 0;
    int occ = 0;
    GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ld_pt_kernel<KIND, INIT>, T, smem));
    if (occ < 1) occ = 1;
    int64_t blocks = std::min<int64_t>((int64_t)di.sms * occ, (s->n + T - 1) / T);
    if (blocks < 1) blocks = 1;
    LdArgs a;
    a.n = s->n;
    a.n_steps = n_steps;
    a.x = s->x;
    a.v = s->v;
    a.Kper = s->K_per;
    a.c = make_coef(s);
    a.taus = h->taus;
    a.r2 = h->r2;
    a.lcg = h->lcg;
    a.S = h->n;
    GB_CHECK(make_sink(h, blocks, out != nullptr, &a.sink));
    ld_pt_kernel<KIND, INIT><<<(unsigned)blocks, T, smem, st>>>(a);
    GB_CUDA(cudaGetLastError());
    return finish_stats(h, a.sink, blocks, n_steps, out, st);
}

int ld_init_pt(const ld_system* s, cudaStream_t st)
{
    if (s->rng->kind == GBRNG_TAUS) return launch_ld<GBRNG_TAUS, true>(s, 0, nullptr, st);
    if (s->rng->kind == GBRNG_LCG) return launch_ld<GBRNG_LCG, true>(s, 0, nullptr, st);
    return launch_ld<GBRNG_RAN2, true>(s, 0, nullptr, st);
}

// Which kernel runs a system.  A run's time is the steps' times the time of a
// step, which for the thread-per-oscillator kernels goes by the warps on the
// busiest scheduler (w1 with one oscillator a thread, w2 with two) and for the
// teams by the oscillators a SM holds, besides their start-up (the jumps).  The
// costs are measured, ns a step over 3000 steps, one a thread by w1, two a thread by w2;
// teams with statistics repeat every update in their producer warps, a fifth more a step
// (the thread-per-oscillator kernels sum the energies in any case).  Without that in the
// rule, runs with statistics took a team too far: 1.1e5 LCG oscillators 522 ns a step instead
// of 365 by two a thread, 58368 257 instead of 198 by one.  Above w1 = 8 two a thread.
enum LdPath { LD_ONE, LD_PAIRS, LD_TEAM };
struct LdCost {
    double one[8], pairs[4], pairs_start;
    // ns: a step, and per oscillator a SM; the start, and per oscillator
    struct Team {
        double step0, step, start0, start;
    } team[2];   // without statistics, with
};
constexpr LdCost kCostTaus = {{113, 188, 286, 375, 467, 557, 649, 739}, {175, 320, 471, 621}, 1500,
                              {{4, 0.755, 1500, 0.3}, {5, 0.89, 6000, 0.44}}};
constexpr LdCost kCostLcg = {{86, 132, 198, 259, 320, 382, 443, 504}, {151, 246, 365, 477}, 1500,
                             {{3, 0.56, 1000, 0.18}, {4, 0.665, 4000, 0.34}}};
constexpr LdCost kCostRan2 = {{183, 245, 340, 440, 537, 631, 729, 824}, {266, 418, 615, 800}, 400,
                              {{1e300, 0, 0, 0}, {1e300, 0, 0, 0}}};   // no team

static LdPath pick_path(int kind, int64_t n, int64_t n_steps, bool stats, int sms)
{
    const int64_t w1 = (n + 128ll * sms - 1) / (128ll * sms), w2 = (n + 256ll * sms - 1) / (256ll * sms);
    if (w1 > 8) return LD_PAIRS;
    const LdCost& c = kind == GBRNG_TAUS ? kCostTaus : kind == GBRNG_LCG ? kCostLcg : kCostRan2;
    const LdCost::Team& t = c.team[stats];
    const double steps = (double)n_steps;
    // the blocks' sums, added up by the last block or by a second kernel
    auto sums = [&](int64_t blocks) { return !stats ? 0.0 : blocks <= kFuseBlocks ? 11.5 * (double)blocks : 4000.0; };
    const double one = c.one[w1 - 1] * steps + sums(n / (w1 <= 2 || kind == GBRNG_RAN2 ? 32 : 128));
    const double pairs = c.pairs[w2 - 1] * steps + c.pairs_start + sums(n / 64);
    // a start counts in full up to some 80 steps; in long runs the blocks drift apart, and the
    // jumps of one pass beside another's steps: less than nothing from 290 on
    const double seen = std::min(1.0, std::max(-0.35, 1.0 - (steps - 80.0) / 210.0));
    const double team = (t.step0 + t.step * (double)n / sms) * steps + (t.start0 + t.start * (double)n) * seen;
    if (n_steps > 0 && team < std::min(one, pairs)) return LD_TEAM;
    return pairs < one ? LD_PAIRS : LD_ONE;
}

template <int KIND>
static int run_kind(const ld_system* s, LdPath path, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    if (path == LD_PAIRS) return launch_pairs<KIND>(s, n_steps, out, st);
    return launch_ld<KIND, false>(s, n_steps, out, st);
}

int ld_run_pt(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    if (s->n == 0) {
        if (out) *out = ld_stats{0, 0, 0, 0, n_steps};
        return GBRNG_OK;
    }
    DevInfo di;
    GB_CHECK(dev_info(s->rng->device, &di));
    const LdPath path = pick_path(s->rng->kind, s->n, n_steps, out != nullptr, di.sms);
    if (path == LD_TEAM) return ld_team(s, n_steps, out, st);
    if (s->rng->kind == GBRNG_TAUS) return run_kind<GBRNG_TAUS>(s, path, n_steps, out, st);
    if (s->rng->kind == GBRNG_LCG) return run_kind<GBRNG_LCG>(s, path, n_steps, out, st);
    return run_kind<GBRNG_RAN2>(s, path, n_steps, out, st);
}

}  // namespace gb
