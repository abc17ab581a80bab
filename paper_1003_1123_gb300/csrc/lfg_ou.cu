// Overdamped runs driven by the shared Lagged Fibonacci sequence (lfg.cuh): particle
// j's step t takes positions p0 + 2 (j + n t) + r, r = 0, 1.
#include <algorithm>

#include "lfg.cuh"
#include "records.h"

namespace gb {

// CTA c owns the particles [c n_c, c n_c + n_c), R and R(0) in shared memory, and a
// round holds whole steps (W = 2 N S).  A worker warp takes units of particles
// through all steps of the round.  STEPS: a lane one particle, two of its steps in
// the lanes of the paired instructions (few particles: the normals' latency
// counts); else a lane two particles.
//
// Records of the positions after t steps: each warp's sums over its units, added
// up unit by unit in its own slot records[rec][warp of the grid][2] (zeroed before
// the launch).
struct OuLfgArgs {
    LfgArgs l;
    OuCoef c;
    float* R;
    const float* R0;   // R(0): R itself, or a copy where a run takes several launches
    int64_t every;     // steps between records
    double* records;   // or null
    int n_c, slots;    // particles and record slots of a CTA
};

template <int K, int NW, int GW, bool STEPS>
__global__ void __launch_bounds__(32 * (NW + GW + 1), 1) lfg_ou_kernel(OuLfgArgs o)
{
    extern __shared__ __align__(16) float ou_sm[];   // [2][n_pad]
    __shared__ int64_t s_failed;
    constexpr int T = 32 * (NW + GW + 1), UP = STEPS ? 32 : 64, ST = STEPS ? 2 : 1;
    const LfgArgs& a = o.l;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t j0 = (int64_t)blockIdx.x * o.n_c;
    const int nc = (int)max((int64_t)0, min(a.N - j0, (int64_t)o.n_c));
    const int n_pad = (o.n_c + 63) & ~63, n_units = (nc + UP - 1) / UP;
    const int S = a.w / (int)(2 * a.N);   // steps a round
    const int64_t n_rounds = (a.n_pos + a.w - 1) / a.w;
    if (threadIdx.x == 0) s_failed = kNoRound;
    for (int i = threadIdx.x; i < nc; i += T) ou_sm[i] = o.R[j0 + i], ou_sm[n_pad + i] = o.R0[j0 + i];
    __syncthreads();
    if (warp >= NW + GW) {
        wait_warp(a, n_rounds, 32 * (GW + 1), T, &s_failed);
    } else if (warp >= NW) {
        gen_warps<K, GW>(a, warp - NW, n_rounds, T, &s_failed);
    } else {
        // sums of positions Ra (and Rb) of the unit at lane's particle j into record rec
        auto record = [&](int64_t rec, int u, int j, float Ra, float Rb) {
            const float* R0 = ou_sm + n_pad + j;
            double v[2] = {j < nc ? (double)Ra : 0.0, j < nc ? (double)Ra * (double)R0[0] : 0.0};
            if (!STEPS && j + 1 < nc) v[0] += (double)Rb, v[1] += (double)Rb * (double)R0[1];
            const double sum = warp_sums(v);
            if (lane < 2) {
                double* d = o.records + 2 * ((rec * gridDim.x + blockIdx.x) * o.slots + warp) + lane;
                *d = u == warp ? sum : *d + sum;
            }
        };
        if (o.records)
            for (int u = warp; u < n_units; u += NW) {
                const int j = UP * u + (STEPS ? lane : 2 * lane);
                record(0, u, j, ou_sm[j], STEPS ? 0.f : ou_sm[j + 1]);
            }
        // slot of this warp's first unit in the round's first step
        uint32_t s_first = slot_add(slot_add(a.base_slot, (uint32_t)(2 * min(j0, a.N)), a.R),
                                    (uint32_t)(2 * UP * min(warp, n_units)), a.R);
        const uint32_t step_slots = (uint32_t)(2 * a.N);
        auto fetch = [&](uint32_t ss) {
            if (!STEPS) return ring_quad(a, slot_add(ss, (uint32_t)(4 * lane), a.R));
            const uint32_t sl = slot_add(ss, (uint32_t)(2 * lane), a.R);
            const uint2 x = ring_two(a, sl), y = ring_two(a, slot_add(sl, step_slots, a.R));
            return make_uint4(x.x, x.y, y.x, y.y);
        };
        for (int64_t p = 0; p < n_rounds; ++p) {
            const int steps = (int)min((int64_t)S, a.n_steps - p * S);
            // first record of the phase: its number, and the steps of the phase taken by then
            const int64_t rec0 = p * S / o.every + 1, at0 = rec0 * o.every - p * S;
            bar_sync(BAR_GO, T);
            if (round_failed(&s_failed, p)) break;
            uint32_t su = s_first;
            uint4 w;   // raw words are loaded one item ahead
            if (warp < n_units) w = fetch(su);
#pragma unroll 1
            for (int u = warp; u < n_units; u += NW) {
                const int j = UP * u + (STEPS ? lane : 2 * lane);
                float Ra = ou_sm[j], Rb = STEPS ? 0.f : ou_sm[j + 1];
                int64_t rec = rec0, at = at0;
                uint32_t ss = su;
                su = u + NW < n_units ? slot_add(su, (uint32_t)(2 * UP * NW), a.R) : su;
#pragma unroll 1
                for (int s = 0; s < steps; s += ST) {
                    ss = slot_add(ss, step_slots, a.R);
                    if (STEPS) ss = slot_add(ss, step_slots, a.R);
                    if (s + ST >= steps) ss = su;
                    const uint4 n = fetch(ss);
                    const float2 us = make_float2(open01_from_u32(w.x), open01_from_u32(w.z));
                    const float2 x4 = __ffma2_rn(splat2(4.0f), make_float2(mant_from_u32(w.y), mant_from_u32(w.w)),
                                                 splat2(-0x1.fffffep+1f));
                    const float2 g = box_muller_cos2(neg2log2(us), x4);
                    Ra = __fmaf_rn(o.c.cs, g.x, __fmaf_rn(-o.c.c1, Ra, Ra));
                    if (!STEPS) Rb = __fmaf_rn(o.c.cs, g.y, __fmaf_rn(-o.c.c1, Rb, Rb));
                    if (o.records && s + 1 == at) record(rec++, u, j, Ra, Rb), at += o.every;
                    if (STEPS && s + 1 < steps) {
                        Ra = __fmaf_rn(o.c.cs, g.y, __fmaf_rn(-o.c.c1, Ra, Ra));
                        if (o.records && s + 2 == at) record(rec++, u, j, Ra, Rb), at += o.every;
                    }
                    w = n;
                }
                ou_sm[j] = Ra;
                if (!STEPS) ou_sm[j + 1] = Rb;
            }
            s_first = slot_add(s_first, (uint32_t)a.w, a.R);
        }
    }
    __syncthreads();
    if (s_failed != kNoRound) return;
    for (int i = threadIdx.x; i < nc; i += T) o.R[j0 + i] = ou_sm[i];
}

constexpr int kOuGen = 16;

// One launch: n_steps steps, records after 0, every, ... of them.
static int launch_ou(const ou_system* s, const float* R0, int64_t n_steps, int64_t every, double* mean, double* corr,
                     cudaStream_t st)
{
    Handle* h = s->rng;
    const int64_t two_n = 2 * s->n, D = (int64_t)h->ll - h->sl;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int64_t G = di.sms;
    const bool rec = mean != nullptr;
    const int64_t n_rec = n_steps / every + 1;
    // the depth set may be below the width a step needs (whole quads): no deeper than D allows
    const int k = lfg_depth(h);
    OuLfgArgs o{};
    o.l = lfg_args(h);
    o.l.N = s->n;
    o.l.n_steps = n_steps;
    o.l.n_pos = two_n * n_steps;
    o.l.vec = o.l.vec && s->n % 2 == 0;   // every step from a multiple of 4 on
    o.l.x = s->R;
    if (const int rc = lfg_team_ou(h, o.l, k, make_ou_coef(s), R0, n_steps, every, rec ? n_rec : 0, st)) {
        if (rc < 0) return rc;
        GB_CHECK(lfg_end(h, o.l, st));
        h->pos += o.l.n_pos;
        return rec ? ou_finish(h, s->n, n_rec, G, mean, corr, st) : GBRNG_OK;
    }
    const int64_t S = std::max<int64_t>(1, std::min<int64_t>(k * D / two_n, n_steps));
    o.l.w = (int)(two_n * S);
    o.c = make_ou_coef(s);
    o.R = s->R;
    o.R0 = R0;
    o.every = every;
    o.n_c = (int)lfg_share(s->n, di.sms);
    const bool steps = S >= 4 && o.n_c <= 32 * kOuWarps * 2;
    o.slots = lfg_record_slots(o.n_c, steps ? 32 : 64);
    if (rec) {
        const int64_t blocks = G * o.slots;
        GB_CHECK(ensure_partials(h, (2 * n_rec * blocks + 2 * n_rec + 3) / 4));
        GB_CUDA(cudaMemsetAsync(h->partials, 0, sizeof(double) * 2 * n_rec * blocks, st));
        o.records = h->partials;
    }
    if (n_steps > 0 || rec) {
        GB_CHECK(lfg_begin(h, o.l, G, st));
        const size_t smem = sizeof(float) * 2 * (size_t)((o.n_c + 63) & ~63);
        void* args[] = {&o};
        GB_CHECK(with_depth(k, [&](auto kk) {
            constexpr int K = decltype(kk)::value;
            const void* fn = steps ? (const void*)lfg_ou_kernel<K, kOuWarps, kOuGen, true>
                                   : (const void*)lfg_ou_kernel<K, kOuWarps, kOuGen, false>;
            return lfg_cooperative(fn, G, 32 * (kOuWarps + kOuGen + 1), args, smem, st);
        }));
        GB_CHECK(lfg_end(h, o.l, st));
        h->pos += o.l.n_pos;
    }
    if (rec) return ou_finish(h, s->n, n_rec, G * o.slots, mean, corr, st);
    return GBRNG_OK;
}

int lfg_ou(const ou_system* s, int64_t n_steps, int64_t every, double* mean, double* corr, cudaStream_t st)
{
    Handle* h = s->rng;
    const int64_t two_n = 2 * s->n, D = (int64_t)h->ll - h->sl;
    if (two_n > lfg_step_width(h))
        return fail(GBRNG_ELAGS,
                    "one round per step needs 2N = %lld within %d times the lag distance "
                    "(ll - sl = %lld)",
                    (long long)two_n, lfg_step_order(h), (long long)D);
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int64_t n_rec = n_steps / every + 1;
    if (mean && records_refused(n_rec, lfg_record_blocks(s->n, di.sms, lfg_step_order(h))))
        return fail(GBRNG_EINVAL, "%lld records of %lld particles exceed the record scratch", (long long)n_rec,
                    (long long)s->n);
    const int64_t most = lfg_launch_records(s->n, di.sms);
    if (!mean || n_rec <= most) return launch_ou(s, s->R, n_steps, every, mean, corr, st);
    // launches of `most` records, the first of each the last of the one before, all against
    // R(0) of the run
    GB_CHECK(ensure_eacc(h, s->n));
    float* R0 = reinterpret_cast<float*>(h->eacc);
    GB_CUDA(cudaMemcpyAsync(R0, s->R, sizeof(float) * s->n, cudaMemcpyDeviceToDevice, st));
    for (int64_t r = 0; r < n_rec - 1; r += most - 1) {
        const int64_t left = n_steps - r * every;
        const int64_t steps = r + most - 1 < n_rec - 1 ? (most - 1) * every : left;
        GB_CHECK(launch_ou(s, R0, steps, every, mean + r, corr + r, st));
    }
    return GBRNG_OK;
}

}  // namespace gb
