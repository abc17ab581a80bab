// Langevin runs of systems too small to fill the GPU with one oscillator a
// thread (Hybrid Taus and the LCG): ld_run's oscillators and ou_run's particles.
//
// A step's update is a short dependent chain (three fused multiply-adds a
// component), but the draws and transforms before it are about 270 cycles of
// latency in one thread: with few oscillators that latency is the run's time and
// most of the chip idles.  Here a block runs G oscillators.  Its producer warps
// generate the normals of many steps at once, each lane those of two oscillators
// (in the lanes of the paired binary32 instructions) over a chunk of consecutive
// steps, its generators jumped ahead to the chunk's first draw (jump.cuh: the same
// words as stepping there).  One consumer warp, a lane per oscillator (or two) and
// component, walks the steps in order, reading the normals from shared memory:
// about 10 cycles a step.  Draws, transforms and update are those of the other
// kernels operation for operation, so x, v, R and the generator states come out
// bit for bit the same.
//
// Energies (runs with statistics).  The consumer leaves x and v at each chunk's
// start; once a stage is consumed, each producer lane repeats the updates of its
// own chunk from there (the normals are still in place) and sums |x|^2 and |v|^2
// over it: a chunk is one block of 16 steps of the other kernels' energy sums, so
// the consumer, adding the chunks' sums up in time order, gets the same bits.
//
// The chunks of one pass over the buffer are dealt to the stages in time order.
// A stage is filled by M warps, handed to the consumer by a named barrier, and
// handed back by another, so the producers refill it as soon as it is consumed.
//
// Two shapes, of 55 KB each (four blocks a SM).  16 oscillators a block (16 chunks a
// pass) and, for the fewest oscillators, 8 a block (32 chunks), which spreads the
// consumers' chains wider.  Hybrid Taus x 1000 steps, one oscillator a thread /
// 16 a block / 8 a block, us: 1000 oscillators 119 / 22.6 / 14.5; 4096 119 / 32.9
// / 32.9; 1e4 119 / 67.7 / 63.6; 2e4 193 / 113 / 112; 5.8e4 287 / 287 (bound there by
// the issue of the instructions that one oscillator a thread does not need, the jumps and
// the hand-over).  With statistics a step costs a fifth more: 1e4 66 ns instead of 55, 5.8e4
// 343 instead of 291, where one oscillator a thread takes 286 either way.
#include <algorithm>
#include <type_traits>

#include "jump.cuh"
#include "internal.cuh"
#include "records.h"

namespace gb {

constexpr int kStages = 4;
// Named barriers: stage s filled, 1 + s; stage s consumed, 1 + kStages + s; every
// producer warp has loaded the generators' states.
constexpr int BAR_LOADED = 1 + 2 * kStages;

// What a team runs: the 3-D oscillators of ld_run or the overdamped particles of
// ou_run.
enum { TEAM_LD = 0, TEAM_OU = 1 };

struct TeamArgs {
    int64_t n, n_steps;
    float* x;           // LD: x; OU: R
    float* v;
    const float* Kper;
    LdCoef c;
    OuCoef oc;
    int64_t every;      // OU: steps between records
    uint4* taus;
    uint32_t* lcg;
    StatsSink sink;     // LD
    double* records;    // OU: [record][gridDim.x][2] or null
};

// PAIRS: oscillator pairs of a block; M: producer warps a stage.
template <int MODEL, int PAIRS, int M>
struct TeamShape {
    static constexpr int kOsc = 2 * PAIRS;
    static constexpr int kNormals = MODEL == TEAM_LD ? 3 : 1;              // a step
    static constexpr int kChunk = MODEL == TEAM_LD ? 16 : 32;              // steps
    static constexpr int kChunkDraws = kChunk * (MODEL == TEAM_LD ? 4 : 2);   // of one stream
    static constexpr int kSub = 32 / PAIRS;                                // chunks of one warp
    static constexpr int kStageSteps = M * kSub * kChunk;
    static constexpr int kChunks = kStages * M * kSub;                     // chunks of one pass
    static constexpr int kPassSteps = kChunks * kChunk;
    static constexpr int kStepWords = kNormals * kOsc;
    // LD: x, v [2][3][kOsc] at the chunk's start, then sum |x|^2, |v|^2 [2][kOsc]
    static constexpr int kStateWords = MODEL == TEAM_LD ? 6 * kOsc : 0;
    static_assert(MODEL != TEAM_LD || kChunk == kEnergyBlock, "a chunk is an energy block");
    // a half-warp's stores of one normal go to 16 / PAIRS chunks: padding a
    // chunk so that they start on different banks
    static constexpr int kChunkWords = kChunk * kStepWords + kStateWords + kOsc;
    static constexpr int kProducers = 32 * kStages * M, kThreads = kProducers + 32;
    static constexpr size_t kBufBytes = sizeof(float) * kChunks * kChunkWords;
};

// The cosine-branch normals of one step of two particles (lane j = particle j),
// each lane ou_run's transform.
template <int KIND>
__device__ __forceinline__ float2 draw_cos2(TausDraw (&td)[2], LcgDraw (&lc)[2])
{
    uint32_t r[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        if (KIND == GBRNG_TAUS)
            taus_draws(td[j].y, r[j]);
        else
            lcg_draws(lc[j].x, r[j]);
    }
    const float2 u = make_float2(open01_from_u32(r[0][0]), open01_from_u32(r[1][0]));
    const float2 x = __ffma2_rn(splat2(4.0f), make_float2(mant_from_u32(r[0][1]), mant_from_u32(r[1][1])),
                                splat2(-0x1.fffffep+1f));
    return box_muller_cos2(neg2log2(u), x);
}

// em_component with cs g formed beforehand: of one oscillator, or of two in the
// lanes of the paired instructions.
__device__ __forceinline__ void team_update(float cdt, float cva, float nck, float csg, float& x, float& v)
{
    const float vn = __fmaf_rn(cva, v, __fmaf_rn(nck, x, csg));
    x = __fmaf_rn(cdt, v, x);
    v = vn;
}
__device__ __forceinline__ void team_update(float2 cdt, float2 cva, float2 nck, float2 csg, float2& x, float2& v)
{
    const float2 vn = __ffma2_rn(cva, v, __ffma2_rn(nck, x, csg));
    x = __ffma2_rn(cdt, v, x);
    v = vn;
}

// Producer warp: the normals of its chunks, pass after pass, and the generators'
// end state.
template <int MODEL, int KIND, class S>
__device__ __forceinline__ void team_produce(const TeamArgs& a, float* buf, int bar_threads)
{
    constexpr int G = S::kOsc, PAIRS = G / 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int stage = warp * S::kSub / (S::kChunks / kStages), pair = lane % PAIRS;
    const int chunk = warp * S::kSub + lane / PAIRS;   // of a pass, in time order
    const int64_t first = blockIdx.x * (int64_t)G;
    TausDraw td[2];
    LcgDraw lc[2];
    Ran2Draw rd[2];
    int64_t idx[2];
    bool live[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        idx[j] = first + 2 * pair + j;
        live[j] = idx[j] < a.n;
        const int64_t i = live[j] ? idx[j] : first;   // a dead lane shadows the block's first
        if (KIND == GBRNG_TAUS)
            td[j].y = taus_load(a.taus[i]);
        else
            lc[j].x = a.lcg[i];
    }
    // every producer warp reads these words, and the one with the run's last chunk
    // replaces them: no warp goes on, or leaves, before all have them
    bar_sync(BAR_LOADED, S::kProducers);
    // to the chunk's first draw: 2^l chunks ahead for every bit l of its number
    auto jump = [&](auto d) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (KIND == GBRNG_TAUS)
                jump_ahead<decltype(d)::value>(td[j].y);
            else
                jump_ahead<decltype(d)::value>(lc[j].x);
        }
    };
    constexpr uint64_t D = S::kChunkDraws;
    if (chunk & 1) jump(std::integral_constant<uint64_t, D>{});
    if (chunk & 2) jump(std::integral_constant<uint64_t, 2 * D>{});
    if (chunk & 4) jump(std::integral_constant<uint64_t, 4 * D>{});
    if (chunk & 8) jump(std::integral_constant<uint64_t, 8 * D>{});
    if (S::kChunks > 16 && (chunk & 16)) jump(std::integral_constant<uint64_t, 16 * D>{});
    static_assert(S::kChunks == 16 || S::kChunks == 32, "jumps of the chunk number's bits");
    const bool energies = MODEL == TEAM_LD && a.sink.partials;
    const float2 cs = splat2(a.c.cs), cdt = splat2(a.c.cdt), cva = splat2(a.c.cva);
    float2 nck = {0.f, 0.f};
    if (energies) {
        float k[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) k[j] = -__fmul_rn(a.c.ckm, a.Kper ? a.Kper[live[j] ? idx[j] : first] : a.c.K);
        nck = make_float2(k[0], k[1]);
    }
    float* out = buf + chunk * S::kChunkWords + 2 * pair;
    // energy sums of this lane's chunk at step t, which has been consumed
    auto chunk_energy = [&](int64_t t) {
        const int nb = (int)max((int64_t)0, min((int64_t)S::kChunk, a.n_steps - t));
        float* state = out + S::kChunk * S::kStepWords;
        float2 X[3], V[3], bx = {0.f, 0.f}, bv = {0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            X[q] = *reinterpret_cast<const float2*>(state + q * G);
            V[q] = *reinterpret_cast<const float2*>(state + (3 + q) * G);
        }
        for (int k = 0; k < nb; ++k) {
#pragma unroll
            for (int q = 0; q < 3; ++q) team_update(cdt, cva, nck, *reinterpret_cast<const float2*>(out + k * S::kStepWords + q * G), X[q], V[q]);
            bx = __fadd2_rn(bx, EnergySum2::norm2x2(X));
            bv = __fadd2_rn(bv, EnergySum2::norm2x2(V));
        }
        *reinterpret_cast<float2*>(state) = bx;
        *reinterpret_cast<float2*>(state + G) = bv;
    };
    if ((int64_t)stage * S::kStageSteps >= a.n_steps) return;
    int64_t t0 = 0;
    for (; t0 + (int64_t)stage * S::kStageSteps < a.n_steps; t0 += S::kPassSteps) {
        if (t0 > 0) {
            bar_sync(1 + kStages + stage, bar_threads);   // the stage has been consumed
            if constexpr (MODEL == TEAM_LD)
                if (energies) chunk_energy(t0 - S::kPassSteps + (int64_t)chunk * S::kChunk);
        }
        const int64_t t = t0 + (int64_t)chunk * S::kChunk;
        const int nb = (int)max((int64_t)0, min((int64_t)S::kChunk, a.n_steps - t));
#pragma unroll 1
        for (int k = 0; k < nb; ++k) {
            float* o = out + k * S::kStepWords;
            if (MODEL == TEAM_LD) {
                float2 g[3];
                draw3x2<KIND>(td, lc, rd, g);
#pragma unroll
                for (int q = 0; q < 3; ++q) *reinterpret_cast<float2*>(o + q * G) = __fmul2_rn(cs, g[q]);
            } else {
                *reinterpret_cast<float2*>(o) = draw_cos2<KIND>(td, lc);
            }
        }
        if (nb > 0 && t + nb == a.n_steps) {   // the run's last draws: the end state
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (live[j]) {
                    if (KIND == GBRNG_TAUS)
                        a.taus[idx[j]] = td[j].y;
                    else
                        a.lcg[idx[j]] = lc[j].x;
                }
        }
        bar_arrive(1 + stage, bar_threads);
        // to the same chunk of the next pass
        if (t + S::kPassSteps < a.n_steps) jump(std::integral_constant<uint64_t, D*(S::kChunks - 1)>{});
        __syncwarp();
    }
    if constexpr (MODEL == TEAM_LD) {
        if (!energies) return;
        bar_sync(1 + kStages + stage, bar_threads);
        chunk_energy(t0 - S::kPassSteps + (int64_t)chunk * S::kChunk);
        bar_arrive(1 + stage, bar_threads);
    }
}

// Consumer warp's walk over the run: full(p) takes the kChunk steps of a whole
// chunk whose first normal of this lane is p[0] (a step's are kStepWords apart),
// one(p) a single step of the run's last, partial chunk; before either, start(c)
// sees the chunk's own area.  With ENERGIES the producers work on every consumed
// stage once more, and fold(c) takes each chunk's results, in time order, when
// the stage comes back.
template <class S, bool ENERGIES, class Start, class Full, class One, class Fold>
__device__ __forceinline__ void team_consume(const TeamArgs& a, float* buf, int off, int bar_threads,
                                             Start&& start, Full&& full, One&& one, Fold&& fold)
{
    constexpr int kPer = S::kChunks / kStages;   // chunks of a stage
    auto fold_stage = [&](int stage, int n_chunks) {
#pragma unroll 1
        for (int k = 0; k < n_chunks; ++k) fold(buf + (stage * kPer + k) * S::kChunkWords);
        __syncwarp();
    };
    int64_t t0 = 0;
    int stage = 0;
    while (t0 < a.n_steps) {
        bar_sync(1 + stage, bar_threads);
        if (ENERGIES && t0 >= S::kPassSteps) fold_stage(stage, kPer);
        const int n_stage = (int)min((int64_t)S::kStageSteps, a.n_steps - t0);
        float* c = buf + stage * kPer * S::kChunkWords;
#pragma unroll 1
        for (int s = S::kChunk; s <= n_stage; s += S::kChunk, c += S::kChunkWords) {
            start(c);
            full(c + off);
        }
        if (n_stage % S::kChunk) {
            start(c);
#pragma unroll 1
            for (int k = 0; k < n_stage % S::kChunk; ++k) one(c + off + k * S::kStepWords);
        }
        // hand the stage back if it is looked at or filled again
        if (ENERGIES || t0 + S::kPassSteps < a.n_steps) {
            bar_arrive(1 + kStages + stage, bar_threads);
        }
        t0 += n_stage;
        stage = (stage + 1) % kStages;
    }
    if (!ENERGIES) return;
    // the stages that have not come back: from the oldest, the last of them partial
    const int last = (int)(((a.n_steps - 1) / S::kStageSteps) % kStages);
    const int64_t uses = (a.n_steps + S::kStageSteps - 1) / S::kStageSteps;
    for (int k = (int)min(uses, (int64_t)kStages) - 1; k >= 0; --k) {
        const int st = (last - k + kStages) % kStages;
        const int n_last = k ? S::kStageSteps : (int)(a.n_steps - (uses - 1) * S::kStageSteps);
        bar_sync(1 + st, bar_threads);
        fold_stage(st, (n_last + S::kChunk - 1) / S::kChunk);
    }
}

// The loads of one lane's normals of a chunk.
template <class S, class T>
__device__ __forceinline__ void load_chunk(const float* p, T (&g)[S::kChunk])
{
#pragma unroll
    for (int k = 0; k < S::kChunk; ++k) g[k] = *reinterpret_cast<const T*>(p + k * S::kStepWords);
}

// Consumer of the oscillators; a lane holds component q of W oscillators.
template <class S, bool ENERGIES>
__device__ __forceinline__ void team_consume_ld(const TeamArgs& a, float* buf, int bar_threads)
{
    constexpr int G = S::kOsc, W = G == 8 ? 1 : 2, LPC = G / W;   // lanes a component
    static_assert(3 * LPC <= 32 && 2 * G <= 32, "one consumer warp");
    using T = typename std::conditional<W == 2, float2, float>::type;
    const int lane = threadIdx.x & 31;
    const int64_t first = blockIdx.x * (int64_t)G;
    const LdCoef c = a.c;
    const bool on = lane < 3 * LPC;
    const int q = on ? lane / LPC : 0, o = W * (on ? lane % LPC : 0);
    auto pack = [](const float (&f)[W]) {
        T r;
        if constexpr (W == 2)
            r = make_float2(f[0], f[1]);
        else
            r = f[0];
        return r;
    };
    auto part = [](T f, int j) {
        if constexpr (W == 2)
            return j ? f.y : f.x;
        else
            return f;
    };
    float xs[W], vs[W], ks[W], c0[W], c1[W];
#pragma unroll
    for (int j = 0; j < W; ++j) {
        const int64_t i = first + o + j < a.n ? first + o + j : first;
        ks[j] = -__fmul_rn(c.ckm, a.Kper ? a.Kper[i] : c.K);
        xs[j] = a.x[3 * i + q], vs[j] = a.v[3 * i + q];
        c0[j] = c.cdt, c1[j] = c.cva;
    }
    T X = pack(xs), V = pack(vs);
    const T nck = pack(ks), cdt = pack(c0), cva = pack(c1);
    Kahan K;   // lanes 0 .. G - 1: sum |x|^2 of oscillator lane; G .. 2G - 1: sum |v|^2
    team_consume<S, ENERGIES>(
        a, buf, q * G + o, bar_threads,
        [&](float* ch) {
            if (!ENERGIES || !on) return;
            float* state = ch + S::kChunk * S::kStepWords + q * G + o;
            *reinterpret_cast<T*>(state) = X;
            *reinterpret_cast<T*>(state + 3 * G) = V;
        },
        [&](const float* p) {
            T g[S::kChunk];
            load_chunk<S>(p, g);
#pragma unroll
            for (int k = 0; k < S::kChunk; ++k) team_update(cdt, cva, nck, g[k], X, V);
        },
        [&](const float* p) { team_update(cdt, cva, nck, *reinterpret_cast<const T*>(p), X, V); },
        [&](const float* ch) {
            if (lane < 2 * G) K.add(ch[S::kChunk * S::kStepWords + lane]);
        });
    double acc[4] = {0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < W; ++j) {
        const int64_t i = first + o + j;
        if (!on || i >= a.n) continue;
        const float x = part(X, j), v = part(V, j);
        a.x[3 * i + q] = x;
        a.v[3 * i + q] = v;
        acc[0] += (double)x * x;
        acc[1] += (double)v * v;
        acc[2] += (double)x * v;
    }
    if (!ENERGIES) return;
    const int64_t ie = first + lane % G;
    if (lane < 2 * G && ie < a.n)
        acc[3] = (double)(lane < G ? 0.5f * (a.Kper ? a.Kper[ie] : c.K) : c.hm) * K.value();
    store_stats(a.sink, warp_sums(acc));
}

// Consumer of the overdamped particles, a lane each; records between steps.
template <class S>
__device__ __forceinline__ void team_consume_ou(const TeamArgs& a, float* buf, int bar_threads)
{
    constexpr int G = S::kOsc;
    static_assert(2 * G <= 32, "two lanes a particle");
    const int lane = threadIdx.x & 31;
    // lanes beyond the first G repeat them: a record's sum of R is theirs, R R(0) the next G's
    const int64_t i = blockIdx.x * (int64_t)G + lane % G;
    const bool live = i < a.n;
    float R = live ? a.x[i] : 0.f;
    const float R0 = R, c1 = a.oc.c1, cs = a.oc.cs;
    int64_t t = 0, rec = 0, next_rec = 0;
    // record of the positions Rt after t steps
    auto record = [&](float Rt) {
        double v = !live ? 0.0 : lane & G ? (double)Rt * (double)R0 : (double)Rt;
#pragma unroll
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 || lane == G) a.records[2 * (rec * gridDim.x + blockIdx.x) + lane / G] = v;
        ++rec;
        next_rec += a.every;
    };
    if (a.records) record(R);
    else next_rec = INT64_MAX;
    auto one = [&](const float* p) {
        R = __fmaf_rn(cs, *p, __fmaf_rn(-c1, R, R));
        if (++t == next_rec) record(R);
    };
    team_consume<S, false>(
        a, buf, lane % G, bar_threads, [](float*) {},
        [&](const float* p) {
            if (a.every < S::kChunk && next_rec != INT64_MAX) {   // several records a chunk
                // the positions take the normals' places, and the records theirs from there
                float* pos = const_cast<float*>(p);
                float g[S::kChunk];
                load_chunk<S>(p, g);
                __syncwarp();
#pragma unroll
                for (int k = 0; k < S::kChunk; ++k) {
                    R = __fmaf_rn(cs, g[k], __fmaf_rn(-c1, R, R));
                    pos[k * S::kStepWords] = R;
                }
                while (next_rec <= t + S::kChunk) record(pos[(next_rec - t - 1) * S::kStepWords]);
                t += S::kChunk;
                return;
            }
            // at most one record inside: keep the positions of its step
            const int at = next_rec - t <= S::kChunk ? (int)(next_rec - t) : -1;
            float g[S::kChunk], Rt = 0.f;
            load_chunk<S>(p, g);
#pragma unroll
            for (int k = 0; k < S::kChunk; ++k) {
                R = __fmaf_rn(cs, g[k], __fmaf_rn(-c1, R, R));
                Rt = k + 1 == at ? R : Rt;
            }
            t += S::kChunk;
            if (at > 0) record(Rt);
        },
        one, [](const float*) {});
    if (live && lane < G) a.x[i] = R;
}

template <int MODEL, int KIND, int PAIRS, int M>
__global__ void __launch_bounds__(TeamShape<MODEL, PAIRS, M>::kThreads) team_kernel(TeamArgs a)
{
    using S = TeamShape<MODEL, PAIRS, M>;
    constexpr int kBarThreads = 32 * (M + 1);
    extern __shared__ __align__(16) float team_sm[];
    if (threadIdx.x < S::kProducers)
        team_produce<MODEL, KIND, S>(a, team_sm, kBarThreads);
    else if constexpr (MODEL == TEAM_OU)
        team_consume_ou<S>(a, team_sm, kBarThreads);
    else if (a.sink.partials)
        team_consume_ld<S, true>(a, team_sm, kBarThreads);
    else
        team_consume_ld<S, false>(a, team_sm, kBarThreads);
}

template <int MODEL, int KIND, int PAIRS, int M>
static int launch_team(TeamArgs& a, cudaStream_t st)
{
    using S = TeamShape<MODEL, PAIRS, M>;
    const int64_t blocks = (a.n + S::kOsc - 1) / S::kOsc;
    const size_t smem = S::kBufBytes;
    auto fn = team_kernel<MODEL, KIND, PAIRS, M>;
    GB_CUDA(cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    fn<<<(unsigned)blocks, S::kThreads, smem, st>>>(a);
    GB_CUDA(cudaGetLastError());
    return GBRNG_OK;
}

// Eight oscillators a block where that leaves at most four blocks a SM, or up to
// twelve when the run is long enough for their start-up (the jumps) not to count.
static bool team_of_8(int64_t n, int64_t n_steps, int sms)
{
    return n <= (int64_t)32 * sms || (n <= (int64_t)96 * sms && n_steps >= 512);
}

int ld_team(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st)
{
    Handle* h = s->rng;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const bool small = team_of_8(s->n, n_steps, di.sms);
    const int64_t blocks = (s->n + (small ? 7 : 15)) / (small ? 8 : 16);
    TeamArgs a{};
    a.n = s->n;
    a.n_steps = n_steps;
    a.x = s->x;
    a.v = s->v;
    a.Kper = s->K_per;
    a.c = make_coef(s);
    a.taus = h->taus;
    a.lcg = h->lcg;
    GB_CHECK(make_sink(h, blocks, out != nullptr, &a.sink));
    if (h->kind == GBRNG_TAUS)
        GB_CHECK((small ? launch_team<TEAM_LD, GBRNG_TAUS, 4, 1>(a, st) : launch_team<TEAM_LD, GBRNG_TAUS, 8, 1>(a, st)));
    else
        GB_CHECK((small ? launch_team<TEAM_LD, GBRNG_LCG, 4, 1>(a, st) : launch_team<TEAM_LD, GBRNG_LCG, 8, 1>(a, st)));
    return finish_stats(h, a.sink, blocks, n_steps, out, st);
}

// Overdamped runs of few particles, of enough steps for the blocks' start-up, some
// 0.6 us per 1000 particles (Hybrid Taus, one a thread / team, us: 5000 particles x 100
// steps 36 / 31; 1e4 x 200 41 / 43, x 400 50 / 48, x 1000 81 / 64; 2e4 x 400 63 / 63,
// x 1000 108 / 92; 4e4 x 1000 140 / 146, x 4000 474 / 441; 6e4 x 4000 591 / 628).
// Returns 1 and the number of blocks when it has launched, else 0 or an error.
int ou_team(const ou_system* s, int64_t n_steps, int64_t every, bool rec, int64_t* blocks_out, cudaStream_t st)
{
    Handle* h = s->rng;
    if (h->kind != GBRNG_TAUS && h->kind != GBRNG_LCG) return 0;
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    const int64_t per_sm = s->n / di.sms;
    if (per_sm >= 256 || n_steps < 48 || (per_sm >= 48 && n_steps < s->n / (per_sm < 128 ? 32 : 16))) return 0;
    const bool small = s->n <= (int64_t)16 * di.sms;
    const int64_t blocks = small ? (s->n + 7) / 8 : (s->n + 15) / 16, n_rec = n_steps / every + 1;
    if (rec) {
        if (!records_fit(n_rec, blocks, s->n)) return 0;
        GB_CHECK(ensure_partials(h, (2 * n_rec * blocks + 2 * n_rec + 3) / 4));
    }
    TeamArgs a{};
    a.n = s->n;
    a.n_steps = n_steps;
    a.x = s->R;
    a.oc = make_ou_coef(s);
    a.every = every;
    a.taus = h->taus;
    a.lcg = h->lcg;
    a.records = rec ? h->partials : nullptr;
    *blocks_out = blocks;
    if (h->kind == GBRNG_TAUS)
        GB_CHECK((small ? launch_team<TEAM_OU, GBRNG_TAUS, 4, 1>(a, st) : launch_team<TEAM_OU, GBRNG_TAUS, 8, 1>(a, st)));
    else
        GB_CHECK((small ? launch_team<TEAM_OU, GBRNG_LCG, 4, 1>(a, st) : launch_team<TEAM_OU, GBRNG_LCG, 8, 1>(a, st)));
    return 1;
}

}  // namespace gb
