// Stand-alone fills for the per-thread generators (Hybrid Taus, the LCG, Ran2):
// out[d*S + s] is the d-th draw of stream s.  One thread owns one stream at a
// time and keeps its state in registers (Taus, the LCG) or in a shared-memory
// column (Ran2's shuffle table) for all of its draws, or, where the streams are
// few, a segment of a stream's draws; stores are coalesced across the streams of
// a warp.
#include <algorithm>

#include "jump.cuh"
#include "internal.cuh"

namespace gb {

enum { FILL_U32 = 0, FILL_UNIFORM = 1, FILL_NORMAL = 2 };

// Item idx from its draws.
template <int MODE>
__device__ __forceinline__ void emit_item(uint32_t r, int64_t idx, void* out)
{
    if (MODE == FILL_U32)
        ((uint32_t*)out)[idx] = r;
    else
        ((float*)out)[idx] = u01_from_u32(r);
}

// n_items = numbers (u32, uniform) or pairs (normal); the items idx, idx + S, ... < end of one
// word chain.  The last few:
template <int MODE, class State>
__device__ __forceinline__ void emit_last(State& y, int64_t idx, int64_t S, int64_t end, void* out)
{
    for (; idx < end; idx += S) {
        if (MODE == FILL_NORMAL) {
            uint32_t r[2];
            float2 g;
            word_draws(y, r);
            box_muller_u32(r[0], r[1], g.x, g.y);
            ((float2*)out)[idx] = g;
        } else {
            uint32_t r[1];
            word_draws(y, r);
            emit_item<MODE>(r[0], idx, out);
        }
    }
}

template <int MODE, class State>
__device__ __forceinline__ void emit_chain(State& y, int64_t idx, int64_t S, int64_t end, void* out)
{
    // four draws in flight per iteration: independent stores, one state chain
    for (; idx + 3 * S < end; idx += 4 * S) {
        if (MODE == FILL_NORMAL) {
            // the four pairs two at a time in the paired instructions' lanes
            uint32_t r[4];
            float2* o = (float2*)out;
            float2 ga, gb;
            word_draws(y, r);
            box_muller_2pairs_u32(r[0], r[1], r[2], r[3], ga, gb);
            o[idx] = ga, o[idx + S] = gb;
            word_draws(y, r);
            box_muller_2pairs_u32(r[0], r[1], r[2], r[3], ga, gb);
            o[idx + 2 * S] = ga, o[idx + 3 * S] = gb;
        } else {
            uint32_t r[4];
            word_draws(y, r);
#pragma unroll
            for (int q = 0; q < 4; ++q) emit_item<MODE>(r[q], idx + q * S, out);
        }
    }
    emit_last<MODE>(y, idx, S, end, out);
}

// The same, words or uniforms, by a group of neighbouring chains that stay together, a
// barrier of its `threads` threads (`id`) every four rows.  Where rows are not whole 32-byte
// sectors, each warp's store ends in two parts of sectors that its neighbours complete; on
// a fill larger than the L2 those that have drifted apart cost it (2^28 words of 208529
// Hybrid Taus streams 352 us, together 214; uniforms of 500001 LCG streams 308, 205; of 1e6
// streams, whole sectors, 170 and 157).  last, last_end: idx and end of the group's last
// chain, which has the fewest items; live: this thread has a chain.
template <int MODE, class State>
__device__ __forceinline__ void emit_together(State& y, bool live, int64_t idx, int64_t S, int64_t end, int64_t last,
                                              int64_t last_end, int id, int threads, void* out)
{
    for (; last + 3 * S < last_end; idx += 4 * S, last += 4 * S) {
        bar_sync(id, threads);
        uint32_t r[4];
        word_draws(y, r);
        if (live)
#pragma unroll
            for (int q = 0; q < 4; ++q) emit_item<MODE>(r[q], idx + q * S, out);
    }
    if (live) emit_last<MODE>(y, idx, S, end, out);
}

// Hybrid Taus (uint4 state) and the LCG (uint32 state): one word chain per stream.
constexpr int kWordThreads = 256;
template <int MODE, bool TOGETHER, class State>
__global__ void __launch_bounds__(kWordThreads) word_fill_kernel(State* __restrict__ st, int64_t S,
                                                                 int64_t n_items, void* __restrict__ out)
{
    const int64_t active = S < n_items ? S : n_items;
    const int64_t s0 = blockIdx.x * (int64_t)kWordThreads;
    if constexpr (TOGETHER) {
        const int64_t s = s0 + threadIdx.x;
        const bool live = s < active;
        State y{};
        if (live) y = word_load(st[s]);
        emit_together<MODE>(y, live, s, S, n_items, min(s0 + kWordThreads, active) - 1, n_items, 0, kWordThreads, out);
        if (live) st[s] = y;
    } else {
        const int64_t stride = (int64_t)gridDim.x * kWordThreads;
        for (int64_t s = s0 + threadIdx.x; s < active; s += stride) {
            State y = word_load(st[s]);
            emit_chain<MODE>(y, s, S, n_items, out);
            st[s] = y;
        }
    }
}

// Few streams: one chain a stream leaves most of the GPU idle (a draw is about 25
// cycles of latency), so a stream's items are cut into segments of L, each thread's
// generator jumped ahead to its segment (jump.cuh: the same words as stepping
// there).  All segments of a group of B streams are in one cluster of blocks, so
// that the states are read, by the cluster's barrier, before any thread replaces
// one; clusters keep B, the streams that a row of stores covers, at least 32 (2^27
// uniforms of 4096 streams: 434 us with 16 in one block, 148 with 32, 181 with 64 and
// twice the blocks a cluster), or, with chains together, at the most that eight blocks
// give (2^28 words of 24001 Hybrid Taus streams: 466 us with B = 64 apart, 377 together, 238
// with B = 512; one chain a stream 310).  One thread a stream, then segments (in brackets with
// the words by funnel shifts), us: 2^20 words of 4096 streams 12.4, 6.3 (6.3); 2^24 uniforms of
// 1024 559, 22.7 (20.6); 2^27 of 4096 1118, 148 (113), of 2e4 233, 173 (131), of 5e4 176,
// 140 (107); 2^27 normals of 4096 1868, 208 (191).
constexpr int kSplitThreads = 512, kSplitMax = 64, kSplitRow = 32;
struct SplitArgs {
    Jump lo[8], hi[kSplitMax / 8];   // g L items ahead for g = 0 .. 7, and 8g L
    int64_t L;
    int B;                           // streams of a cluster; kSplitThreads / B segments a block
};

template <int MODE, bool TOGETHER, class State>
__global__ void __launch_bounds__(kSplitThreads) word_split_kernel(State* st, int64_t S, int64_t n_items,
                                                                   void* __restrict__ out,
                                                                   const __grid_constant__ SplitArgs a)
{
    uint32_t rank, blocks;   // of the cluster
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(blocks));
    const int64_t s = blockIdx.x / blocks * (int64_t)a.B + threadIdx.x % a.B;
    const int g = (int)rank * (kSplitThreads / a.B) + threadIdx.x / a.B;
    const int64_t first = s + g * a.L * S, end = min(n_items, first + a.L * S);
    const bool live = s < S && first < n_items;
    State y;
    if constexpr (TOGETHER) y = State{};
    if (live) {
        y = word_load(st[s]);
        if (g & 7) jump_ahead(y, a.lo[g & 7]);
        if (g >> 3) jump_ahead(y, a.hi[g >> 3]);
    }
    cluster_sync();
    if constexpr (TOGETHER) {
        const int64_t last = min(s - threadIdx.x % a.B + a.B, S) - 1 + g * a.L * S;
        emit_together<MODE>(y, live, first, S, end, last, min(n_items, last + a.L * S), threadIdx.x / a.B, a.B, out);
        if (!live) return;
    } else {
        if (!live) return;
        emit_chain<MODE>(y, first, S, end, out);
    }
    if (first + ((end - first - 1) / S) * S + S >= n_items) st[s] = y;   // the stream's last item
}

constexpr int kRan2Threads = 128;

// The table's 32 words are loaded, and stored, all at once: at 134 draws a stream of 1e6
// streams the state is a third of the traffic, and four words at a time its latency shows
// (2^27 uniforms 167 us, eight or sixteen at a time 160, all 150; 2^24 70 and 62).
// Eight blocks a SM, 64 registers: with the compiler's 128 half as many warps are there to
// hide a draw's chain (2^27 from 1e6 streams, 128 registers / six / eight / ten / twelve
// blocks: uniforms 150 / 142 / 140 / 142 / 160 us, normals 201 / 191 / 193 / 191 / 197; 2^24
// uniforms of 4096 streams 152 / 160 / 154 / 167 / 168).
template <int MODE>
__global__ void __launch_bounds__(kRan2Threads, 8) ran2_fill_kernel(int32_t* __restrict__ st, int64_t S,
                                                        int64_t n_items, void* __restrict__ out)
{
    extern __shared__ int32_t tab[];      // [32][blockDim.x]
    const int64_t active = S < n_items ? S : n_items;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < active; s += stride) {
        Ran2Draw rd;
        rd.load<32>(st + s, S, tab, kRan2Threads);
        auto emit = [&](int64_t idx) {
            if (MODE == FILL_U32) {
                ((uint32_t*)out)[idx] = (uint32_t)-rd.next();
            } else if (MODE == FILL_UNIFORM) {
                ((float*)out)[idx] = u01_from_ran2(rd.next());
            } else {
                const float u1 = u01_from_ran2(rd.next());
                const float u2 = u01_from_ran2(rd.next());
                float2 g;
                box_muller(u1, u2, g.x, g.y);
                ((float2*)out)[idx] = g;
            }
        };
        int64_t idx = s;
        // four draws a loop iteration: one bound check for four stores
        for (; idx + 3 * S < n_items; idx += 4 * S) {
            if (MODE == FILL_NORMAL) {
                // the four pairs two at a time in the paired instructions' lanes
                int32_t n[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) n[q] = rd.next();
                float2* o = (float2*)out;
                float2 ga, gb;
                box_muller_2pairs_ran2(n[0], n[1], n[2], n[3], ga, gb);
                o[idx] = ga, o[idx + S] = gb;
                box_muller_2pairs_ran2(n[4], n[5], n[6], n[7], ga, gb);
                o[idx + 2 * S] = ga, o[idx + 3 * S] = gb;
            } else {
                emit(idx);
                emit(idx + S);
                emit(idx + 2 * S);
                emit(idx + 3 * S);
            }
        }
        for (; idx < n_items; idx += S) emit(idx);
        rd.store<32>(st + s, S);
    }
}

// When to cut streams into segments, from the items of the longest chain: a thread a stream
// takes `one` us an item where no SM has more than one block of 256 threads and `two` where
// one has two (up to 400 streams a SM; beyond, segments never pay), `ragged` times that where
// rows are not whole sectors, a segment's item `seg` for every block of 512 on the busiest
// SM, and the jump as much as `jump` items, besides 5 (normals 7) and 6.6 us of either launch.  Fitted to 31 stream counts from 1024 to 1e6, 2^16 to 2^28 items
// each; where the rule and the faster side differ, they are within 2 us or 5% of each other.
//
// Together: words whose rows are not whole sectors, in a fill of more than the L2 keeps (2^25
// words, 134 MB, still 3 to 40% faster apart, 2^26 5 to 45% faster together) and, in segments,
// of streams enough for rows of some hundred (2^26 words of 1025 streams 113 us apart, 120
// together; of 2501 144, 103).  Normal pairs take longer to form than such stores.
// (The LCG's, which draw faster, from 2^25 words on: 33691 streams 41 us apart, 30 together.)
template <class State>
constexpr int64_t kTogetherBytes = (int64_t)(sizeof(State) == 4 ? 120 : 192) << 20;
constexpr int64_t kTogetherStreams = 2048;
struct FillCost {
    double one, two, ragged, seg, jump;
};
constexpr FillCost kFillCost[2][2] = {   // [Hybrid Taus, the LCG][words, normal pairs]
    {{0.029, 0.0535, 1, 0.044, 20}, {0.0915, 0.172, 1, 0.165, 15}},
    {{0.020, 0.041, 1.2, 0.0425, 5}, {0.071, 0.128, 1, 0.117, 7}}};

static bool split_pays(const FillCost& c, bool normal, bool ragged, int64_t S, int64_t items, int Q, int64_t blocks,
                       int sms)
{
    const double each = ((S + 255) / 256 > sms ? c.two : c.one) * (ragged ? c.ragged : 1.0);
    const double w = (double)((blocks + sms - 1) / sms), whole = (normal ? 7.0 : 5.0) + (double)items * each;
    return 6.6 + ((double)items / Q + c.jump) * c.seg * w < whole;
}

// Segments: powers of two that bring the threads to about 1024 a SM, of at least 32 items.
// Returns 1 when it has launched, 0 for one thread a stream, or an error.
template <int MODE, class State>
static int fill_split(Handle* h, State* states, void* dst, int64_t n_items, bool ragged, bool together,
                      cudaStream_t st)
{
    const int64_t S = h->n, items = (n_items + S - 1) / S;   // of the longest chain
    DevInfo di;
    GB_CHECK(dev_info(h->device, &di));
    int Q = 1;
    while (S <= (int64_t)di.sms * 400 && Q < kSplitMax && S * Q < (int64_t)di.sms * 1024 && items / (2 * Q) >= 32) Q *= 2;
    if (Q < 2) return 0;
    const int few = std::max(1, Q * kSplitRow / kSplitThreads);
    const int64_t rows = kSplitThreads * few / Q;
    if (!split_pays(kFillCost[h->kind == GBRNG_LCG][MODE == FILL_NORMAL], MODE == FILL_NORMAL, ragged && !together, S,
                    items, Q, (S + rows - 1) / rows * few, di.sms))
        return 0;
    if (S < kTogetherStreams) together = false;
    const int C = together ? std::min(8, Q) : few;   // blocks of a cluster
    SplitArgs a;
    a.B = kSplitThreads * C / Q;
    a.L = (items + Q - 1) / Q;
    const Jump one = jump_of((uint64_t)a.L * (MODE == FILL_NORMAL ? 2 : 1));
    a.lo[0] = a.hi[0] = jump_of(0);
    for (int g = 1; g < 8 && g < Q; ++g) a.lo[g] = jump_sum(a.lo[g - 1], one);
    if (Q > 8) {
        const Jump eight = jump_sum(a.lo[7], one);
        for (int g = 1; g < Q / 8; ++g) a.hi[g] = jump_sum(a.hi[g - 1], eight);
    }
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((S + a.B - 1) / a.B * C));
    cfg.blockDim = dim3(kSplitThreads);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    GB_CUDA(cudaLaunchKernelEx(&cfg, together ? word_split_kernel<MODE, MODE != FILL_NORMAL, State>
                                        : word_split_kernel<MODE, false, State>,
                               states, S, n_items, dst, a));
    return 1;
}

template <int MODE, class State>
static int fill_words(Handle* h, State* states, void* dst, int64_t n_items, cudaStream_t st)
{
    const int64_t S = h->n, active = std::min(S, n_items);
    const bool ragged = MODE != FILL_NORMAL && (S % 8 || (uintptr_t)dst % 32);
    const bool together = ragged && 4 * n_items >= kTogetherBytes<State>;
    if (const int rc = fill_split<MODE>(h, states, dst, n_items, ragged, together, st)) return rc < 0 ? rc : GBRNG_OK;
    const unsigned blocks = (unsigned)((active + kWordThreads - 1) / kWordThreads);
    if (together)
        word_fill_kernel<MODE, MODE != FILL_NORMAL, State><<<blocks, kWordThreads, 0, st>>>(states, S, n_items, dst);
    else
        word_fill_kernel<MODE, false, State><<<blocks, kWordThreads, 0, st>>>(states, S, n_items, dst);
    GB_CUDA(cudaGetLastError());
    return GBRNG_OK;
}

// Grid: one thread per stream (up to the streams a fill touches), in as many
// waves as that takes, rather than one resident wave looping over streams:
// the blocks then start, and load their streams' state, at staggered times
// instead of all together under the fill's store traffic (2^30 numbers from
// 1e6 streams: Ran2 uniform 1.15 -> 1.09 ms, normal 1.91 -> 1.82, Taus uniform
// 0.91 -> 0.87, normal 1.59 -> 1.57).  The kernels keep their stream loop, so
// any grid covers every stream.
template <int MODE>
static int fill_pt(Handle* h, void* dst, int64_t n_items, cudaStream_t st)
{
    const int64_t active = h->n < n_items ? h->n : n_items;
    if (h->kind == GBRNG_TAUS) return fill_words<MODE>(h, h->taus, dst, n_items, st);
    if (h->kind == GBRNG_LCG) return fill_words<MODE>(h, h->lcg, dst, n_items, st);
    const int T = kRan2Threads;
    const size_t smem = sizeof(int32_t) * 32 * T;
    const int64_t blocks = (active + T - 1) / T;
    ran2_fill_kernel<MODE><<<(unsigned)blocks, T, smem, st>>>(h->r2, h->n, n_items, dst);
    GB_CUDA(cudaGetLastError());
    return GBRNG_OK;
}

int fill_u32_pt(Handle* h, uint32_t* dst, int64_t n, cudaStream_t st)
{
    return fill_pt<FILL_U32>(h, dst, n, st);
}

int fill_uniform_pt(Handle* h, float* dst, int64_t n, cudaStream_t st)
{
    return fill_pt<FILL_UNIFORM>(h, dst, n, st);
}

int fill_normal_pt(Handle* h, float* dst, int64_t n, cudaStream_t st)
{
    return fill_pt<FILL_NORMAL>(h, dst, n / 2, st);
}

}  // namespace gb
