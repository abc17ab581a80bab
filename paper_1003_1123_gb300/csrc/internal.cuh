// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>

#include <nvtx3/nvToolsExt.h>

#include "gbrng.h"

namespace gb {

// ---------------------------------------------------------------- errors
int fail(int code, const char* fmt, ...);
void clear_error();

#define GB_CUDA(call)                                                                   \
    do {                                                                                \
        cudaError_t e_ = (call);                                                        \
        if (e_ != cudaSuccess)                                                          \
            return ::gb::fail(GBRNG_ECUDA, "%s failed: %s (%s:%d)", #call,              \
                              cudaGetErrorString(e_), __FILE__, __LINE__);              \
    } while (0)

#define GB_CHECK(expr)                                                                  \
    do {                                                                                \
        int rc_ = (expr);                                                               \
        if (rc_ != GBRNG_OK) return rc_;                                                \
    } while (0)

// Status values of a Lagged Fibonacci launch.
enum : int { DEV_OK = 0, DEV_TIMEOUT = 1 };

// NVTX range named after the C ABI call, open for the call's duration (a
// no-op unless a profiler or tracer is attached).
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};

// ---------------------------------------------------------------- handle
struct Handle {
    int kind = 0;
    uint64_t seed = 0;
    int64_t n = 0;       // streams (per-thread kinds) or threads per step (LFG)
    int device = 0;

    uint4* taus = nullptr;     // [n] (y1, y2, y3, y4)
    int32_t* r2 = nullptr;     // [35][n]: idum, idum2, iy, iv[0..31]
    uint32_t* lcg = nullptr;   // [n] Quick and Dirty LCG words

    // Lagged Fibonacci: the sequence value at position p lives in
    // ring[p mod ring_size], those of the last lfg_history() positions before pos
    // always.  depth: the deepest fan the ring serves; order_max (2 or 4): the
    // highest order a paper-form or overdamped step may need (lfg.cuh).
    int row = -1;
    int32_t sl = 0, ll = 0;
    int order_max = 2, depth = 0;
    uint32_t ring_size = 0;
    uint32_t* ring = nullptr;
    int64_t pos = 0;           // next position to generate

    // scratch owned by the handle
    uint64_t* progress = nullptr;   // grid-barrier arrival counter, status (LFG)
    int64_t progress_cap = 0;
    unsigned* ticket = nullptr;     // blocks that have left their statistics (0 between launches)
    double* partials = nullptr;     // per-block reduction partials
    int64_t partials_cap = 0;
    float2* eacc = nullptr;         // paper-form runs: per-oscillator energy sum (Kahan s, c)
    int64_t eacc_cap = 0;
    float* adj = nullptr;           // adjoint checkpoints and noise (history or one segment)
    size_t adj_bytes = 0;
};

// Positions before the next one that a handle's ring holds: D + depth sl.
inline int64_t lfg_history(const Handle* h) { return (int64_t)h->ll - h->sl + (int64_t)h->depth * h->sl; }

// Device attributes used for launch sizing (cached per device).
struct DevInfo {
    int sms = 0;
    int max_threads_sm = 0;
    size_t smem_optin = 0;
};
int dev_info(int device, DevInfo* out);

// cudaMalloc, a second time without the kept rings (runtime.cu) where memory has run out.
cudaError_t device_alloc(void** p, size_t bytes);
int ensure_partials(Handle* h, int64_t count);
int ensure_progress(Handle* h, int64_t count);

uint64_t wait_limit_ns();
int64_t test_stall_chunk();

// Kernel-side parameters of one Langevin system (binary32 coefficients,
// computed once on the host from the double parameters).
struct LdCoef {
    float cdt, cva, ckm, cs, sv, kT, K, hm;
};
LdCoef make_coef(const ld_system* s);
int check_system(const ld_system* s, bool need_rng);

// Per-thread generator entry points (fill.cu, ld.cu)
int fill_u32_pt(Handle* h, uint32_t* dst, int64_t n, cudaStream_t st);
int fill_uniform_pt(Handle* h, float* dst, int64_t n, cudaStream_t st);
int fill_normal_pt(Handle* h, float* dst, int64_t n, cudaStream_t st);
int ld_init_pt(const ld_system* s, cudaStream_t st);
int ld_run_pt(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st);
// Small systems, Hybrid Taus and the LCG, n_steps >= 1 (team.cu).
int ld_team(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st);

// Lagged Fibonacci entry points (lfg.cu)
int lfg_seed(Handle* h, cudaStream_t st);
void lfg_new_handle(Handle* h);   // order_max, depth and ring_size of a new handle
int lfg_fill(Handle* h, void* dst, int64_t n, int mode, cudaStream_t st);  // mode 0 u32, 1 uniform, 2 normal
int lfg_ld(const ld_system* s, int64_t n_steps, int init, ld_stats* out, cudaStream_t st);

// Paper-form runs, one launch per step (stepwise.cu, lfg.cu).
int ld_run_stepwise_pt(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st);
int lfg_ld_stepwise(const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st);
int ensure_eacc(Handle* h, int64_t n);
int ensure_adj(Handle* h, size_t bytes);
// Final-state sums and the per-oscillator energy sums of a paper-form run.
int stepwise_stats(Handle* h, const ld_system* s, int64_t n_steps, ld_stats* out, cudaStream_t st);

// Overdamped 1-D runs (ou.cu, lfg.cu).  Records land in
// partials[(rec * blocks + block) * 2 + {0, 1}] (sums of R and R R0).
struct OuCoef {
    float c1, cs;
};
OuCoef make_ou_coef(const ou_system* s);
int ou_run_pt(const ou_system* s, int64_t n_steps, int64_t every, double* mean, double* corr,
              cudaStream_t st);
int lfg_ou(const ou_system* s, int64_t n_steps, int64_t every, double* mean, double* corr,
           cudaStream_t st);
int ou_finish(Handle* h, int64_t n, int64_t n_rec, int64_t blocks, double* mean, double* corr,
              cudaStream_t st);

int ou_team(const ou_system* s, int64_t n_steps, int64_t every, bool rec, int64_t* blocks_out, cudaStream_t st);

// Pinned mapped memory of this host thread for a call's results (at most
// kHostBlock bytes): a call that has kernels write there reads it, synchronised,
// before it returns.  Null if it cannot be allocated.
constexpr size_t kHostBlock = 65536;
void* host_block();
// Wait for st before the block is read (a failure leaves the thread without that block).
int sync_results(cudaStream_t st);

// Statistics.  make_sink: where a launch of `blocks` blocks leaves its sums
// (partials grown if needed).  finish_stats: add them up if the launch has not,
// synchronise st and fill out (no-op for out == null).
struct StatsSink;
int make_sink(Handle* h, int64_t blocks, bool want, StatsSink* out);
int finish_stats(Handle* h, const StatsSink& sink, int64_t blocks, int64_t n_steps, ld_stats* out,
                 cudaStream_t st);

// Lagged Fibonacci Table I (row 4 as sl = 13470).
int lfg_lags(int row, int32_t* sl, int32_t* ll);
int lfg_default_row(int64_t n_threads);

}  // namespace gb

struct gbrng_rng : gb::Handle {};
