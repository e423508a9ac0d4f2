// kernels.h -- host-side launchers of the NI-ORCA stages (internal).
#pragma once
#include <cuda_runtime.h>

#include "adj.cuh"

namespace niorca {

// Per-call work memory, carved from one pool allocation.
struct Work {
    int n = 0, m = 0;
    int graphs = 1;          // graphs of a batch (n and m are their sums)
    int ntiles = 0;          // relabel tiles of RL_TILE vertices
    int2 *vinfo = nullptr;   // old id -> (new id, degree)
    int *perm = nullptr;     // new id -> old id
    int *chist = nullptr;    // class histogram, NCLASS x ntiles (class-major)
    int *coff = nullptr;     // exclusive scan of chist
    int *nrow = nullptr;     // relabelled offsets, n + 1
    int *split = nullptr;    // scan input: degree of each new id
    int4 *rinfo = nullptr;   // {row start, split, row end, 0} per new id
    int *ncol = nullptr;     // relabelled neighbours, m
    int *tcnt = nullptr;     // triangle count of each out-entry (u, v), u < v; m ints in a region of 8 m bytes
    VAcc *vacc = nullptr;    // per-vertex accumulators, n
    int *scan_part = nullptr;// scan block partials
    int *lists = nullptr;    // heavy-vertex lists, 6 x n
    int *counters = nullptr; // list lengths and flags, 16 ints
    int *status = nullptr;   // device status word (not part of the carve)
    int num_sms = 0;
    int tune[11] = {16, 8, 8, 8, 8, 32, 1536, 64, 1152, 8192, 12288};  // see TuneIndex
    int induced = 0;         // write induced instead of non-induced counts
};

// Runtime tuning knobs (niorca_set_tuning): CTAs per SM of the persistent
// warp-tier kernels, and the thresholds that route vertices to a warp or a CTA.
enum TuneIndex {
    TUNE_GRID_RELABEL = 0,   // k_relabel_rows CTAs per SM
    TUNE_GRID_TRI = 1,       // k_tri_warp
    TUNE_GRID_AGG = 2,       // k_agg_warp
    TUNE_GRID_C4 = 3,        // k_c4_filter, k_c4_warp
    TUNE_GRID_SOLVE = 4,     // k_solve
    TUNE_LONG_ROW_CLASS = 5, // degree class from which a row is relabelled by a whole CTA
    TUNE_C4_WARP_MAXW = 6,   // largest wedge count W of a 4-cycle root kept in one warp (<= 1536)
    TUNE_WARP_MAXD = 7,      // largest out-degree of a triangle root kept in one warp (<= 64)
    TUNE_TRI_BITS_MAXD = 8,  // largest out-degree of a CTA-tier triangle root that keeps the bit matrix R (<= 1152)
    TUNE_TRI_HASH_MAXD = 9,  // largest out-degree of a CTA-tier triangle root that hashes N+(u) (<= 8192)
    TUNE_C4_TEAM_MINW = 10,  // 4-cycle roots with more wedges than this go to the key-tiled tier (<= 12288)
    TUNE_COUNT = 11
};

// Indices into Work::counters.
// The triangle and aggregate heavy lists hold two tiers each: CTA-sized
// roots from the front (CNT_*_HEAVY), the largest from the back (CNT_*_BIG).
// The *_NEXT entries are the work counters of the CTA tiers: each CTA takes
// its next root from the queue's counter, so a CTA that starts late (or a
// root that takes long) leaves no other CTA idle.
enum { CNT_TRI_HEAVY = 0, CNT_AGG_HEAVY = 1, CNT_C4_CTA = 2, CNT_C4_TEAM = 3, CNT_DMAX = 4, CNT_C4_MID = 5,
       CNT_C4_MIDP = 6, CNT_TRI_BIG = 7, CNT_AGG_BIG = 8, CNT_C4_LEFT = 9, CNT_C4_TILED_NEXT = 10,
       CNT_TRI_CTA_NEXT = 11, CNT_TRI_BIG_NEXT = 12, CNT_AGG_CTA_NEXT = 13, CNT_AGG_BIG_NEXT = 14,
       CNT_C4_MID_NEXT = 15, CNT_C4_MIDP_NEXT = 16, CNT_C4_CTA_NEXT = 17,
       CNT_BAD_ROWS = 18,   // a row is not strictly increasing, or out of range (recorded in the status too)
       CNT_ADJ_ON = 19,     // the triangle and aggregate stages probe the adjacency bitmap (AdjBits)
       CNT_SCAN_DONE = 20,  // blocks of a scan's first pass that are done (0 between scans)
       CNT_C4_MIDP_LEFT = 21,   // roots that k_c4_warp_left appends to k_c4_mid's packed queue
       CNT_C4_MODE = 22,    // of the first 4-cycle kernels, set by k_c4_wedge_len (0: the call is stopped)
       CNT_SAMPLE_DONE = 23,   // warps of k_c4_wedge_len that are done with the sample below
       CNT_CLUSTER = 24,    // two 64-bit sums over a sample of the vertices: 2 x triangles, ordered pairs of neighbours
       CNT_BAD_OFFSETS = 28,   // the CSR offsets fall, leave [0, m] or do not span it (recorded in the status too)
       NCOUNTERS = 32 };

// The next item of a work queue, for the whole CTA: thread 0 takes it from
// the queue's counter, every thread returns the same index.
__device__ __forceinline__ int cta_next(int *ctr) {
    __shared__ int s_item;
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(ctr, 1);
    __syncthreads();
    return s_item;
}

// Programmatic dependent launch: every kernel of the library is launched
// with launch_pdl, so that the next kernel on the stream is set up while
// the CTAs of the one before it drain (which hides most of the launch gap
// between the short kernels of a small graph), and begins with pdl_begin:
// it waits until the kernel before it has completed and its writes are
// visible, before touching memory. No kernel triggers its dependents early:
// CTAs of the next kernel waiting on SMs from the start of a kernel made
// the ER n = 1e6 call 35% slower.
__device__ __forceinline__ void pdl_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
void launch_pdl(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// CTAs of `kernel` (launched with `threads` threads and `smem` bytes of
// dynamic shared memory) that one SM holds at once: the size of a
// persistent grid is SMs times this.
int resident_ctas(const void *kernel, int threads, size_t smem);

// Whether the degree pass stopped the call; its error is recorded already, and
// every kernel after the relabelling returns at once. A degree above MAX_DEGREE
// (NIORCA_EOVERFLOW): the fixed-size shared buffers and 32-bit partial sums of
// those kernels rely on the bound (Sec. 3 bounds the work by the largest
// degree; the bound itself is this library's choice, see MAX_DEGREE). CSR
// offsets that fall or leave [0, m] (NIORCA_EINVAL): the rows that remain may
// overlap, so that their degrees sum to more than m and a copy of them has no
// place in the work memory; the row relabelling returns too. Bad offsets raise
// CNT_DMAX as well, so that a kernel waits for one load here (a second flag
// after it: about 1 us a kernel).
__device__ __forceinline__ void stop_bad_offsets(int *counters) {
    atomicOr(&counters[CNT_BAD_OFFSETS], 1);
    atomicMax(&counters[CNT_DMAX], 0x7fffffff);
}
__device__ __forceinline__ bool call_stopped(const int *counters) {
    return *reinterpret_cast<const volatile int *>(counters + CNT_DMAX) > MAX_DEGREE;
}

constexpr int RL_TILE = 2048;        // vertices per class-histogram tile
constexpr int SCAN_TILE = 4096;      // elements per scan block
constexpr int LONG_ROW_CLASS = 32;   // deg_class(512): rows from here on get a CTA each

size_t scan_partials(long long len);
// `done`: a counter that is 0 (and is again afterwards)
void launch_exclusive_scan(const int *in, int *out, long long len, bool write_total, int *part, int *done,
                           cudaStream_t st);

void launch_relabel(const int *rowptr, const int *colidx, Work &w, cudaStream_t st);
// The adjacency bitmap of a call (see AdjBits), over the second half of the
// triangle-count region, which is unused until the 4-cycle stage.
AdjBits adj_bits(const Work &w);
// Small graphs have none: their triangle stage takes a few microseconds either
// way, as much as the launch that builds it (G(3213, mean degree 31): 110 us a
// call without, 120 with), except dense ones (G(387, 0.53): 561 us without,
// 410 with).
inline bool adj_wanted(int n, int m) { return m >= 1 << 17 || (m >= 1 << 14 && m >= 64ll * n); }
// Whether a graph of m entries may have an out-degree above d: u's d+
// out-neighbours have u's degree class at least, so degrees of 4/5 of u's and
// more, and all degrees sum to m: 0.8 (d+)^2 <= m.
inline bool out_degree_above(int d, int m) { return (long long)d * d * 4 < 5ll * m; }
void launch_stage1(Work &w, cudaStream_t st);
void launch_stage2(Work &w, cudaStream_t st);
void launch_cycle4(Work &w, cudaStream_t st);
void launch_solve(Work &w, long long *out, cudaStream_t st);
void launch_validate(const int *rowptr, const int *colidx, int n, int m, int *status, int num_sms,
                     cudaStream_t st);

// Kernel ids for the optional per-kernel event timing and launch counting.
enum KernelId {
    K_CLASS_HIST, K_SCAN, K_CLASS_SCATTER, K_RELABEL, K_BATCH_SETUP,
    K_TRI_WARP, K_TRI_CTA, K_AGG_WARP, K_AGG_CTA, K_C4_WARP, K_C4_CTA, K_C4_PLAN, K_C4_TILED,
    K_SOLVE, K_VALIDATE, K_C4_MID, K_TRI_BIG, K_AGG_BIG, K_C4_WARP_LEFT, K_C4_WEDGE_LEN, K_ADJ_BITS, K_C4_FILTER,
    K_COUNT
};
const char *kernel_name(int id);

// Called after every kernel launch: counts it and, when timing is on,
// records an event on the launching stream.
void after_launch(cudaStream_t st, int id);

}  // namespace niorca
