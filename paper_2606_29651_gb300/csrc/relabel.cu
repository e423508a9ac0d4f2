// relabel.cu -- degree-ordered relabelling of the input CSR.
//
// Algorithm 2 orients every edge from the smaller to the larger vertex id
// (y.id > x.id) so that each triangle and each K4 is found once. Any total
// order keeps that property; this implementation uses (degree class, id),
// with four classes per octave of degree, so that the out-lists of the
// oriented graph stay short on skewed graphs (a hub only points at other
// hubs). Vertices are renumbered in that order; in the relabelled CSR every
// row is ascending, so N+(u) = {v in N(u): v > u} is the suffix of row u
// starting at split[u], and N-(u) is the prefix.
//
// Because new ids inside one class follow old ids, a row of the input that
// is sorted by old id becomes sorted by new id after a stable partition by
// class: no sort is needed, only per-class counting.
#include "kernels.h"

namespace niorca {

// ------------------------------------------------------------ exclusive scan

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_PER_THREAD = SCAN_TILE / SCAN_THREADS;

size_t scan_partials(long long len) { return (size_t)((len + SCAN_TILE - 1) / SCAN_TILE) + 1; }

__device__ __forceinline__ int block_exclusive_scan(int v, int *wsum, int *total) {
    const int lane = lane_id(), w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int incl = warp_inclusive_scan(v);
    if (lane == 31) wsum[w] = incl;
    __syncthreads();
    if (w == 0) {
        int x = lane < nw ? wsum[lane] : 0;
        int xi = warp_inclusive_scan(x);
        if (lane < nw) wsum[lane] = xi - x;
        if (lane == nw - 1) *total = xi;
    }
    __syncthreads();
    int r = incl - v + wsum[w];
    __syncthreads();
    return r;
}

// Sums of the tiles; the block that finishes last scans them (no block waits
// for another).
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(const int *in, long long len, int *part, int *done) {
    pdl_begin();
    __shared__ int wsum[32];
    __shared__ int tot;
    __shared__ bool last;
    const long long base = (long long)blockIdx.x * SCAN_TILE;
    int s = 0;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        long long g = base + i;
        if (g < len) s += in[g];
    }
    block_exclusive_scan(s, wsum, &tot);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = tot;
        __threadfence();
        last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int nblocks = gridDim.x;
    volatile int *vp = part;
    int carry = 0;
    for (int b0 = 0; b0 < nblocks; b0 += 4 * SCAN_THREADS) {
        const int i = b0 + 4 * threadIdx.x;
        int v[4], sum = 0;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            v[h] = i + h < nblocks ? vp[i + h] : 0;
            sum += v[h];
        }
        int ex = block_exclusive_scan(sum, wsum, &tot) + carry;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (i + h < nblocks) vp[i + h] = ex;
            ex += v[h];
        }
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        vp[nblocks] = carry;
        *done = 0;
    }
}

// With part == nullptr a single block scans the whole array (len <= SCAN_TILE).
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_down(const int *in, int *out, long long len, const int *part,
                                                           int write_total) {
    pdl_begin();
    __shared__ int tile[SCAN_TILE];
    __shared__ int wsum[32];
    __shared__ int tot;
    const long long base = (long long)blockIdx.x * SCAN_TILE;
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        long long g = base + i;
        tile[i] = g < len ? in[g] : 0;
    }
    __syncthreads();
    int local[SCAN_PER_THREAD];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        local[k] = tile[threadIdx.x * SCAN_PER_THREAD + k];
        s += local[k];
    }
    int ex = block_exclusive_scan(s, wsum, &tot) + (part ? part[blockIdx.x] : 0);
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        tile[threadIdx.x * SCAN_PER_THREAD + k] = ex;
        ex += local[k];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SCAN_TILE; i += SCAN_THREADS) {
        long long g = base + i;
        if (g < len) out[g] = tile[i];
    }
    if (write_total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[len] = part ? part[gridDim.x] : tot;
}

void launch_exclusive_scan(const int *in, int *out, long long len, bool write_total, int *part, int *done,
                           cudaStream_t st) {
    const int nb = (int)((len + SCAN_TILE - 1) / SCAN_TILE);
    if (nb == 0) {
        if (write_total) cudaMemsetAsync(out, 0, sizeof(int), st);
        return;
    }
    if (nb == 1) {   // one tile: one launch
        launch_pdl(k_scan_down, 1, SCAN_THREADS, 0, st, in, out, len, nullptr, write_total ? 1 : 0);
        after_launch(st, K_SCAN);
        return;
    }
    launch_pdl(k_scan_reduce, nb, SCAN_THREADS, 0, st, in, len, part, done);
    after_launch(st, K_SCAN);
    launch_pdl(k_scan_down, nb, SCAN_THREADS, 0, st, in, out, len, part, write_total ? 1 : 0);
    after_launch(st, K_SCAN);
}

// ------------------------------------------------------------- class order

constexpr int RL_THREADS = 256;

// Degrees (with offset validation) and the class histogram of each tile.
__global__ void __launch_bounds__(RL_THREADS) k_class_hist(const int *rowptr, int n, int m, int2 *vinfo, int *chist,
                                                           int ntiles, int *counters, int *status) {
    pdl_begin();
    __shared__ int h[NCLASS];
    __shared__ int smax;
    for (int c = threadIdx.x; c < NCLASS; c += RL_THREADS) h[c] = 0;
    if (threadIdx.x == 0) smax = 0;
    __syncthreads();
    int lmax = 0, bad = 0;
    const int tile = blockIdx.x;
    for (int i = threadIdx.x; i < RL_TILE; i += RL_THREADS) {
        const long long x = (long long)tile * RL_TILE + i;
        if (x >= n) break;
        const int a = rowptr[x], b = rowptr[x + 1];
        const bool ok = a >= 0 && b >= a && b <= m;
        const int d = ok ? b - a : 0;
        if (!ok || (x == 0 && a != 0) || (x == n - 1 && b != m)) bad = 1;
        vinfo[x] = make_int2(-1, d);
        atomicAdd(&h[deg_class(d)], 1);
        lmax = max(lmax, d);
    }
    if (bad) {
        set_status(status, ST_EINVAL);
        stop_bad_offsets(counters);
    }
    lmax = warp_max(lmax);
    if (lane_id() == 0) atomicMax(&smax, lmax);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&counters[CNT_DMAX], smax);
        if (smax > MAX_DEGREE) set_status(status, ST_EOVERFLOW);
    }
    for (int c = threadIdx.x; c < NCLASS; c += RL_THREADS) chist[c * ntiles + tile] = h[c];
}

// New id of every vertex: class offset + stable rank by old id within class.
__global__ void __launch_bounds__(RL_THREADS) k_class_scatter(int n, int2 *vinfo, const int *coff, int ntiles,
                                                              int *perm, int *ndeg) {
    pdl_begin();
    constexpr int NW = RL_THREADS / 32;
    __shared__ int run[NCLASS];
    __shared__ int tot[NCLASS];
    __shared__ int wc[NW][NCLASS];
    const int tile = blockIdx.x, lane = lane_id(), w = threadIdx.x >> 5;
    for (int c = threadIdx.x; c < NCLASS; c += RL_THREADS) run[c] = 0;
    for (int k = 0; k < RL_TILE / RL_THREADS; ++k) {
        for (int i = threadIdx.x; i < NW * NCLASS; i += RL_THREADS) (&wc[0][0])[i] = 0;
        __syncthreads();
        const long long x = (long long)tile * RL_TILE + k * RL_THREADS + threadIdx.x;
        const bool valid = x < n;
        const int d = valid ? vinfo[x].y : 0;
        const int c = valid ? deg_class(d) : NCLASS + lane;  // invalid lanes match only themselves
        const unsigned peers = __match_any_sync(FULL, c);
        const int rank = __popc(peers & lanemask_lt());
        if (valid && rank == 0) wc[w][c] = __popc(peers);
        __syncthreads();
        if (threadIdx.x < NCLASS) {
            int s = 0;
            for (int ww = 0; ww < NW; ++ww) {
                int t = wc[ww][threadIdx.x];
                wc[ww][threadIdx.x] = s;
                s += t;
            }
            tot[threadIdx.x] = s;
        }
        __syncthreads();
        if (valid) {
            const int id = coff[c * ntiles + tile] + run[c] + wc[w][c] + rank;
            vinfo[x].x = id;
            perm[id] = (int)x;
            ndeg[id] = d;
        }
        __syncthreads();
        if (threadIdx.x < NCLASS) run[threadIdx.x] += tot[threadIdx.x];
        __syncthreads();
    }
}

// The class order of a graph of at most RL_TILE vertices in one CTA, with no
// launch in between: the degree pass and class histogram of k_class_hist,
// the scan of the class offsets, the stable class scatter of k_class_scatter
// and the scan of the new degrees into the new row offsets (nrow[n] = m).
constexpr int RS_THREADS = 1024;
__global__ void __launch_bounds__(RS_THREADS) k_class_small(const int *rowptr, int n, int m, int2 *vinfo, int *coff,
                                                            int *perm, int *nrow, int *counters, int *status) {
    pdl_begin();
    constexpr int NW = RS_THREADS / 32;
    __shared__ int h[NCLASS];          // class counts, then each class's next id
    __shared__ int wc[NW][NCLASS];     // per-warp class counts, then offsets
    __shared__ int deg[RL_TILE];       // degree of each vertex
    __shared__ int nd[RL_TILE];        // degree of each new id
    __shared__ int wsum[32];
    __shared__ int tot, smax;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    for (int c = threadIdx.x; c < NCLASS; c += RS_THREADS) h[c] = 0;
    if (threadIdx.x == 0) smax = 0;
    __syncthreads();
    int lmax = 0, bad = 0;
    for (int x = threadIdx.x; x < n; x += RS_THREADS) {
        const int a = rowptr[x], b = rowptr[x + 1];
        const bool ok = a >= 0 && b >= a && b <= m;
        const int d = ok ? b - a : 0;
        if (!ok || (x == 0 && a != 0) || (x == n - 1 && b != m)) bad = 1;
        deg[x] = d;
        atomicAdd(&h[deg_class(d)], 1);
        lmax = max(lmax, d);
    }
    if (bad) {
        set_status(status, ST_EINVAL);
        stop_bad_offsets(counters);
    }
    lmax = warp_max(lmax);
    if (lane == 0) atomicMax(&smax, lmax);
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicMax(&counters[CNT_DMAX], smax);
        if (smax > MAX_DEGREE) set_status(status, ST_EOVERFLOW);
    }
    {   // class offsets (NCLASS <= RS_THREADS)
        const int ex = block_exclusive_scan(threadIdx.x < NCLASS ? h[threadIdx.x] : 0, wsum, &tot);
        if (threadIdx.x < NCLASS) {
            h[threadIdx.x] = ex;
            coff[threadIdx.x] = ex;
        }
    }
    // new ids: stable rank by old id within the class, RS_THREADS vertices at a time
    for (int x0 = 0; x0 < n; x0 += RS_THREADS) {
        for (int i = threadIdx.x; i < NW * NCLASS; i += RS_THREADS) (&wc[0][0])[i] = 0;
        __syncthreads();
        const int x = x0 + threadIdx.x;
        const bool valid = x < n;
        const int d = valid ? deg[x] : 0;
        const int c = valid ? deg_class(d) : NCLASS + lane;   // invalid lanes match only themselves
        const unsigned peers = __match_any_sync(FULL, c);
        const int rank = __popc(peers & lanemask_lt());
        if (valid && rank == 0) wc[w][c] = __popc(peers);
        __syncthreads();
        if (threadIdx.x < NCLASS) {
            int run = h[threadIdx.x];
            for (int ww = 0; ww < NW; ++ww) {
                const int t = wc[ww][threadIdx.x];
                wc[ww][threadIdx.x] = run;
                run += t;
            }
            h[threadIdx.x] = run;
        }
        __syncthreads();
        if (valid) {
            const int id = wc[w][c] + rank;
            vinfo[x] = make_int2(id, d);
            perm[id] = x;
            nd[id] = d;
        }
        __syncthreads();
    }
    int carry = 0;   // new row offsets
    for (int i0 = 0; i0 < n; i0 += RS_THREADS) {
        const int i = i0 + threadIdx.x;
        const int ex = block_exclusive_scan(i < n ? nd[i] : 0, wsum, &tot);
        if (i < n) nrow[i] = carry + ex;
        carry += tot;
    }
    if (threadIdx.x == 0) nrow[n] = carry;
}

// Union id of a column entry: graphs of a batch store ids local to the graph,
// whose vertices occupy [vr.x, vr.y) of the union; -1 if out of range.
__device__ __forceinline__ int global_id(int y, int2 vr, int n) {
    const long long g = (long long)vr.x + y;
    return (y >= 0 && g < vr.y && g >= 0 && g < n) ? (int)g : -1;
}

__device__ __forceinline__ long long c2m1(int d) {  // C(d - 1, 2)
    long long a = d - 1;
    return a * (a - 1) / 2;
}

// Place of every active lane's entry among the entries of its group (a mask
// of the active lanes), stable by degree class: the entries of a lower class
// plus those of its own class before it, from ballots over the class bits. A
// bit that all active entries of the warp share costs its ballot only.
__device__ __forceinline__ int class_rank(int c, bool act, unsigned group) {
    static_assert(NCLASS <= 128, "classes fit seven bits");
    const unsigned all = __ballot_sync(FULL, act);
    unsigned eq = group, lt = 0;
#pragma unroll
    for (int bit = 6; bit >= 0; --bit) {
        const bool one = act && ((c >> bit) & 1);
        const unsigned ones = __ballot_sync(FULL, one);
        if (ones == 0 || ones == all) continue;
        if (one) lt |= eq & ~ones;
        eq &= one ? ones : ~ones;
    }
    return __popc(lt) + __popc(eq & lanemask_lt());
}

struct RelabelArgs {
    const int *rowptr, *colidx;
    int n;
    const int2 *vrange, *vinfo;
    const int *perm, *nrow, *coff;
    int ntiles;
    int *ncol;
    int4 *rinfo;
    VAcc *vacc;
    int *tcnt, *status;
    int long_class;
    int *counters;
};

// Rows x of at most L entries each, one per group of L lanes (x, r, d, ob are
// the group's; d = 0 for none): one entry per lane. Every lane stores one
// accumulator of its row, or a few (L = 8: the row's 64 bytes at once).
template <int L>
__device__ __forceinline__ int relabel_group(const RelabelArgs &A, int x, int r, int d, int ob, bool have) {
    const int lane = lane_id(), l = lane & (L - 1), first = lane & ~(L - 1);
    const int nb = have ? A.nrow[r] : 0;
    const bool act = l < d;
    int2 vr = make_int2(0, A.n);
    if (A.vrange && act) vr = A.vrange[x];
    const int y = act ? A.colidx[ob + l] : 0;
    const int yp = __shfl_up_sync(FULL, y, 1);
    int bad = 0, nid = 0, c = 0, dy = 0;
    if (act) {
        int ys = global_id(y, vr, A.n);
        if (ys < 0) { bad = ST_EINVAL; ys = x; }
        else if (ys == x || (l > 0 && y <= yp)) bad = ST_ENOTSIMPLE;
        const int2 vi = A.vinfo[ys];
        nid = vi.x;
        dy = vi.y;
        c = deg_class(dy);
    }
    const unsigned group = __ballot_sync(FULL, act) & ((L == 32 ? FULL : (1u << (L & 31)) - 1u) << first);
    const int rank = class_rank(c, act, group);
    if (act) A.ncol[nb + rank] = nid;
    const int below = __popc(__ballot_sync(FULL, act && nid < r) & group);
    // sums over the group: degrees (at most 2^20 each, 32 of them fit 32 bits) and C(d - 1, 2)
    unsigned s1 = (unsigned)dy;
    long long p6;
    if (L == 32) {
        s1 = __reduce_add_sync(FULL, s1);
    } else {
#pragma unroll
        for (int o = 1; o < L; o <<= 1) s1 += __shfl_xor_sync(FULL, s1, o);
    }
    if (!__any_sync(FULL, dy > 8192)) {   // C(8191, 2) < 2^25
        unsigned p = act ? (unsigned)(dy - 1) * (unsigned)(dy - 2) / 2u : 0u;
        if (L == 32) {
            p = __reduce_add_sync(FULL, p);
        } else {
#pragma unroll
            for (int o = 1; o < L; o <<= 1) p += __shfl_xor_sync(FULL, p, o);
        }
        p6 = p;
    } else {
        p6 = act ? c2m1(dy) : 0;
#pragma unroll
        for (int o = 1; o < L; o <<= 1) p6 += __shfl_xor_sync(FULL, p6, o);
    }
    const int sp = nb + below;
    if (have) {
        if (l == 0) A.rinfo[r] = make_int4(nb, sp, nb + d, 0);
        if (l < 8) reinterpret_cast<long long *>(&A.vacc[r])[l] = l == 0 ? (long long)s1 : l == 2 ? p6 : 0;   // S1, P6
    }
    if (sp + l < nb + d) A.tcnt[sp + l] = 0;
    return bad;
}

// A row of 33 to 64 entries, two per lane.
__device__ __forceinline__ int relabel_two(const RelabelArgs &A, int x, int r, int d, int ob) {
    const int lane = lane_id();
    const int nb = A.nrow[r];
    const int2 vr = A.vrange ? A.vrange[x] : make_int2(0, A.n);
    const bool act = 32 + lane < d;
    const int y0 = A.colidx[ob + lane], y1 = act ? A.colidx[ob + 32 + lane] : 0;
    const int p0 = __shfl_up_sync(FULL, y0, 1), mid = __shfl_sync(FULL, y0, 31);
    int p1 = __shfl_up_sync(FULL, y1, 1);
    if (lane == 0) p1 = mid;
    int bad = 0;
    auto look = [&](int y, int before, bool first) {
        int ys = global_id(y, vr, A.n);
        if (ys < 0) { bad |= ST_EINVAL; ys = x; }
        else if (ys == x || (!first && y <= before)) bad |= ST_ENOTSIMPLE;
        return A.vinfo[ys];
    };
    const int2 v0 = look(y0, p0, lane == 0);
    const int2 v1 = act ? look(y1, p1, false) : make_int2(0, 0);
    const int c0 = deg_class(v0.y), c1 = deg_class(v1.y);
    const unsigned in1 = __ballot_sync(FULL, act);
    // entries of a lower class / of the same class, in each half of the row
    unsigned eq00 = FULL, eq01 = in1, eq10 = FULL, eq11 = in1, lt00 = 0, lt01 = 0, lt10 = 0, lt11 = 0;
#pragma unroll
    for (int bit = 6; bit >= 0; --bit) {
        const bool b0 = (c0 >> bit) & 1, b1 = act && ((c1 >> bit) & 1);
        const unsigned o0 = __ballot_sync(FULL, b0), o1 = __ballot_sync(FULL, b1);
        if ((o0 | o1) == 0 || (o0 == FULL && o1 == in1)) continue;
        if (b0) { lt00 |= eq00 & ~o0; lt01 |= eq01 & ~o1; }
        eq00 &= b0 ? o0 : ~o0;
        eq01 &= b0 ? o1 : ~o1;
        if (b1) { lt10 |= eq10 & ~o0; lt11 |= eq11 & ~o1; }
        eq10 &= b1 ? o0 : ~o0;
        eq11 &= b1 ? o1 : ~o1;
    }
    A.ncol[nb + __popc(lt00) + __popc(lt01) + __popc(eq00 & lanemask_lt())] = v0.x;
    if (act) A.ncol[nb + __popc(lt10) + __popc(lt11) + __popc(eq10) + __popc(eq11 & lanemask_lt())] = v1.x;
    const int below = __popc(__ballot_sync(FULL, v0.x < r)) + __popc(__ballot_sync(FULL, act && v1.x < r));
    // 64 degrees of at most 2^20 fit 32 bits
    const long long s1 = __reduce_add_sync(FULL, (unsigned)(v0.y + v1.y));
    long long p6;
    if (!__any_sync(FULL, max(v0.y, v1.y) > 8192)) {   // 64 values below 2^25
        unsigned p = (unsigned)(v0.y - 1) * (unsigned)(v0.y - 2) / 2u;
        if (act) p += (unsigned)(v1.y - 1) * (unsigned)(v1.y - 2) / 2u;
        p6 = __reduce_add_sync(FULL, p);
    } else {
        p6 = warp_sum(c2m1(v0.y) + (act ? c2m1(v1.y) : 0ll));
    }
    const int sp = nb + below;
    if (lane == 0) A.rinfo[r] = make_int4(nb, sp, nb + d, 0);
    if (lane < 8) reinterpret_cast<long long *>(&A.vacc[r])[lane] = lane == 0 ? s1 : lane == 2 ? p6 : 0;   // S1, P6
    for (int p = sp + lane; p < nb + d; p += 32) A.tcnt[p] = 0;
    return bad;
}

// A row of more than 64 entries, one warp: pass 1 validates it, counts its
// classes (H) and sums neighbour degrees; pass 2 writes every new id at its
// class offset (stable within a class). With KEEP the first 64 entries stay in
// registers between the passes: read again, they cross the host link twice when
// the CSR is in host memory (G(4e5, mean degree 80): 1528 us, 997 so).
template <bool KEEP>
__device__ __forceinline__ int relabel_row(const RelabelArgs &A, int x, int r, int d, int ob, int *H) {
    const int lane = lane_id();
    const int nb = A.nrow[r];
    const int2 vr = A.vrange ? A.vrange[x] : make_int2(0, A.n);
    int bad = 0;
    for (int c = lane; c < NCLASS; c += 32) H[c] = 0;
    __syncwarp();
    long long s1 = 0, p6 = 0;
    int below = 0, last = -1;
    int nid0 = 0, c0 = 0, nid1 = 0, c1 = 0;   // new ids and classes of entries lane and 32 + lane
    for (int k = 0; k < d; k += 32) {
        const int i = k + lane;
        const bool act = i < d;
        const int y = act ? A.colidx[ob + i] : 0;
        int yp = __shfl_up_sync(FULL, y, 1);
        if (lane == 0) yp = last;
        last = __shfl_sync(FULL, y, 31);
        if (act) {
            int ys = global_id(y, vr, A.n);
            if (ys < 0) { bad |= ST_EINVAL; ys = x; }
            else if (ys == x || (i > 0 && y <= yp)) bad |= ST_ENOTSIMPLE;
            const int2 vi = A.vinfo[ys];
            const int c = deg_class(vi.y);
            atomicAdd(&H[c], 1);
            s1 += vi.y;
            p6 += c2m1(vi.y);
            below += vi.x < r;
            if (KEEP && k == 0) { nid0 = vi.x; c0 = c; }
            else if (KEEP && k == 32) { nid1 = vi.x; c1 = c; }
        }
    }
    // exclusive scan of the 128 class counts: 4 per lane
    __syncwarp();
    {
        int a0 = H[4 * lane], a1 = H[4 * lane + 1], a2 = H[4 * lane + 2], a3 = H[4 * lane + 3];
        int sum = a0 + a1 + a2 + a3;
        int ex = warp_inclusive_scan(sum) - sum;
        H[4 * lane] = ex;
        H[4 * lane + 1] = ex + a0;
        H[4 * lane + 2] = ex + a0 + a1;
        H[4 * lane + 3] = ex + a0 + a1 + a2;
    }
    __syncwarp();
    for (int k = 0; k < d; k += 32) {
        const int i = k + lane;
        const bool act = i < d;
        int nid = k == 0 ? nid0 : nid1, c = k == 0 ? c0 : c1;   // (the row has more than 64 entries)
        if (!KEEP || k >= 64) {
            int ys = act ? global_id(A.colidx[ob + i], vr, A.n) : 0;
            if (ys < 0) ys = x;
            const int2 vi = act ? A.vinfo[ys] : make_int2(0, 0);
            nid = vi.x;
            c = act ? deg_class(vi.y) : NCLASS + lane;
        }
        const unsigned peers = __match_any_sync(FULL, c);
        const int rank = __popc(peers & lanemask_lt());
        int pos = 0;
        if (act) pos = H[c] + rank;
        __syncwarp();
        if (act && rank == 0) H[c] += __popc(peers);
        __syncwarp();
        if (act) A.ncol[nb + pos] = nid;
    }
    s1 = warp_sum(s1);
    p6 = warp_sum(p6);
    below = warp_sum(below);
    const int sp = nb + below;
    if (lane == 0) A.rinfo[r] = make_int4(nb, sp, nb + d, 0);
    if (lane < 8) reinterpret_cast<long long *>(&A.vacc[r])[lane] = lane == 0 ? s1 : lane == 2 ? p6 : 0;   // S1, P6
    for (int p = sp + lane; p < nb + d; p += 32) A.tcnt[p] = 0;
    __syncwarp();
    return bad;
}

// A long row (from LONG_ROW_CLASS on), the whole CTA: every warp counts and
// then places a part of the row of its own, U steps of 32 entries in flight,
// with the CTA's barriers between the two passes only. (Placing 256 entries
// at a time, with five barriers each, took 5.9 ms for a row of 1e6 entries,
// 3.1 ms with 512 threads; 3.0 ms now, R-MAT 18 261 -> 197 us a call.)
constexpr int RLR_THREADS = 256;
struct LongRowSmem {
    int H[NCLASS];
    int wc[RLR_THREADS / 32][NCLASS];
    long long red[3][RLR_THREADS / 32];
};
__device__ __forceinline__ int relabel_long(const RelabelArgs &A, int r, LongRowSmem &S) {
    constexpr int NW = RLR_THREADS / 32, U = 4;
    const int lane = lane_id(), w = threadIdx.x >> 5;
    int bad = 0;
    const int x = A.perm[r];
    const int nb = A.nrow[r], d = A.nrow[r + 1] - nb;
    const int ob = d > 0 ? A.rowptr[x] : 0;
    const int2 vr = A.vrange ? A.vrange[x] : make_int2(0, A.n);
    const int part = (d / (NW * 32) + 1) * 32, lo = min(d, w * part), len = min(part, d - lo);   // (no sum passes 2^31)
    int *const wc = S.wc[w];
    for (int c = lane; c < NCLASS; c += 32) wc[c] = 0;
    __syncwarp();
    const int *const col = A.colidx + ob + lo;   // the warp's part
    // its entries k + 32 h + lane, h < U: caller id, new id and degree (`left`: entries from k on)
    auto load = [&](int k, int left, int (&y)[U], int2 (&vi)[U]) {
#pragma unroll
        for (int h = 0; h < U; ++h) y[h] = 32 * h + lane < left ? col[k + 32 * h + lane] : 0;
#pragma unroll
        for (int h = 0; h < U; ++h) {
            vi[h] = make_int2(0, 0);
            if (32 * h + lane < left) {
                const int ys = global_id(y[h], vr, A.n);
                vi[h] = A.vinfo[ys < 0 ? x : ys];
            }
        }
    };
    long long s1 = 0, p6 = 0, below = 0;
    for (int k = 0, left = len; left > 0; k += 32 * U, left -= 32 * U) {
        int y[U];
        int2 vi[U];
        load(k, left, y, vi);
#pragma unroll
        for (int h = 0; h < U; ++h) {
            if (32 * h + lane >= left) continue;
            const int i = k + 32 * h + lane, ys = global_id(y[h], vr, A.n);
            if (ys < 0) bad |= ST_EINVAL;
            else if (ys == x || (lo + i > 0 && y[h] <= col[i - 1])) bad |= ST_ENOTSIMPLE;
            atomicAdd(&wc[deg_class(vi[h].y)], 1);
            s1 += vi[h].y;
            p6 += c2m1(vi[h].y);
            below += vi[h].x < r;
        }
    }
    s1 = warp_sum(s1);
    p6 = warp_sum(p6);
    below = warp_sum(below);
    if (lane == 0) { S.red[0][w] = s1; S.red[1][w] = p6; S.red[2][w] = below; }
    __syncthreads();
    if (threadIdx.x < NCLASS) {   // entries of the class in the parts before
        int sum = 0;
        for (int ww = 0; ww < NW; ++ww) {
            const int t = S.wc[ww][threadIdx.x];
            S.wc[ww][threadIdx.x] = sum;
            sum += t;
        }
        S.H[threadIdx.x] = sum;
    }
    __syncthreads();
    if (w == 0) {
        int a0 = S.H[4 * lane], a1 = S.H[4 * lane + 1], a2 = S.H[4 * lane + 2], a3 = S.H[4 * lane + 3];
        int sum = a0 + a1 + a2 + a3;
        int ex = warp_inclusive_scan(sum) - sum;
        S.H[4 * lane] = ex;
        S.H[4 * lane + 1] = ex + a0;
        S.H[4 * lane + 2] = ex + a0 + a1;
        S.H[4 * lane + 3] = ex + a0 + a1 + a2;
    }
    __syncthreads();
    for (int k = 0, left = len; left > 0; k += 32 * U, left -= 32 * U) {
        int y[U];
        int2 vi[U];
        load(k, left, y, vi);
#pragma unroll
        for (int h = 0; h < U; ++h) {
            if (32 * h >= left) break;
            const bool act = 32 * h + lane < left;
            const int c = act ? deg_class(vi[h].y) : NCLASS + lane;   // inactive lanes match only themselves
            const unsigned peers = __match_any_sync(FULL, c);
            const int rank = __popc(peers & lanemask_lt());
            int pos = 0;
            if (act) pos = S.H[c] + wc[c] + rank;
            __syncwarp();
            if (act && rank == 0) wc[c] += __popc(peers);
            __syncwarp();
            if (act) A.ncol[nb + pos] = vi[h].x;
        }
    }
    long long a = 0, b = 0, c = 0;
    for (int ww = 0; ww < NW; ++ww) { a += S.red[0][ww]; b += S.red[1][ww]; c += S.red[2][ww]; }
    const int sp = nb + (int)c;
    if (threadIdx.x == 0) A.rinfo[r] = make_int4(nb, sp, nb + d, 0);
    if (threadIdx.x < 8)
        reinterpret_cast<long long *>(&A.vacc[r])[threadIdx.x] = threadIdx.x == 0 ? a : threadIdx.x == 2 ? b : 0;   // S1, P6
    for (int p = sp + threadIdx.x; p < nb + d; p += RLR_THREADS) A.tcnt[p] = 0;
    __syncthreads();
    return bad;
}

// Row relabelling. Long rows first, a CTA each; then the others, taken in
// input order so that they are read sequentially and written scattered. A
// warp takes one row at a time, or, with FOUR, four: rows of at most 8
// entries at once (eight lanes each), of at most 16 in pairs, longer ones in
// turn. A row is a chain of four dependent loads, so FOUR pays where rows are
// short (G(3e6, mean degree 6): 861 -> 410 us; 433 with KEEP, which needs
// registers that its code for short rows misses) and where every warp has many
// rows (a power-law graph of 1e5 vertices: 44 us alone, 74 us by fours).
template <bool FOUR>
__global__ void __launch_bounds__(RLR_THREADS, 6) k_relabel_rows(RelabelArgs A) {
    pdl_begin();
    __shared__ union {
        int H[RLR_THREADS / 32][NCLASS];
        LongRowSmem S;
    } sm;
    const int stop = A.counters[CNT_BAD_OFFSETS], bound = A.coff[A.long_class * A.ntiles];   // (loaded together)
    if (stop) return;
    int bad = 0;
    for (int r = bound + blockIdx.x; r < A.n; r += gridDim.x) bad |= relabel_long(A, r, sm.S);
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    auto row = [&](int x, int r, int d, int ob) {
        if (d <= 32) bad |= relabel_group<32>(A, x, r, d, ob, true);
        else if (d <= 64) bad |= relabel_two(A, x, r, d, ob);
        else bad |= relabel_row<!FOUR>(A, x, r, d, ob, sm.H[threadIdx.x >> 5]);
    };
    for (int x = FOUR ? A.n : gw; x < A.n; x += nw) {
        const int2 vx = A.vinfo[x];   // new id, degree
        if (deg_class(vx.y) < A.long_class) row(x, vx.x, vx.y, vx.y > 0 ? A.rowptr[x] : 0);
    }
    for (long long x0 = FOUR ? 4ll * gw : A.n; x0 < A.n; x0 += 4ll * nw) {
        // lanes 8 q ..: row x0 + q
        const int x = (int)min(x0 + (lane >> 3), (long long)A.n - 1);
        bool have = x0 + (lane >> 3) < A.n;
        const int2 vx = A.vinfo[x];
        const int r = vx.x;
        int d = vx.y;
        const int ob = d > 0 ? A.rowptr[x] : 0;
        if (deg_class(d) >= A.long_class) have = false;   // done by a CTA
        if (!have) d = 0;
        const int top = (int)__reduce_max_sync(FULL, (unsigned)d);
        if (top <= 8) {
            bad |= relabel_group<8>(A, x, r, d, ob, have);
            continue;
        }
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            const int src = top <= 16 ? 8 * (q + (lane >> 4)) : 8 * q;
            const int xq = __shfl_sync(FULL, x, src), rq = __shfl_sync(FULL, r, src), dq = __shfl_sync(FULL, d, src);
            const int oq = __shfl_sync(FULL, ob, src);
            const bool hq = __shfl_sync(FULL, (int)have, src);
            if (top <= 16) {
                bad |= relabel_group<16>(A, xq, rq, dq, oq, hq);
                ++q;
            } else if (hq) {
                row(xq, rq, dq, oq);
            }
        }
    }
    bad = __reduce_or_sync(FULL, bad);
    if (lane == 0 && bad) {
        set_status(A.status, bad);
        atomicOr(&A.counters[CNT_BAD_ROWS], 1);
    }
}

static void relabel_common(const int *rowptr, const int *colidx, const int2 *vrange, Work &w, cudaStream_t st) {
    const int nt = w.ntiles;
    if (nt == 1) {   // one tile: the class order in one launch
        launch_pdl(k_class_small, 1, RS_THREADS, 0, st, rowptr, w.n, w.m, w.vinfo, w.coff, w.perm, w.nrow, w.counters,
                   w.status);
        after_launch(st, K_CLASS_HIST);
    } else {
        launch_pdl(k_class_hist, nt, RL_THREADS, 0, st, rowptr, w.n, w.m, w.vinfo, w.chist, nt, w.counters, w.status);
        after_launch(st, K_CLASS_HIST);
        launch_exclusive_scan(w.chist, w.coff, (long long)NCLASS * nt, false, w.scan_part, w.counters + CNT_SCAN_DONE, st);
        // ndeg (degree of each new id) is staged in `split`, then scanned into nrow
        launch_pdl(k_class_scatter, nt, RL_THREADS, 0, st, w.n, w.vinfo, w.coff, nt, w.perm, w.split);
        after_launch(st, K_CLASS_SCATTER);
        launch_exclusive_scan(w.split, w.nrow, w.n, true, w.scan_part, w.counters + CNT_SCAN_DONE, st);
    }
    // more CTAs than an SM holds: with rows of uneven length, the later
    // waves act as load balancing
    const RelabelArgs A{rowptr, colidx, w.n, vrange, w.vinfo, w.perm, w.nrow, w.coff, nt, w.ncol, w.rinfo, w.vacc, w.tcnt,
                        w.status, w.tune[TUNE_LONG_ROW_CLASS], w.counters};
    const int grid = w.num_sms * w.tune[TUNE_GRID_RELABEL];
    // by fours: short rows, and at least 32 rows for every warp of the grid
    const bool four = w.m < 16ll * w.n && w.n >= 32ll * grid * (RLR_THREADS / 32) / 4;
    if (four) launch_pdl(k_relabel_rows<true>, grid, RLR_THREADS, 0, st, A);
    else launch_pdl(k_relabel_rows<false>, grid, RLR_THREADS, 0, st, A);
    after_launch(st, K_RELABEL);
}

void launch_relabel(const int *rowptr, const int *colidx, Work &w, cudaStream_t st) {
    relabel_common(rowptr, colidx, nullptr, w, st);
}

void launch_relabel_batch(const int *rowptr, const int *colidx, const int2 *vrange, Work &w, cudaStream_t st) {
    relabel_common(rowptr, colidx, vrange, w, st);
}

// Batch set-up: the union-id range of the graph that owns every vertex, and
// consistency of the offsets with rowptr.
__global__ void k_batch_setup(const int *rowptr, const long long *vo, const long long *eo, int G, int total_n,
                              int2 *vrange, int *status) {
    pdl_begin();
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long nthreads = (long long)gridDim.x * blockDim.x;
    int bad = 0;
    for (long long g = tid; g <= G; g += nthreads) {
        const long long a = vo[g];
        if (a < 0 || a > total_n || (g == 0 && a != 0) || (g == G && a != total_n)) bad = 1;
        else if (g < G && vo[g + 1] < a) bad = 1;
        else if (eo[g] != (long long)rowptr[a]) bad = 1;
    }
    for (long long x = tid; x < total_n; x += nthreads) {
        int lo = 0, hi = G - 1;  // last g with vo[g] <= x
        while (lo < hi) {
            int mid = (lo + hi + 1) >> 1;
            if (vo[mid] <= x) lo = mid; else hi = mid - 1;
        }
        long long a = vo[lo], b = vo[lo + 1];
        if (a < 0 || b > total_n || a > x || b <= x) { bad = 1; a = x; b = x + 1; }
        vrange[x] = make_int2((int)a, (int)b);
    }
    if (bad) set_status(status, ST_EINVAL);
}

void launch_batch_setup(const int *rowptr, const long long *vtx_offset, const long long *edge_offset, int num_graphs,
                        int total_n, int2 *vrange, int *status, int num_sms, cudaStream_t st) {
    launch_pdl(k_batch_setup, num_sms * 4, 256, 0, st, rowptr, vtx_offset, edge_offset, num_graphs, total_n, vrange, status);
    after_launch(st, K_BATCH_SETUP);
}

}  // namespace niorca
