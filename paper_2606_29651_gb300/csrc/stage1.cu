// stage1.cu -- Stage I (per-edge triangle counts, Algorithm 1) fused with
// Stage II (K4 per vertex, Algorithm 2).
//
// In the relabelled graph every triangle u < v < w is found once, at its
// lowest vertex u, as w in N+(u) ∩ N+(v) (Algorithm 2 enumerates the same
// way with ids). Two ways to intersect, by graph (k_adj_bits decides):
//   - hubs: the rows N+(v) of a skewed graph are long whatever the length of
//     N+(u) (on R-MAT 22 a mean of 360 to 540 entries for roots of any
//     out-degree), so the pairs (v, w) of N+(u) are probed in an adjacency
//     bitmap of the hubs instead (adj.cuh): 7e9 tests there, against 2.8e10
//     entries to stream;
//   - no hubs: N+(v) of every v in N+(u) is streamed past a bit filter of
//     N+(u) (warp tier) or a hash of it (CTA tiers).
// A hit is a triangle (u, v, w): t(v,w) is added to global memory at the
// position of w in row v (for a probe: a prefix count and a popcount), and
// the hit sets R[j] bit i and R[i] bit j of the symmetric adjacency
// bit-matrix of N+(u) (v = N+(u)[j], w = N+(u)[i]). The K4s of u are the
// triangles of R, counted from common bits of adjacent rows (Algorithm 2's
// pairwise test over `neigh` as word-wide bit operations), so the cost follows
// the edges of R and not the (much larger) number of K4s of dense hub
// neighbourhoods.
//
// Measured on GB300, triangle and aggregate stages together: R-MAT 22 220 ->
// 91 ms, R-MAT 18 5.9 -> 2.8 ms, G(1501, 0.5) 3.3 -> 2.0 ms, against hash
// probes of every streamed entry; G(3e6, mean degree 6) 1.40 -> 0.41 ms and
// 8192 power-law graphs in a batch 6.6 -> 3.2 ms with four small roots per warp.
#include "kernels.h"

namespace niorca {

// ----------------------------------------------------------- warp tier

constexpr int TW_MAXD = 64;   // out-degree handled by one warp
constexpr int TS_MAXD = 256;  // out-degree handled by a 256-thread CTA (k_tri_cta)
constexpr int TW_WARPS = 8;

struct __align__(16) TriWarpSmem {
    Filter filter;
    int cnt[TW_MAXD];
    unsigned R[TW_MAXD][2];
};

// K4s of a warp-tier root from its symmetric bit matrix R, a row per lane: the
// triangles of R through y number half the common bits of y's row and its
// neighbours' rows.
__device__ __forceinline__ void warp_k4(const Graph &g, VAcc *vacc, int u, int s, int dp, const unsigned (*R)[2]) {
    const int lane = lane_id();
    unsigned ku = 0;
    for (int y = lane; y < dp; y += 32) {
        const uint2 ry = *reinterpret_cast<const uint2 *>(R[y]);
        unsigned k = 0;
        for (unsigned m = ry.x; m; m &= m - 1) {
            const uint2 rz = *reinterpret_cast<const uint2 *>(R[__ffs(m) - 1]);
            k += __popc(ry.x & rz.x) + __popc(ry.y & rz.y);
        }
        for (unsigned m = ry.y; m; m &= m - 1) {
            const uint2 rz = *reinterpret_cast<const uint2 *>(R[31 + __ffs(m)]);
            k += __popc(ry.x & rz.x) + __popc(ry.y & rz.y);
        }
        if (!k) continue;
        ku += k;
        add64(&vacc[g.ncol[s + y]].K4, k / 2);
    }
    ku = __reduce_add_sync(FULL, ku);   // each K4 at three of N+(u), twice
    if (lane == 0 && ku) add64(&vacc[u].K4, ku / 6);
    __syncwarp();
}

// ------------------------------------------------- adjacency bitmap

// Words of the bitmap, one thread each: its entries' position in N+(v) by a
// search, then the few entries themselves. Also decides whether the call's
// triangle and aggregate stages probe (CNT_ADJ_ON): at least half of the
// entries belong to vertices with a bitmap row, and those are hubs (at least
// twice their share) or all vertices. Without hubs, out-lists are as short as
// the rows they point at and streaming is as good (G(3213, mean degree 31):
// 118 us a call streamed, 134 us probed with a bitmap of 2/3 of the rows). A
// malformed graph (rows out of order) is not probed: the positions rely on
// sorted rows.
__global__ void __launch_bounds__(256) k_adj_bits(Graph g, AdjBits A, const int *nrow, unsigned *words,
                                                  unsigned short *prefix, int *counters) {
    pdl_begin();
    if (call_stopped(counters)) return;
    const int total = nrow[g.n];
    const long long own = total - nrow[A.base], rows = g.n - A.base;
    const bool on = rows > 0 && !counters[CNT_BAD_ROWS] && 2 * own >= total &&
                    (A.base == 0 || own * g.n >= 2 * rows * total);
    if (blockIdx.x == 0 && threadIdx.x == 0) counters[CNT_ADJ_ON] = on;
    if (!on) return;
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    for (int v = A.base + gw; v < g.n; v += nw) {   // longest rows first
        const int4 rv = g.rinfo[v];
        const int at = A.row(v), nq = ((g.n - 1 - v) >> 5) + 1;
        const int y = rv.y, z = rv.z - y < 65536 ? rv.z : y;   // (more out-entries: only in an asymmetric CSR)
        for (int q = lane; q < nq; q += 32) {
            const int top = g.n - 1 - 32 * q;   // id of bit 0
            int p = lower_bound(g.ncol, y, z, top - 31);
            prefix[at + q] = (unsigned short)(p - y);
            unsigned bits = 0;
            for (; p < z; ++p) {
                const int k = top - g.ncol[p];
                if (k < 0) break;
                bits |= 1u << k;
            }
            words[at + q] = bits;
        }
    }
}

AdjBits adj_bits(const Work &w) {
    // 6 bytes per word (word and prefix) in 4 m bytes
    long long lo = 0, hi = w.n;
    while (lo < hi) {
        const long long mid = (lo + hi + 1) / 2;
        if (6 * AdjBits::row_words(mid) <= 4ll * w.m) lo = mid; else hi = mid - 1;
    }
    AdjBits A;
    A.words = reinterpret_cast<const unsigned *>(w.tcnt + w.m);
    A.prefix = reinterpret_cast<const unsigned short *>(A.words + AdjBits::row_words(lo));
    A.n = w.n;
    A.base = w.n - (int)lo;
    return A;
}

// One warp-tier root over the adjacency bitmap: its pairs of out-neighbours
// are probed 32 columns at a time, dp^2 / 2 tests instead of the sum of its
// out-neighbours' row lengths. A ballot is a row of R, and a lane counts its
// own column.
__device__ __forceinline__ void tri_root_probe(const Graph &g, const AdjBits &A, int *tcnt, VAcc *vacc, int u, int s, int dp,
                                               TriWarpSmem &S) {
    const int lane = lane_id();
    const OutList L = out_list(g, A, s, dp);
    int c0 = 0, c1 = 0;                        // t(u, .) of entries lane, 32 + lane
    unsigned r00 = 0, r01 = 0, r10 = 0, r11 = 0;   // the lane's rows of the symmetric R: entry lane, 32 + lane
    out_pairs(g, A, L, FULL, FULL, lane < dp, 32 + lane < dp, [&](int b, int r, bool hit, int pos) {
        const unsigned bal = __ballot_sync(FULL, hit);
        if (hit) {
            atomicAdd(&tcnt[pos], 1);
            if (b == 0) { ++c0; r00 |= 1u << r; }
            else if (b == 1) { ++c1; r10 |= 1u << r; }
            else { ++c1; r11 |= 1u << r; }
        }
        if (lane == r) {
            if (b == 0) r00 |= bal;
            else if (b == 1) r01 = bal;
            else r11 |= bal;
            if (b == 2) c1 += __popc(bal); else c0 += __popc(bal);
        }
    });
    if (!__any_sync(FULL, c0 | c1)) return;
    if (c0) atomicAdd(&tcnt[s + lane], c0);
    if (c1) atomicAdd(&tcnt[s + 32 + lane], c1);
    S.R[lane][0] = r00;
    S.R[lane][1] = r01;
    S.R[32 + lane][0] = r10;
    S.R[32 + lane][1] = r11;
    __syncwarp();
    warp_k4(g, vacc, u, s, dp, S.R);
}

// One warp-tier root whose out-neighbours' rows (r0, r1: entries lane and 32
// + lane, ids w0, w1) are streamed past a filter of N+(u).
__device__ __forceinline__ void tri_root_stream(const Graph &g, int *tcnt, VAcc *vacc, int u, int s, int dp, TriWarpSmem &S) {
    const int lane = lane_id();
    int w0 = -1, w1 = -1;
    int2 r0 = make_int2(0, 0), r1 = r0;
    auto fill = [&](int i, int &w, int2 &r) {
        if (i >= dp) return;
        w = g.ncol[s + i];
        if (i == dp - 1) return;   // the last out-neighbour has no row to walk
        const int4 rw = g.rinfo[w];
        r = make_int2(rw.y, rw.z);
    };
    fill(lane, w0, r0);
    if (dp > 32) fill(32 + lane, w1, r1);
    S.filter.set(w0, w1, w0 >= 0, w1 >= 0);
    S.cnt[lane] = S.cnt[32 + lane] = 0;
    *reinterpret_cast<uint4 *>(S.R[2 * lane]) = make_uint4(0, 0, 0, 0);
    __syncwarp();
    bool found = false;
    filter_walk(g.ncol, S.filter, r0, r1, dp, [&](int j, int pos, int w) {
        const int i = S.filter.find(w, dp);
        if (i < 0) return;
        atomicAdd(&S.cnt[j], 1);
        atomicAdd(&S.cnt[i], 1);
        atomicOr(&S.R[j][i >> 5], 1u << (i & 31));
        atomicOr(&S.R[i][j >> 5], 1u << (j & 31));
        atomicAdd(&tcnt[pos], 1);
        found = true;
    });
    if (!__any_sync(FULL, found)) return;
    __syncwarp();
    for (int i = lane; i < dp; i += 32)
        if (S.cnt[i]) atomicAdd(&tcnt[s + i], S.cnt[i]);
    warp_k4(g, vacc, u, s, dp, S.R);
}

// Four roots of out-degree at most 8, eight lanes each (lane 8 q + l: entry l
// of root q, id w, row r).
__device__ __forceinline__ void tri_roots_small(const Graph &g, int *tcnt, VAcc *vacc, int u, int s, int dp, int w, int2 r) {
    const int lane = lane_id(), l = lane & 7;
    unsigned R = 0;   // the lane's row of the root's oriented 8 x 8 matrix
    int t = 0;
    small_walk(g.ncol, w, r, [&](int pos, int x) {
        for (int i = l + 1; i < dp; ++i)
            if (g.ncol[s + i] == x) {
                R |= 1u << i;
                ++t;
                atomicAdd(&tcnt[s + i], 1);
                atomicAdd(&tcnt[pos], 1);
            }
    });
    if (t) atomicAdd(&tcnt[s + l], t);
    if (!__any_sync(FULL, R & (R - 1))) return;   // a K4 has two triangles in the row of its second vertex
    for (int i = 1; i < 8; ++i) {
        const unsigned Ri = __shfl_sync(FULL, R, (lane & 24) | i);
        unsigned x = (R >> i) & 1u ? R & Ri : 0u;
        if (!x) continue;
        const int k = __popc(x);
        add64(&vacc[u].K4, k);
        add64(&vacc[w].K4, k);
        add64(&vacc[g.ncol[s + i]].K4, k);
        for (; x; x &= x - 1) add64(&vacc[g.ncol[s + __ffs(x) - 1]].K4, 1);
    }
}

// The warp tier, over the adjacency bitmap when the call has one, else
// streaming rows. Six CTAs per SM (40 registers): eight make the streaming
// path spill more than the occupancy gains (G(1e6, mean degree 32): 641
// against 539 us).
__global__ void __launch_bounds__(TW_WARPS * 32, 6) k_tri_warp(Graph g, AdjBits A, int *tcnt, VAcc *vacc, int *heavy,
                                                            int *counters, int maxd, const int *coff, int ntiles) {
    pdl_begin();
    __shared__ TriWarpSmem sm_all[TW_WARPS];
    TriWarpSmem &S = sm_all[threadIdx.x >> 5];
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    if (call_stopped(counters)) return;
    const bool probe = counters[CNT_ADJ_ON];
    auto root = [&](int u, int s, int dp) {
        if (dp < 2) return;
        if (dp > maxd) {
            if (lane == 0) {
                if (dp <= TS_MAXD) heavy[atomicAdd(&counters[CNT_TRI_HEAVY], 1)] = u;
                else heavy[g.n - 1 - atomicAdd(&counters[CNT_TRI_BIG], 1)] = u;
            }
            return;
        }
        if (probe) tri_root_probe(g, A, tcnt, vacc, u, s, dp, S);
        else tri_root_stream(g, tcnt, vacc, u, s, dp, S);
        __syncwarp();
    };
    // ids of low degree: four roots at a time, eight lanes each
    const int low = probe ? 0 : low_degree_ids(g.n, nw, coff, ntiles);
    for (long long u0 = 4ll * gw; u0 < low; u0 += 4ll * nw) {
        const int u = (int)u0 + (lane >> 3), l = lane & 7;
        int4 ru = make_int4(0, 0, 0, 0);
        if (u < low) ru = g.rinfo[u];
        const int s = ru.y, dp = ru.z - s;
        if (!__any_sync(FULL, dp > min(SMALL_DP, maxd))) {
            int w = -1;
            int2 r = make_int2(0, 0);
            if (dp >= 2 && l < dp) {
                w = g.ncol[s + l];
                if (l < dp - 1) {
                    const int4 rw = g.rinfo[w];
                    r = make_int2(rw.y, rw.z);
                }
            }
            if (!__any_sync(FULL, r.y - r.x > SMALL_ROW)) {
                tri_roots_small(g, tcnt, vacc, u, s, dp, w, r);
                continue;
            }
        }
        for (int q = 0; q < 4; ++q) root((int)u0 + q, __shfl_sync(FULL, s, 8 * q), __shfl_sync(FULL, dp, 8 * q));
    }
    for (int u = low + gw; u < g.n; u += nw) {
        const int4 ru = g.rinfo[u];
        root(u, ru.y, ru.z - ru.y);
    }
}

// ------------------------------------------------------------ CTA tiers

// Roots with out-degree above the warp tier get a CTA each, in two sizes:
// k_tri_cta (256 threads, dp <= TS_MAXD) needs 26 KB of shared memory,
// so several CTAs share an SM; k_tri_big (1024 threads) takes the rest with
// the bit matrix R up to TB_BITMAT_MAXD (hash of N+(u) capped at 4096 slots),
// a 16384-slot hash up to TB_HASH_MAXD, and binary searches beyond.
// k_tri_warp queues the first kind from the front of the heavy list and the
// second from its back.
constexpr int TS_THREADS = 256;
constexpr int TB_THREADS = 1024;
constexpr int TB_BITMAT_MAXD = 1152;
constexpr int TB_BITMAT_HSLOTS = 4096;
constexpr int TB_HASH_MAXD = 8192;

// Dynamic shared memory of one CTA: hash keys + values (hslots), cnt + kc
// (nloc), per warp a segment table and a 64-entry buffer of row indices,
// 4 work words, and R (rows of an odd number of 16-byte groups, to spread the
// banks).
__host__ __device__ constexpr int tc_rowstride(int rows) { return ((rows + 127) / 128 | 1) * 4; }
constexpr size_t tc_smem(int threads, int hslots, int nloc, int rows) {
    return (size_t)2 * hslots * 4 + (size_t)2 * nloc * 4 + (size_t)(threads / 32) * (sizeof(SegTab) + 128) + 16 +
           (size_t)rows * tc_rowstride(rows) * 4;
}
constexpr size_t TS_SMEM = tc_smem(TS_THREADS, 4 * TS_MAXD, TS_MAXD, TS_MAXD);
constexpr size_t TB_SMEM_BITS = tc_smem(TB_THREADS, TB_BITMAT_HSLOTS, TB_BITMAT_MAXD, TB_BITMAT_MAXD);
constexpr size_t TB_SMEM_HASH = tc_smem(TB_THREADS, 2 * TB_HASH_MAXD, TB_HASH_MAXD, 0);
constexpr size_t TB_SMEM = TB_SMEM_BITS > TB_SMEM_HASH ? TB_SMEM_BITS : TB_SMEM_HASH;
static_assert(TB_SMEM <= 227 * 1024, "k_tri_big shared memory");

__device__ __forceinline__ int out_index(const int *hk, const int *hv, unsigned mask, bool use_hash, const int *ncol,
                                         int s, int e, int w) {
    if (use_hash) return hset_find(hk, hv, mask, w);
    int p = find_sorted(ncol, s, e, w);
    return p < 0 ? -1 : p - s;
}

// One CTA per root u of the list (roots list[0 .. count) or, with BACK,
// list[n - 1], list[n - 2], ...). A root keeps the bit matrix R up to
// bits_maxd and the hash of N+(u) up to hash_maxd (run-time limits no larger
// than the compiled ones, bits_maxd <= hash_maxd), else it probes N+(u) by
// binary search and enumerates the K4 of each triangle.
template <int THREADS, int BITMAT_MAXD, int BITMAT_HSLOTS, int HASH_MAXD, bool BACK, int HMUL>
__device__ __forceinline__ void tri_cta(const Graph &g, const AdjBits &A, bool probe, int *tcnt, VAcc *vacc,
                                        const int *list, int count, int *next, int bits_maxd, int hash_maxd) {
    extern __shared__ __align__(16) unsigned char dsm[];
    constexpr int TC_THREADS = THREADS;
    constexpr int NW = THREADS / 32;
    __shared__ long long s_ku;   // K4s of the root, three times each
    if (threadIdx.x == 0) s_ku = 0;
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    for (int h = cta_next(next); h < count; h = cta_next(next)) {
        const int u = BACK ? list[g.n - 1 - h] : list[h];
        const int4 ru = g.rinfo[u];
        const int s = ru.y, e = ru.z, dp = e - s;
        const bool use_hash = dp <= HASH_MAXD && dp <= hash_maxd;
        const bool use_bits = use_hash && dp <= BITMAT_MAXD && dp <= bits_maxd;
        // rows js .. of N+(u) are probed in the bitmap, the ones before streamed
        const int js = use_bits && probe ? lower_bound(g.ncol, s, e, A.base) - s : dp;
        unsigned H = use_hash && js > 0 ? next_pow2(HMUL * dp) : 0;   // hash load at most 1 / HMUL, within the carve:
        const unsigned hcap = use_bits ? BITMAT_HSLOTS : 2 * HASH_MAXD;   // its mode's slots
        if (H > hcap) H = hcap;
        const unsigned mask = H ? H - 1 : 0;
        const int W = (dp + 31) >> 5;  // bit-matrix words per row
        const int WP = tc_rowstride(dp);   // row stride of R
        // carve shared memory
        // beyond HASH_MAXD the per-position counters live in global memory
        const int nloc = use_hash ? dp : 0;
        int *hk = reinterpret_cast<int *>(dsm);
        int *hv = hk + H;
        int *cnt = hv + H;
        int *kc = cnt + ((nloc + 1) & ~1);
        SegTab *segs = reinterpret_cast<SegTab *>(kc + ((nloc + 1) & ~1));   // one per warp
        unsigned short *zb = reinterpret_cast<unsigned short *>(segs + NW) + wid * 64;  // 64 per warp
        int *work = reinterpret_cast<int *>(reinterpret_cast<unsigned short *>(segs + NW) + NW * 64);
        unsigned *R = reinterpret_cast<unsigned *>(work + 4);
        SegTab &seg = segs[wid];
        for (int i = threadIdx.x; i < (int)H; i += TC_THREADS) hk[i] = -1;
        for (int i = threadIdx.x; i < nloc; i += TC_THREADS) { cnt[i] = 0; kc[i] = 0; }
        if (use_bits)
            for (int i = threadIdx.x; i < dp * WP; i += TC_THREADS) R[i] = 0;
        if (threadIdx.x < 4) work[threadIdx.x] = 0;
        __syncthreads();
        if (H)
            for (int i = threadIdx.x; i < dp; i += TC_THREADS) hset_insert(hk, hv, mask, g.ncol[s + i], i);
        const int umax = g.ncol[e - 1];
        long long ku = 0;
        if (js < dp) {
            // Probe blocks of 32 rows x 32 columns (rows jb, columns t >= jb), a
            // warp each: a ballot is a row's word of R, a lane's hits over the
            // rows the word of its mirror image.
            const int b0 = js >> 5;   // the first block of rows
            for (int it = b0 * (b0 + 1) / 2 + wid; it < W * (W + 1) / 2; it += NW) {
                int t, jb;
                block_pair(it, t, jb);
                if (jb < b0) continue;
                const int i = 32 * t + lane, j = 32 * jb + lane;
                const int k = i < dp ? g.n - 1 - g.ncol[s + i] : 0;
                int roff = 0, ry = 0;
                if (j >= js && j < dp) {
                    const int v = g.ncol[s + j];
                    roff = A.row(v);
                    ry = g.rinfo[v].y;
                }
                const bool diag = t == jb;
                unsigned row = 0, col = 0;
                const unsigned rows = __ballot_sync(FULL, j >= js && j < dp - 1);
                adj_probe<(THREADS > 256 ? 8 : 4), false>(A, rows, roff, ry, k, i < dp, diag, nullptr,
                                                          [&](int r, bool hit, int pos, int) {
                    const unsigned bal = __ballot_sync(FULL, hit);
                    if (lane == r) row = bal;
                    if (hit) {
                        col |= 1u << r;
                        atomicAdd(&tcnt[pos], 1);
                    }
                });
                if (diag) {
                    if (i < dp) R[i * WP + t] = row | col;
                } else {
                    if (j < dp) R[j * WP + t] = row;
                    if (i < dp) R[i * WP + jb] = col;
                }
            }
        }
        __syncthreads();
        // every warp takes every chunk of 32 out-neighbours and the windows
        // wid, wid + NW, ... of its concatenated lists: no warp waits on a
        // larger chunk of another
        const int jend = min(js, dp - 1);   // the last out-neighbour has no row to walk
        for (int jb = 0; jb < jend; jb += 32) {
            const int j = jb + lane;
            int len = 0, vs = 0;
            if (j < jend) {
                const int4 rv = g.rinfo[g.ncol[s + j]];
                vs = rv.y;
                len = rv.z - rv.y;
            }
            int mypre;
            const int total = seg_build(seg, vs, len, mypre);
            seg_visit<4, true>(g.ncol, seg, mypre, len, total, wid * 32, NW * 32, [&](bool valid, int q, int pos, int w) {
                const int i = (valid && w <= umax) ? out_index(hk, hv, mask, use_hash, g.ncol, s, e, w) : -1;
                const bool hit = i >= 0;
                if (!__any_sync(FULL, hit)) return;
                const int jj = jb + q;
                if (use_bits) {
                    // both halves of R; t(u, v) and t(u, w) follow from its rows
                    if (hit) {
                        atomicOr(&R[jj * WP + (i >> 5)], 1u << (i & 31));
                        atomicOr(&R[i * WP + (jj >> 5)], 1u << (jj & 31));
                        atomicAdd(&tcnt[pos], 1);
                    }
                    return;
                }
                if (!hit) return;
                atomicAdd(use_hash ? &cnt[jj] : &tcnt[s + jj], 1);
                atomicAdd(use_hash ? &cnt[i] : &tcnt[s + i], 1);
                atomicAdd(&tcnt[pos], 1);
                {
                    // K4 with this triangle (u, v, w): x in N+(w) ∩ N+(u) ∩ N+(v)
                    const int v = g.ncol[s + jj];
                    const int4 rv = g.rinfo[v], rw = g.rinfo[w];
                    const int vs0 = rv.y, ve0 = rv.z;
                    const int ws0 = rw.y, we0 = rw.z;
                    for (int p = ws0; p < we0; ++p) {
                        const int x = g.ncol[p];
                        if (x > umax) break;
                        const int ix = out_index(hk, hv, mask, use_hash, g.ncol, s, e, x);
                        if (ix < 0 || find_sorted(g.ncol, vs0, ve0, x) < 0) continue;
                        ku += 1;
                        if (use_hash) {
                            atomicAdd(&kc[jj], 1);
                            atomicAdd(&kc[i], 1);
                            atomicAdd(&kc[ix], 1);
                        } else {
                            add64(&vacc[v].K4, 1);
                            add64(&vacc[w].K4, 1);
                            add64(&vacc[x].K4, 1);
                        }
                    }
                }
            });
            __syncwarp();
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nloc; i += TC_THREADS)
            if (cnt[i]) atomicAdd(&tcnt[s + i], cnt[i]);
        if (use_bits) {
            // K4s of u: the triangles of R. A warp takes a row y and, one per
            // lane, its neighbours z < y, 32 at a time (collected in zb), and
            // adds the common bits of rows y and z to both. Every triangle is
            // counted by three pairs, and added twice to each of its corners.
            // Whole rows in 16-byte groups: the words below z and above y
            // alone, two thirds of them, which count each triangle where it
            // is needed, took two masked words and loops of different length
            // in every lane (R-MAT 18: k_tri_cta 912 -> 817 us, k_tri_big 545
            // -> 504, both then less by the probes' loads ahead; G(1501, 1/2):
            // 141 -> 121, 1068 -> 1045, where rows are longest; carry-save adders to save population counts: no
            // faster). The loop is bound by shared memory and by latency.
            // The row's popcount is t(u, N+(u)[y]) from the triangles
            // rooted at u.
            for (;;) {
                int y = 0;
                if (lane == 0) y = dp - 1 - atomicAdd(&work[0], 1);   // most neighbours below first
                y = __shfl_sync(FULL, y, 0);
                if (y < 0) break;
                const unsigned *ry = R + y * WP;
                const int wy = y >> 5;
                unsigned acc = 0;
                auto batch = [&](int cnt) {
                    if (lane >= cnt) return;
                    const int z = zb[lane];
                    const unsigned *rz = R + z * WP;
                    unsigned k = 0;
#pragma unroll 1
                    for (int t = 0; t < W; t += 4) {   // (words past W are 0)
                        const uint4 a = *reinterpret_cast<const uint4 *>(ry + t), b = *reinterpret_cast<const uint4 *>(rz + t);
                        k += __popc(a.x & b.x) + __popc(a.y & b.y) + __popc(a.z & b.z) + __popc(a.w & b.w);
                    }
                    if (k) {
                        acc += k;
                        ku += k;
                        atomicAdd(&kc[z], (int)k);
                    }
                };
                int tuy = 0;   // set bits of row y
                for (int t = lane; t < W; t += 32) tuy += __popc(ry[t]);
                tuy = (int)__reduce_add_sync(FULL, (unsigned)tuy);
                if (tuy == 0) continue;
                if (lane == 0) atomicAdd(&tcnt[s + y], tuy);
                int nb = 0;   // entries waiting in zb (warp-uniform)
                for (int t = 0; t <= wy; ++t) {
                    const bool set = ((ry[t] >> lane) & 1u) && t * 32 + lane < y;
                    const unsigned bal = __ballot_sync(FULL, set);
                    if (set) zb[nb + __popc(bal & lanemask_lt())] = (unsigned short)(t * 32 + lane);
                    nb += __popc(bal);
                    __syncwarp();
                    if (nb >= 32) {
                        batch(32);
                        __syncwarp();
                        if (lane < nb - 32) zb[lane] = zb[32 + lane];
                        nb -= 32;
                        __syncwarp();
                    }
                }
                if (nb) batch(nb);
                acc = __reduce_add_sync(FULL, acc);   // at most 1152^2
                if (lane == 0 && acc) atomicAdd(&kc[y], (int)acc);
                __syncwarp();
            }
        }
        __syncthreads();
        ku = warp_sum(ku);
        if (lane == 0 && ku) add64(use_bits ? &s_ku : &vacc[u].K4, ku);
        for (int i = threadIdx.x; i < nloc; i += TC_THREADS)
            if (kc[i]) add64(&vacc[g.ncol[s + i]].K4, use_bits ? kc[i] >> 1 : kc[i]);
        if (use_bits) {
            __syncthreads();
            if (threadIdx.x == 0 && s_ku) {
                add64(&vacc[u].K4, s_ku / 3);
                s_ku = 0;
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(TS_THREADS) k_tri_cta(Graph g, AdjBits A, int *tcnt, VAcc *vacc, const int *heavy,
                                                        int *counters, int bits_maxd, int hash_maxd) {
    pdl_begin();
    if (call_stopped(counters)) return;
    tri_cta<TS_THREADS, TS_MAXD, 4 * TS_MAXD, TS_MAXD, false, 4>(g, A, counters[CNT_ADJ_ON], tcnt, vacc, heavy,
                                                            counters[CNT_TRI_HEAVY], counters + CNT_TRI_CTA_NEXT,
                                                            bits_maxd, hash_maxd);
}

__global__ void __launch_bounds__(TB_THREADS) k_tri_big(Graph g, AdjBits A, int *tcnt, VAcc *vacc, const int *heavy,
                                                        int *counters, int bits_maxd, int hash_maxd) {
    pdl_begin();
    if (call_stopped(counters)) return;
    tri_cta<TB_THREADS, TB_BITMAT_MAXD, TB_BITMAT_HSLOTS, TB_HASH_MAXD, true, 4>(g, A, counters[CNT_ADJ_ON], tcnt, vacc, heavy,
                                                                            counters[CNT_TRI_BIG],
                                                                            counters + CNT_TRI_BIG_NEXT, bits_maxd,
                                                                            hash_maxd);
}


void launch_stage1(Work &w, cudaStream_t st) {
    Graph g{w.n, w.m, w.rinfo, w.ncol};
    const int maxd = w.tune[TUNE_WARP_MAXD] < TW_MAXD ? w.tune[TUNE_WARP_MAXD] : TW_MAXD;
    static const int occ_w = resident_ctas((const void *)k_tri_warp, TW_WARPS * 32, 0);
    static const int occ_c = resident_ctas((const void *)k_tri_cta, TS_THREADS, TS_SMEM);
    static const int occ_b = resident_ctas((const void *)k_tri_big, TB_THREADS, TB_SMEM);
    const AdjBits A = adj_bits(w);
    if (adj_wanted(w.n, w.m)) {
        launch_pdl(k_adj_bits, w.num_sms * 8, 256, 0, st, g, A, w.nrow, const_cast<unsigned *>(A.words),
                   const_cast<unsigned short *>(A.prefix), w.counters);
        after_launch(st, K_ADJ_BITS);
    }
    launch_pdl(k_tri_warp, w.num_sms * min(w.tune[TUNE_GRID_TRI], occ_w), TW_WARPS * 32, 0, st, g, A, w.tcnt, w.vacc, w.lists,
               w.counters, maxd, w.coff, w.ntiles);
    after_launch(st, K_TRI_WARP);
    const int bits = w.tune[TUNE_TRI_BITS_MAXD], hash = w.tune[TUNE_TRI_HASH_MAXD];
    if (out_degree_above(maxd, w.m)) {
        launch_pdl(k_tri_cta, w.num_sms * occ_c, TS_THREADS, TS_SMEM, st, g, A, w.tcnt, w.vacc, w.lists, w.counters, bits, hash);
        after_launch(st, K_TRI_CTA);
    }
    if (out_degree_above(TS_MAXD, w.m)) {
        launch_pdl(k_tri_big, w.num_sms * occ_b, TB_THREADS, TB_SMEM, st, g, A, w.tcnt, w.vacc, w.lists, w.counters, bits, hash);
        after_launch(st, K_TRI_BIG);
    }
}

void configure_stage1() {
    cudaFuncSetAttribute(k_tri_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TS_SMEM);
    cudaFuncSetAttribute(k_tri_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TB_SMEM);
}

}  // namespace niorca
