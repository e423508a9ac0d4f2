// stage2.cu -- edge aggregates and the triangle-opposite term, after the
// per-edge triangle counts t are final.
//
// For every out-edge (u, v) with t = t_uv > 0 (edges without a triangle add
// nothing), both endpoints receive
//   A1 += t, A2 += t^2, A3 += t * d(other end),
// the neighbour sums from which the f* variables of Table 1 that involve
// t_xy follow (f_13^14 = A2 - A1, f_11^13 = (d-1) A1 - A2, ...).
// Every triangle u < v < w is listed again (as in Stage I) and each corner
// receives t of the opposite edge minus one:
//   D12[u] += t_vw - 1, D12[v] += t_uw - 1, D12[w] += t_uv - 1,
// so that D12(x) = sum over triangles {x,y,z} of (t_yz - 1) = f_12^14
// (Table 1: the triangles of e_yz other than xyz). Only out-edges with
// t > 0 are expanded.
#include <type_traits>

#include "kernels.h"

namespace niorca {

constexpr int AW_MAXD = 64;
constexpr int AW_WARPS = 8;
constexpr int AS_MAXD = 256;   // out-degree handled by a 256-thread CTA (k_agg_cta)

struct __align__(16) AggWarpSmem {
    Filter filter;
    long long dc[AW_MAXD];   // D12 sums of N+(u)
};

// Edge aggregates of u's out-edges; returns the warp's sum of t (0: none has a
// triangle).
__device__ __forceinline__ long long edge_aggregates(const Graph &g, const int *tcnt, VAcc *vacc, int u, int s, int dp,
                                                int first, int stride) {
    const int4 ru = g.rinfo[u];
    const int du = ru.z - ru.x;
    long long a1 = 0, a2 = 0, a3 = 0;
    for (int j = first; j < dp; j += stride) {
        const long long t = tcnt[s + j];
        if (!t) continue;
        const int v = g.ncol[s + j];
        const int4 rv = g.rinfo[v];
        const long long dv = rv.z - rv.x;
        a1 += t;
        a2 += t * t;
        a3 += t * dv;
        add64(&vacc[v].A1, t);
        add64(&vacc[v].A2, t * t);
        add64(&vacc[v].A3, t * du);
    }
    a1 = warp_sum(a1);
    a2 = warp_sum(a2);
    a3 = warp_sum(a3);
    if (lane_id() == 0 && a1) {
        add64(&vacc[u].A1, a1);
        add64(&vacc[u].A2, a2);
        add64(&vacc[u].A3, a3);
    }
    return a1;
}

// One warp-tier root over the adjacency bitmap: the pairs of u's
// out-neighbours whose edges to u close triangles are probed, as in Stage I.
// A column's sum of t(u, row) - 1 and a row's sum of t(u, column) - 1 stay in
// its lane.
__device__ __forceinline__ void agg_root_probe(const Graph &g, const AdjBits &A, const int *tcnt, VAcc *vacc, int u, int s,
                                               int dp) {
    const int lane = lane_id();
    const OutList L = out_list(g, A, s, dp);
    const int t0 = lane < dp ? tcnt[s + lane] : 0, t1 = 32 + lane < dp ? tcnt[s + 32 + lane] : 0;
    long long du12 = 0, d0 = 0, d1 = 0;   // D12 of u, of entries lane and 32 + lane
    out_pairs(g, A, L, __ballot_sync(FULL, t0 > 0), __ballot_sync(FULL, t1 > 0), t0 > 0, t1 > 0,
              [&](int b, int r, bool hit, int pos) {
                  const int tr = __shfl_sync(FULL, b == 2 ? t1 : t0, r);   // t(u, row)
                  const int tc = b == 0 ? t0 : t1;                         // t(u, column)
                  // (32 counts of at most 2^20 fit 32 bits)
                  const int sum = (int)__reduce_add_sync(FULL, (unsigned)(hit ? tc - 1 : 0));
                  if (hit) {
                      du12 += tcnt[pos] - 1;
                      if (b == 0) d0 += tr - 1; else d1 += tr - 1;
                  }
                  if (lane == r) {
                      if (b == 2) d1 += sum; else d0 += sum;
                  }
              });
    du12 = warp_sum(du12);
    if (lane == 0 && du12) add64(&vacc[u].D12, du12);
    if (d0) add64(&vacc[L.w0].D12, d0);
    if (d1) add64(&vacc[L.w1].D12, d1);
}

// One warp-tier root whose out-neighbours' rows are streamed past a filter of
// N+(u), as in Stage I; only rows of edges with triangles.
__device__ __forceinline__ void agg_root_stream(const Graph &g, const int *tcnt, VAcc *vacc, int u, int s, int dp,
                                                AggWarpSmem &S) {
    const int lane = lane_id();
    int w0 = -1, w1 = -1;
    bool in0 = false, in1 = false;   // entries with t(u, .) > 0
    int2 r0 = make_int2(0, 0), r1 = r0;
    auto fill = [&](int i, int &w, bool &in, int2 &r) {
        if (i >= dp) return;
        w = g.ncol[s + i];
        in = tcnt[s + i] > 0;
        if (!in || i == dp - 1) return;
        const int4 rw = g.rinfo[w];
        r = make_int2(rw.y, rw.z);
    };
    fill(lane, w0, in0, r0);
    if (dp > 32) fill(32 + lane, w1, in1, r1);
    S.filter.set(w0, w1, in0, in1);
    S.dc[lane] = S.dc[32 + lane] = 0;
    __syncwarp();
    long long du12 = 0;
    filter_walk_some(g.ncol, S.filter, r0, r1, [&](int j, int pos, int w) {
        const int i = S.filter.find(w, dp);
        if (i < 0) return;
        add64(&S.dc[j], tcnt[s + i] - 1);   // t(u, w) - 1 -> v
        du12 += tcnt[pos] - 1;              // t(v, w) - 1 -> u
        add64(&S.dc[i], tcnt[s + j] - 1);   // t(u, v) - 1 -> w
    });
    du12 = warp_sum(du12);
    if (lane == 0 && du12) add64(&vacc[u].D12, du12);
    __syncwarp();
    for (int i = lane; i < dp; i += 32)
        if (S.dc[i]) add64(&vacc[g.ncol[s + i]].D12, S.dc[i]);
}

__global__ void __launch_bounds__(AW_WARPS * 32, 6) k_agg_warp(Graph g, AdjBits A, const int *tcnt, VAcc *vacc, int *heavy,
                                                            int *counters, int maxd, const int *coff, int ntiles) {
    pdl_begin();
    __shared__ AggWarpSmem sm_all[AW_WARPS];
    AggWarpSmem &S = sm_all[threadIdx.x >> 5];
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    if (call_stopped(counters)) return;
    const bool probe = counters[CNT_ADJ_ON];
    auto triangles = [&](int u, int s, int dp) {
        if (probe) agg_root_probe(g, A, tcnt, vacc, u, s, dp);
        else agg_root_stream(g, tcnt, vacc, u, s, dp, S);
        __syncwarp();
    };
    auto root = [&](int u, int s, int dp) {
        if (dp < 1) return;
        if (dp > maxd) {
            if (lane == 0) {
                if (dp <= AS_MAXD) heavy[atomicAdd(&counters[CNT_AGG_HEAVY], 1)] = u;
                else heavy[g.n - 1 - atomicAdd(&counters[CNT_AGG_BIG], 1)] = u;
            }
            return;
        }
        if (edge_aggregates(g, tcnt, vacc, u, s, dp, lane, 32) != 0 && dp >= 2) triangles(u, s, dp);
    };
    // ids of low degree: four roots at a time, eight lanes each
    const int low = low_degree_ids(g.n, nw, coff, ntiles);
    for (long long u0 = 4ll * gw; u0 < low; u0 += 4ll * nw) {
        const int u = (int)u0 + (lane >> 3);
        int4 ru = make_int4(0, 0, 0, 0);
        if (u < low) ru = g.rinfo[u];
        const int dp = ru.z - ru.y;
        if (!__any_sync(FULL, dp > min(SMALL_DP, maxd))) {
            // edge aggregates of the four roots' out-edges
            const int l = lane & 7;
            const long long t = l < dp ? tcnt[ru.y + l] : 0;
            if (!__any_sync(FULL, t != 0)) continue;
            int w = -1;
            int2 r = make_int2(0, 0);
            long long a1 = t, a2 = t * t, a3 = 0;
            if (t) {
                w = g.ncol[ru.y + l];
                const int4 rw = g.rinfo[w];
                a3 = t * (rw.z - rw.x);
                add64(&vacc[w].A1, t);
                add64(&vacc[w].A2, t * t);
                add64(&vacc[w].A3, t * (ru.z - ru.x));
                if (l < dp - 1) r = make_int2(rw.y, rw.z);
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                a1 += __shfl_xor_sync(FULL, a1, o);
                a2 += __shfl_xor_sync(FULL, a2, o);
                a3 += __shfl_xor_sync(FULL, a3, o);
            }
            if (l == 0 && a1) {
                add64(&vacc[u].A1, a1);
                add64(&vacc[u].A2, a2);
                add64(&vacc[u].A3, a3);
            }
            if (!__any_sync(FULL, r.y - r.x > SMALL_ROW)) {
                long long du12 = 0, dv = 0;
                small_walk(g.ncol, w, r, [&](int pos, int x) {
                    for (int i = l + 1; i < dp; ++i)
                        if (g.ncol[ru.y + i] == x) {
                            dv += tcnt[ru.y + i] - 1;               // t(u, w) - 1 -> v
                            du12 += tcnt[pos] - 1;                  // t(v, w) - 1 -> u
                            if (t > 1) add64(&vacc[x].D12, t - 1);  // t(u, v) - 1 -> w
                        }
                });
                if (dv) add64(&vacc[w].D12, dv);
                if (du12) add64(&vacc[u].D12, du12);
                continue;
            }
            for (int q = 0; q < 4; ++q) {
                const int s = __shfl_sync(FULL, ru.y, 8 * q), d = __shfl_sync(FULL, dp, 8 * q);
                if (d >= 2 && __shfl_sync(FULL, (int)(a1 != 0), 8 * q)) triangles((int)u0 + q, s, d);
            }
            continue;
        }
        for (int q = 0; q < 4; ++q) root((int)u0 + q, __shfl_sync(FULL, ru.y, 8 * q), __shfl_sync(FULL, dp, 8 * q));
    }
    for (int u = low + gw; u < g.n; u += nw) {
        const int4 ru = g.rinfo[u];
        root(u, ru.y, ru.z - ru.y);
    }
}

// Roots above the warp tier: k_agg_cta (256 threads, dp <= AS_MAXD, several
// CTAs per SM) and k_agg_big (1024 threads), from the front and the back of
// the heavy list. Out-neighbours with a bitmap row are probed in blocks of 32
// rows x 32 columns, a warp each: a column's and a row's sums stay in its
// lane until the block ends. The rows of the others are streamed against a
// hash of N+(u) up to AB_HASH_MAXD with a credit per triangle in shared
// memory; above that, binary searches and credits in global memory.
//
// In a call without a bitmap a root whose out-edges have AGG_BITS_T triangles
// each on average keeps its triangles as the symmetric bit matrix R of N+(u)
// (as in Stage I) up to AB_BITMAT_MAXD, and each y of N+(u) then receives the
// sum over its neighbours z in R of t(u, z) - 1: two 64-bit shared atomics per
// triangle, most lanes of a window to one word, cost more than two bits and a
// pass over R where triangles are many (k_agg_cta: 2000 cliques of 150 in one
// graph 22.5 -> 7.6 ms, a batch of 100 graphs G(400, 1/2) 3358 -> 1588 us; with
// R for every root 952 us on G(50000, mean degree 200), where an edge is in
// 0.8 triangles, 776 with the line).
constexpr int AS_THREADS = 256;
constexpr int AB_THREADS = 1024;
constexpr int AB_BITMAT_MAXD = 1152;
constexpr int AB_BITMAT_HSLOTS = 4096;
constexpr int AB_HASH_MAXD = 8192;
constexpr int AGG_BITS_T = 16;
__host__ __device__ constexpr int ac_rowstride(int rows) { return ((rows + 31) / 32) | 1; }   // odd: spreads the banks
// D12 sums (nloc x 8 B), hash (2 x hslots ints), a segment table per warp and
// R. (What is left of an SM's shared memory caches the gathers of t.)
constexpr size_t ac_smem(int threads, int hslots, int nloc, int rows) {
    return (size_t)nloc * 8 + (size_t)2 * hslots * 4 + (size_t)(threads / 32) * sizeof(SegTab) +
           (size_t)rows * 4 * ac_rowstride(rows);
}
constexpr size_t max_size(size_t a, size_t b) { return a > b ? a : b; }
constexpr size_t AS_SMEM = max_size(ac_smem(AS_THREADS, 4 * AS_MAXD, 0, AS_MAXD), ac_smem(AS_THREADS, 4 * AS_MAXD, AS_MAXD, 0));
constexpr size_t AB_SMEM = max_size(ac_smem(AB_THREADS, AB_BITMAT_HSLOTS, 0, AB_BITMAT_MAXD),
                                    ac_smem(AB_THREADS, 2 * AB_HASH_MAXD, AB_HASH_MAXD, 0));
static_assert(AB_SMEM <= 227 * 1024, "k_agg_big shared memory");

// (PROBE, the call has a bitmap, or not: two bodies, each with the registers
// its own loops need.)
template <bool PROBE, int THREADS, int BITMAT_MAXD, int BITMAT_HSLOTS, int HASH_MAXD, int HSLOTS, bool BACK>
__device__ __forceinline__ void agg_cta(const Graph &g, const AdjBits &A, const int *tcnt, VAcc *vacc,
                                        const int *heavy, int nh, int *next, int bits_maxd, int hash_maxd) {
    extern __shared__ __align__(16) unsigned char dsm[];
    constexpr int NW = THREADS / 32;
    __shared__ long long sum_t;   // of t(u, .)
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    for (int h = cta_next(next); h < nh; h = cta_next(next)) {
        const int u = BACK ? heavy[g.n - 1 - h] : heavy[h];
        const int4 ru = g.rinfo[u];
        const int s = ru.y, e = ru.z, dp = e - s;
        if (threadIdx.x == 0) sum_t = 0;
        __syncthreads();
        const long long tw = edge_aggregates(g, tcnt, vacc, u, s, dp, threadIdx.x, THREADS);
        if (tw && lane == 0) add64(&sum_t, tw);
        __syncthreads();
        if (!sum_t) continue;
        const bool use_hash = dp <= HASH_MAXD && dp <= hash_maxd;
        // rows js .. of N+(u) are probed in the bitmap, the ones before streamed
        const int js = PROBE && use_hash ? lower_bound(g.ncol, s, e, A.base) - s : dp;
        const bool use_bits =
            !PROBE && use_hash && dp <= BITMAT_MAXD && dp <= bits_maxd && sum_t >= (long long)AGG_BITS_T * dp;
        unsigned H = use_hash && js > 0 ? next_pow2(4 * dp) : 0;   // hash load at most 1/4, within the carve
        const unsigned hcap = use_bits ? BITMAT_HSLOTS : HSLOTS;
        if (H > hcap) H = hcap;
        const unsigned mask = H ? H - 1 : 0;
        const int W = (dp + 31) >> 5;
        const int WP = ac_rowstride(dp);   // row stride of R
        const int nloc = use_hash && !use_bits ? dp : 0;
        long long *dc = reinterpret_cast<long long *>(dsm);   // D12 sums of N+(u)
        int *hk = reinterpret_cast<int *>(dc + ((nloc + 1) & ~1));   // 16-byte aligned buckets
        int *hv = hk + H;
        SegTab *segs = reinterpret_cast<SegTab *>(hv + H);   // one per warp
        SegTab &seg = segs[wid];
        unsigned *R = reinterpret_cast<unsigned *>(segs + NW);
        for (int i = threadIdx.x; i < (int)H; i += THREADS) hk[i] = -1;
        for (int i = threadIdx.x; i < nloc; i += THREADS) dc[i] = 0;
        if (use_bits)
            for (int i = threadIdx.x; i < dp * WP; i += THREADS) R[i] = 0;
        __syncthreads();
        if (H)
            for (int i = threadIdx.x; i < dp; i += THREADS) hset_insert(hk, hv, mask, g.ncol[s + i], i);
        const int umax = g.ncol[e - 1];
        long long du12 = 0;
        if (PROBE && js < dp) {
            const int b0 = js >> 5;   // the first block of rows
            for (int it = b0 * (b0 + 1) / 2 + wid; it < W * (W + 1) / 2; it += NW) {
                int t, jb;
                block_pair(it, t, jb);
                if (jb < b0) continue;
                const int i = 32 * t + lane, j = 32 * jb + lane;
                const int tc = i < dp ? tcnt[s + i] : 0, tr = j >= js && j < dp - 1 ? tcnt[s + j] : 0;   // t(u, .)
                const int k = i < dp ? g.n - 1 - g.ncol[s + i] : 0;
                int roff = 0, ry = 0;
                if (tr > 0) {
                    const int v = g.ncol[s + j];
                    roff = A.row(v);
                    ry = g.rinfo[v].y;
                }
                unsigned rsum = 0, csum = 0;   // 32 counts of at most 2^20 each
                adj_probe<4, true>(A, __ballot_sync(FULL, tr > 0), roff, ry, k, tc > 0, t == jb, tcnt,
                                   [&](int r, bool hit, int, int tvw) {
                                       const int tw = __shfl_sync(FULL, tr, r);
                                       const unsigned sum = __reduce_add_sync(FULL, (unsigned)(hit ? tc - 1 : 0));
                                       if (lane == r) rsum = sum;
                                       if (hit) {
                                           csum += tw - 1;      // t(u, v) - 1 -> w
                                           du12 += tvw - 1;     // t(v, w) - 1 -> u
                                       }
                                   });
                if (rsum) add64(&dc[j], rsum);   // t(u, w) - 1 -> v
                if (csum) add64(&dc[i], csum);
            }
        }
        __syncthreads();
        const int jend = min(js, dp - 1);
        auto stream = [&](auto hit) {   // hit(j, i, pos, w): N+(u)[i] = w is at pos of the row of N+(u)[j]
            for (int jb = 0; jb < jend; jb += 32) {   // all warps share each chunk
                const int j = jb + lane;
                int len = 0, vs = 0;
                if (j < jend && tcnt[s + j] > 0) {
                    const int4 rv = g.rinfo[g.ncol[s + j]];
                    vs = rv.y;
                    len = rv.z - rv.y;
                }
                int mypre;
                const int total = seg_build(seg, vs, len, mypre);
                seg_visit<4, true>(g.ncol, seg, mypre, len, total, wid * 32, NW * 32, [&](bool valid, int q, int pos, int w) {
                    int i = -1;
                    if (valid && w <= umax) {
                        if (use_hash) {
                            i = hset_find(hk, hv, mask, w);
                        } else {
                            const int p = find_sorted(g.ncol, s, e, w);
                            i = p < 0 ? -1 : p - s;
                        }
                    }
                    if (i >= 0) hit(jb + q, i, pos, w);
                });
                __syncwarp();
            }
        };
        if (use_bits) {
            stream([&](int j, int i, int pos, int) {
                du12 += tcnt[pos] - 1;   // t(v, w) - 1 -> u
                atomicOr(&R[j * WP + (i >> 5)], 1u << (i & 31));
                atomicOr(&R[i * WP + (j >> 5)], 1u << (j & 31));
            });
        } else {
            stream([&](int j, int i, int pos, int w) {
                du12 += tcnt[pos] - 1;                                                     // t(v, w) - 1 -> u
                const long long tv = tcnt[s + i] - 1, tw = tcnt[s + j] - 1;
                add64(use_hash ? &dc[j] : &vacc[g.ncol[s + j]].D12, tv);                   // t(u, w) - 1 -> v
                add64(use_hash ? &dc[i] : &vacc[w].D12, tw);                               // t(u, v) - 1 -> w
            });
        }
        du12 = warp_sum(du12);
        if (lane == 0 && du12) add64(&vacc[u].D12, du12);
        __syncthreads();
        if (use_bits)
            for (int y = wid; y < dp; y += NW) {
                const unsigned *ry = R + y * WP;
                unsigned c = 0;   // 1152 counts of at most 2^20 fit 32 bits
                for (int t = 0; t < W; ++t)
                    if ((ry[t] >> lane) & 1u) c += tcnt[s + 32 * t + lane] - 1;
                c = __reduce_add_sync(FULL, c);
                if (lane == 0 && c) add64(&vacc[g.ncol[s + y]].D12, c);
            }
        for (int i = threadIdx.x; i < nloc; i += THREADS)
            if (dc[i]) add64(&vacc[g.ncol[s + i]].D12, dc[i]);
        __syncthreads();
    }
}

__global__ void __launch_bounds__(AS_THREADS, 6) k_agg_cta(Graph g, AdjBits A, const int *tcnt, VAcc *vacc, const int *heavy,
                                                        int *counters, int bits_maxd, int hash_maxd) {
    pdl_begin();
    if (call_stopped(counters)) return;
    auto run = [&](auto probe) {
        agg_cta<decltype(probe)::value, AS_THREADS, AS_MAXD, 4 * AS_MAXD, AS_MAXD, 4 * AS_MAXD, false>(
            g, A, tcnt, vacc, heavy, counters[CNT_AGG_HEAVY], counters + CNT_AGG_CTA_NEXT, bits_maxd, hash_maxd);
    };
    if (counters[CNT_ADJ_ON]) run(std::true_type{});
    else run(std::false_type{});
}

__global__ void __launch_bounds__(AB_THREADS) k_agg_big(Graph g, AdjBits A, const int *tcnt, VAcc *vacc, const int *heavy,
                                                        int *counters, int bits_maxd, int hash_maxd) {
    pdl_begin();
    if (call_stopped(counters)) return;
    auto run = [&](auto probe) {
        agg_cta<decltype(probe)::value, AB_THREADS, AB_BITMAT_MAXD, AB_BITMAT_HSLOTS, AB_HASH_MAXD, 2 * AB_HASH_MAXD, true>(
            g, A, tcnt, vacc, heavy, counters[CNT_AGG_BIG], counters + CNT_AGG_BIG_NEXT, bits_maxd, hash_maxd);
    };
    if (counters[CNT_ADJ_ON]) run(std::true_type{});
    else run(std::false_type{});
}

void launch_stage2(Work &w, cudaStream_t st) {
    Graph g{w.n, w.m, w.rinfo, w.ncol};
    int *heavy = w.lists + (size_t)w.n;
    const int maxd = w.tune[TUNE_WARP_MAXD] < AW_MAXD ? w.tune[TUNE_WARP_MAXD] : AW_MAXD;
    static const int occ_w = resident_ctas((const void *)k_agg_warp, AW_WARPS * 32, 0);
    static const int occ_c = resident_ctas((const void *)k_agg_cta, AS_THREADS, AS_SMEM);
    static const int occ_b = resident_ctas((const void *)k_agg_big, AB_THREADS, AB_SMEM);
    const AdjBits A = adj_bits(w);
    launch_pdl(k_agg_warp, w.num_sms * min(w.tune[TUNE_GRID_AGG], occ_w), AW_WARPS * 32, 0, st, g, A, w.tcnt, w.vacc, heavy,
               w.counters, maxd, w.coff, w.ntiles);
    after_launch(st, K_AGG_WARP);
    const int bits = w.tune[TUNE_TRI_BITS_MAXD], hash = w.tune[TUNE_TRI_HASH_MAXD];
    if (out_degree_above(maxd, w.m)) {
        launch_pdl(k_agg_cta, w.num_sms * occ_c, AS_THREADS, AS_SMEM, st, g, A, w.tcnt, w.vacc, heavy, w.counters, bits, hash);
        after_launch(st, K_AGG_CTA);
    }
    if (out_degree_above(AS_MAXD, w.m)) {
        launch_pdl(k_agg_big, w.num_sms * occ_b, AB_THREADS, AB_SMEM, st, g, A, w.tcnt, w.vacc, heavy, w.counters, bits, hash);
        after_launch(st, K_AGG_BIG);
    }
}

void configure_stage2() {
    cudaFuncSetAttribute(k_agg_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AS_SMEM);
    cudaFuncSetAttribute(k_agg_big, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AB_SMEM);
}

}  // namespace niorca
