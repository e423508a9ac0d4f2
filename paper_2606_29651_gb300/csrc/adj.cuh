// adj.cuh -- the adjacency bitmap of the hubs, probed by the triangle and
// aggregate stages (built by k_adj_bits in stage1.cu).
#pragma once
#include "common.cuh"

namespace niorca {

// Adjacency bitmap of the `rows` highest ids (the hubs, which most
// out-entries of a skewed graph point at). Row v (v >= base) holds N+(v): bit
// k & 31 of word k >> 5 stands for id n - 1 - k, so that a row ends with the
// word of its own id and the rows form a triangle; prefix holds, per word,
// how many entries of N+(v) have ids below the word's. Testing whether (v, w)
// is an edge is one word, and its position in N+(v) one prefix and a
// popcount, where a walk of N+(v) (mean length 360-540 on R-MAT 22, whatever
// the length of N+(u)) would stream the whole row.
struct AdjBits {
    const unsigned *words;
    const unsigned short *prefix;
    int n, base;
    // first word of the row of the id with r ids above it: the sum of i / 32 + 1 over i < r
    __host__ __device__ static __forceinline__ long long row_words(long long r) {
        const long long q = r >> 5;
        return r + 16 * q * (q - 1) + q * (r & 31);
    }
    __device__ __forceinline__ int row(int v) const { return (int)row_words(n - 1 - v); }
};

// Probes up to 32 rows of the bitmap (bit r of `rows`: lane r holds the row's
// first word in `roff` and its first position in `ry`) for the lane's id
// n - 1 - k (where `ok`; with `diag` only in rows r below the lane), U rows in
// flight. f(r, hit, pos, val) on every lane, per row with a hit: the entry's
// position and, with LOAD, tcnt[pos]. The prefix of a word is loaded with the
// word, hit or not, and the values of all U rows before the first is used:
// loaded at each row's hits, they were waited for one after the other (R-MAT
// 22: k_tri_big 31.8 -> 27.5 ms, k_tri_cta 16.9 -> 14.4, k_agg_big 22.2 ->
// 14.1, k_agg_cta 15.3 -> 11.5; G(1501, 1/2): 1077 -> 905 us, 120 -> 117, 627
// -> 376, 81 -> 76; R-MAT 14, warp tiers: 41 -> 35 us, 63 -> 60). U is what
// the registers of each kernel allow without losing a CTA per SM.
template <int U, bool LOAD, class F>
__device__ __forceinline__ void adj_probe(const AdjBits &A, unsigned rows, int roff, int ry, int k, bool ok, bool diag,
                                          const int *tcnt, F f) {
    const int lane = lane_id(), kw = k >> 5;
    while (rows) {
        int r[U], pos[U], val[U];
        unsigned w[U];
#pragma unroll
        for (int h = 0; h < U; ++h) {
            r[h] = rows ? __ffs(rows) - 1 : 32;
            rows &= rows - 1;
            const int at = __shfl_sync(FULL, roff, r[h] & 31) + kw;
            w[h] = 0;
            pos[h] = 0;
            if (ok && (diag ? r[h] < lane : r[h] < 32)) {
                w[h] = __ldg(A.words + at);
                pos[h] = __ldg(A.prefix + at);
            }
        }
#pragma unroll
        for (int h = 0; h < U; ++h) {
            pos[h] += __shfl_sync(FULL, ry, r[h] & 31) + __popc((w[h] >> (k & 31)) >> 1);
            w[h] = (w[h] >> (k & 31)) & 1u;
            val[h] = 0;
            if (LOAD && w[h]) val[h] = tcnt[pos[h]];
        }
#pragma unroll
        for (int h = 0; h < U; ++h)
            if (__any_sync(FULL, w[h])) f(r[h], w[h] != 0, pos[h], val[h]);
    }
}

// Block `it` of the upper triangle of 32 x 32 blocks: column block t, row
// block jb <= t, numbered column by column.
__device__ __forceinline__ void block_pair(int it, int &t, int &jb) {
    t = (int)((sqrtf(8.0f * it + 1.0f) - 1.0f) * 0.5f);
    if ((t + 1) * (t + 2) / 2 <= it) ++t;
    if (t * (t + 1) / 2 > it) --t;
    jb = it - t * (t + 1) / 2;
}

// The out-list of a warp-tier root (dp <= 64) spread over the lanes: entries
// lane and 32 + lane.
struct OutList {
    int w0, w1;              // ids (-1: none)
    int k0, k1;              // n - 1 - id
    int a0, a1;              // first word of the bitmap row
    int2 r0, r1;             // N+ of the entry: [x, y)
    unsigned in0, in1;       // entries with a bitmap row, entries without
    unsigned out0, out1;
};

__device__ __forceinline__ OutList out_list(const Graph &g, const AdjBits &A, int s, int dp) {
    const int lane = lane_id();
    OutList L;
    auto fill = [&](int i, int &w, int &k, int &a, int2 &r, unsigned &in, unsigned &out) {
        w = i < dp ? g.ncol[s + i] : -1;
        k = g.n - 1 - w;
        a = 0;
        r = make_int2(0, 0);
        if (i < dp - 1) {   // the last entry has no row to probe
            const int4 rw = g.rinfo[w];
            r = make_int2(rw.y, rw.z);
            if (w >= A.base) a = A.row(w);
        }
        in = __ballot_sync(FULL, i < dp - 1 && w >= A.base);
        out = __ballot_sync(FULL, i < dp - 1 && w < A.base);
    };
    fill(lane, L.w0, L.k0, L.a0, L.r0, L.in0, L.out0);
    L.w1 = -1, L.k1 = 0, L.a1 = 0, L.r1 = make_int2(0, 0), L.in1 = L.out1 = 0;
    if (dp > 32) fill(32 + lane, L.w1, L.k1, L.a1, L.r1, L.in1, L.out1);
    return L;
}

// Every pair (j, i) of the out-list with N+(u)[i] in N+(N+(u)[j]), i > j:
// f(block, r, hit, pos) on every lane per row with a hit, where block 0 is
// rows and columns below 32, 1 rows below 32 with columns above, 2 both
// above; lane = column, r = row in its half; pos = the entry's position. Rows
// of the bitmap are probed; others are searched (their vertices have lower
// degree, so their rows are short). rows0 / rows1 and ok0 / ok1 select rows
// and columns.
template <class F>
__device__ __forceinline__ void out_pairs(const Graph &g, const AdjBits &A, const OutList &L, unsigned rows0,
                                          unsigned rows1, bool ok0, bool ok1, F f) {
    const int lane = lane_id();
    auto block = [&](int b, unsigned in, unsigned out, int a, int2 r, int w, int k, bool ok, bool diag) {
        adj_probe<2, false>(A, in, a, r.x, k, ok, diag, nullptr,
                            [&](int row, bool hit, int pos, int) { f(b, row, hit, hit ? pos : 0); });
        for (; out; out &= out - 1) {
            const int row = __ffs(out) - 1;
            const int x = __shfl_sync(FULL, r.x, row), z = __shfl_sync(FULL, r.y, row);
            const int p = ok && (!diag || lane > row) ? find_sorted(g.ncol, x, z, w) : -1;
            if (__any_sync(FULL, p >= 0)) f(b, row, p >= 0, p);
        }
    };
    block(0, L.in0 & rows0, L.out0 & rows0, L.a0, L.r0, L.w0, L.k0, ok0, true);
    if (__any_sync(FULL, ok1)) {
        block(1, L.in0 & rows0, L.out0 & rows0, L.a0, L.r0, L.w1, L.k1, ok1, false);
        block(2, L.in1 & rows1, L.out1 & rows1, L.a1, L.r1, L.w1, L.k1, ok1, true);
    }
}

// ------------------------------------------------ graphs without a bitmap
//
// There rows are about as long as out-lists, and a triangle is rare: a root's
// out-neighbours' rows are streamed past a bit filter of N+(u), and only an
// entry that passes is searched in N+(u). Measured against a hash set of N+(u)
// with 16-byte buckets (G(1e6, mean degree 32), k_tri_warp): see there.
constexpr int FILTER_WORDS = 128;   // 4096 bits: at most 64 set
constexpr int SMALL_DP = 8;         // roots of at most this out-degree go four to a warp ...
constexpr int SMALL_ROW = 32;       // ... when no out-neighbour's row is longer than this

// Ids below this one go four to a warp: degrees below 16 (most of them small
// roots; higher ones take a warp each from the start, so that four long roots
// in a row never share one), in graphs with more than four vertices per warp
// of the grid (in a smaller one a warp with four roots in turn is the
// kernel's tail: G(2000, 0.01) 10 -> 22 us).
__device__ __forceinline__ int low_degree_ids(int n, int warps, const int *coff, int ntiles) {
    return n > 4ll * warps ? min(coff[deg_class(16) * ntiles], n) : 0;
}

// A warp's filter of an out-list of at most 64 ids, and the list itself.
struct Filter {
    unsigned bits[FILTER_WORDS];
    int ids[64];
    int2 rows[32];   // filter_walk_some: first position, length | index << 24 of the rows to walk
    // fills it with entries lane and 32 + lane (ids w0, w1; in0, in1: pass the filter)
    __device__ __forceinline__ void set(int w0, int w1, bool in0, bool in1) {
        const int lane = lane_id();
        reinterpret_cast<uint4 *>(bits)[lane] = make_uint4(0, 0, 0, 0);
        ids[lane] = w0;
        ids[32 + lane] = w1;
        __syncwarp();
        if (in0) atomicOr(&bits[(w0 >> 5) & (FILTER_WORDS - 1)], 1u << (w0 & 31));
        if (in1) atomicOr(&bits[(w1 >> 5) & (FILTER_WORDS - 1)], 1u << (w1 & 31));
        __syncwarp();
    }
    __device__ __forceinline__ bool pass(int w) const {
        return (bits[(w >> 5) & (FILTER_WORDS - 1)] >> (w & 31)) & 1u;
    }
    // index of w among the first dp ids (ascending), or -1
    __device__ __forceinline__ int find(int w, int dp) const {
        int lo = 0;
#pragma unroll
        for (int step = 32; step > 0; step >>= 1)
            if (lo + step < dp && ids[lo + step] <= w) lo += step;
        return ids[lo] == w ? lo : -1;
    }
};

// Streams two rows, entries [xa, xa + na) and [xc, xc + nc), of each group of
// eight lanes past the filter, 16 entries of each in flight: f(second, pos,
// w) on the lanes whose entry passes.
template <class F>
__device__ __forceinline__ void filter_rows(const int *__restrict__ col, const Filter &S, int xa, int na, int xc, int nc, F f) {
    const int sub = lane_id() & 7;
    const int longest = (int)__reduce_max_sync(FULL, (unsigned)max(na, nc));
    for (int o = sub; o - sub < longest; o += 16) {
        int w[4];
        w[0] = o < na ? __ldg(col + xa + o) : -1;
        w[1] = o + 8 < na ? __ldg(col + xa + o + 8) : -1;
        w[2] = o < nc ? __ldg(col + xc + o) : -1;
        w[3] = o + 8 < nc ? __ldg(col + xc + o + 8) : -1;
#pragma unroll
        for (int h = 0; h < 4; ++h)
            if (w[h] >= 0 && S.pass(w[h])) f((h & 2) != 0, (h & 2 ? xc : xa) + o + (h & 1 ? 8 : 0), w[h]);
    }
    __syncwarp();
}

// Streams the rows of the warp's out-list (lane: rows r0 = [x, y) of entry
// lane and r1 of entry 32 + lane; the list has dp entries, the last one's row
// is empty) past the filter, eight rows at a time: f(j, pos, w) on the lanes
// whose entry w at pos of row j passes.
template <class F>
__device__ __forceinline__ void filter_walk(const int *__restrict__ col, const Filter &S, int2 r0, int2 r1, int dp, F f) {
    const int q = lane_id() >> 3;
    for (int jb = 0; jb < dp - 1; jb += 8) {
        const int2 r = jb < 32 ? r0 : r1;
        const int ja = (jb + q) & 31, jc = (jb + 4 + q) & 31;
        const int xa = __shfl_sync(FULL, r.x, ja), na = __shfl_sync(FULL, r.y, ja) - xa;
        const int xc = __shfl_sync(FULL, r.x, jc), nc = __shfl_sync(FULL, r.y, jc) - xc;
        filter_rows(col, S, xa, na, xc, nc, [&](bool second, int pos, int w) { f(jb + q + (second ? 4 : 0), pos, w); });
    }
}

// The same for lists with few rows to walk: the empty ones are squeezed out.
template <class F>
__device__ __forceinline__ void filter_walk_some(const int *__restrict__ col, Filter &S, int2 r0, int2 r1, F f) {
    const int lane = lane_id(), q = lane >> 3;
    for (int half = 0; half < 2; ++half) {
        const int2 r = half ? r1 : r0;
        const unsigned some = __ballot_sync(FULL, r.y > r.x);   // a row has at most 2^20 entries
        if (r.y > r.x) S.rows[__popc(some & lanemask_lt())] = make_int2(r.x, (r.y - r.x) | (32 * half + lane) << 24);
        __syncwarp();
        const int cnt = __popc(some);
        for (int k = 0; k < cnt; k += 8) {
            const int2 a = k + q < cnt ? S.rows[k + q] : make_int2(0, 0);
            const int2 c = k + 4 + q < cnt ? S.rows[k + 4 + q] : make_int2(0, 0);
            filter_rows(col, S, a.x, a.y & 0xffffff, c.x, c.y & 0xffffff,
                        [&](bool second, int pos, int w) { f((second ? c.y : a.y) >> 24, pos, w); });
        }
        __syncwarp();
    }
}

// The small roots of a warp: lane 8 q + l holds entry l of root q's out-list
// (w, -1: none) and streams the entry's row r by itself past a 64-bit filter
// of the root's list: f(pos, w) on the lanes whose entry passes.
template <class F>
__device__ __forceinline__ void small_walk(const int *__restrict__ col, int w, int2 r, F f) {
    unsigned lo = w >= 0 && !(w & 32) ? 1u << (w & 31) : 0u, hi = w >= 0 && (w & 32) ? 1u << (w & 31) : 0u;
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        lo |= __shfl_xor_sync(FULL, lo, o);
        hi |= __shfl_xor_sync(FULL, hi, o);
    }
    for (int p = r.x; p < r.y; ++p) {
        const int x = __ldg(col + p);
        if (((x & 32 ? hi : lo) >> (x & 31)) & 1u) f(p, x);
    }
    __syncwarp();
}

}  // namespace niorca
