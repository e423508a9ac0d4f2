// cycle4.cu -- 4-cycles through every vertex (psi_8).
//
// The paper obtains psi_8 from Stage III's `common[z]` array: for a fixed x,
// common[z] counts the 2-paths x-y-z, and f_8^12 sums common[z] - 1 over the
// paths (Table 1, Fig. 3d; Appendix, o8). Per vertex this equals
// psi_8(x) = sum over w != x of C(c_xw, 2), c_xw = |N(x) ∩ N(w)|.
// Here every 4-cycle is built once, from its highest vertex u (in the
// degree order of the relabelling): wedges u - v - w with v < u and w < u
// are counted per end point w in a hash table, c_w = number of such wedges;
// then
//   u gets sum_w C(c_w, 2), w gets C(c_w, 2),
//   each middle vertex v gets sum over its wedges of (c_w - 1).
// The wedges through v are the entries of row v below u: a prefix of row v
// ending at the position of u, which a search of N+(v) finds. Roots with few
// repeated keys need no counts: a Bloom filter finds the keys that may repeat
// (k_c4_filter). The others are routed by their wedge count W (a count is at
// most W too): one warp with a 6 or 8 KB table (k_c4_warp_left, also for all
// roots of graphs of many triangles; k_c4_warp in small graphs; both go
// without the filter), four warps (k_c4_mid, packed or
// split tables), a 512-thread CTA (k_c4_cta), or, for the largest roots, and
// for every root with more than WL_MAXD in-neighbours, a CTA with a directly
// indexed counter per key in shared memory (k_c4_tiled). The other tables are
// open-addressing hash tables in shared memory, either split (key and count
// arrays) or packed
// (key << cb | count in one 32-bit word, cb = 32 - bits(n - 1) count bits,
// usable while W < 2^cb - 1), which holds twice the keys in the same space.
// Each table is emptied once per CTA; afterwards a warp sweeps the region
// its root used, and a CTA empties the slots it filled (kept in a 16-bit
// `touched` list).
#include <type_traits>

#include "kernels.h"

namespace niorca {

constexpr int CW_WARPS = 4;
constexpr int CW_WORDS = 1536;      // table words per warp of k_c4_warp: 6 KB, 8 CTAs of 4 warps per SM
constexpr int CWB_WORDS = 2048;     // split tables: 8 KB, 6 CTAs per SM
constexpr int CW_MAXW = 1536;       // largest W of a root in the warp tiers
constexpr int CW_SMALL_MAXW = 32;   // the same, for graphs of up to 16 vertices a multiprocessor
constexpr int CW_FEW_MAXW = 128;    // and of up to 32
constexpr int CW_DUPS = 32;         // repeated keys a warp credits by search at most
constexpr int CW_LEFT_LIST = 0;     // list slot of the roots of k_c4_warp_left: the triangle heavy list,
                                    // which nothing reads after that stage
constexpr int CM_THREADS = 128;
constexpr int CM_SLOTS = 4096;      // split; 8192 when packed
constexpr int CM_MAXW = 3072;      // split; 6144 when packed
constexpr int CC_THREADS = 512;
constexpr int CC_SLOTS = 16384;     // split
constexpr int CC_MAXW = 12288;
constexpr unsigned EMPTY = 0xffffffffu;

__device__ __forceinline__ long long c2(long long c) { return c * (c - 1) / 2; }

// Adds c - 1 to pv[q] (shared) for the lanes with c > 1; lanes of one
// in-neighbour q are consecutive in a window, so one add per run. A window
// that lies inside one in-neighbour's run (the usual case on long rows)
// takes one warp reduction and one add.
__device__ __forceinline__ void add_middle(long long *pv, int q, int c) {
    const unsigned v = c > 1 ? (unsigned)(c - 1) : 0u;
    if (!__any_sync(FULL, v != 0)) return;
    const int q0 = __shfl_sync(FULL, q, 0);
    if (__all_sync(FULL, q == q0 || v == 0)) {
        const unsigned t = __reduce_add_sync(FULL, v);
        if (lane_id() == 0) atomicAdd(reinterpret_cast<unsigned long long *>(&pv[q0]), (unsigned long long)t);
        return;
    }
    run_add(&pv[q], q, v);
}

// Wedges u - v - w through the in-neighbour v of root u: the entries of row
// v below u, i.e. the position of u in row v (u is in N+(v)), found by a
// search of N+(v) whose last steps touch the lines the walk reads next.
__device__ __forceinline__ int wedge_len(const Graph &g, int u, const int4 &rv) {
    return lower_bound(g.ncol, rv.y, rv.z, u) - rv.x;
}

// The wedge segment {row start, length} of the in-neighbour at position p of
// row u (din = u's in-degree): from the table k_c4_wedge_len filled, for the
// rows it covers, else by a search of N+(v).
__device__ __forceinline__ int2 wedge_seg(const Graph &g, int u, int din, int p) {
    if (din <= WL_MAXD) return g.wl[p];
    const int4 rv = g.rinfo[g.ncol[p]];
    return make_int2(rv.x, wedge_len(g, u, rv));
}

// The wedge segment of every in-entry of the rows with at most WL_MAXD
// in-neighbours, a group of L lanes per row (16, or 8 for graphs of mean
// degree below 16), a CTA per row from degree WL_LONG on (first, so that no
// group walks a long row alone: R-MAT of 4610 vertices 129 -> 13 us): the row
// gather and binary search of each entry, made here with every thread
// independent, so that the per-root kernels read one coalesced 8-byte entry
// per in-neighbour.
//
// The kernel also samples the graph's triangles and sets CNT_C4_MODE: the
// filter expects few repeated keys from the number of wedges alone, as in a
// random graph, which fails where neighbourhoods overlap. There nearly every
// root repeats keys, and the filter's walk of it is lost (and one atomic per
// root queued). A graph in which more than a third of the pairs of neighbours
// are edges goes to the count tables at once (us a call, filter first /
// tables at once: 1e6 vertices on a ring, degree 32, 10% rewired, 0.53 of the
// pairs: 8131 / 7635; random points in the plane, 3e5 of mean degree 24,
// 0.59: 2080 / 1912; dense parts of 50, 0.43: 6490 / 6035; R-MAT 14, 0.25:
// 471 / 500; R-MAT 16, 0.20: 1315 / 1343). Graphs of mean degree below 12 are
// not sampled: their roots have few wedges (a grid with diagonals, degree 8,
// 0.43: 1151 / 1603).
constexpr int WL_LONG = 128;
constexpr int SAMPLE_CTAS = 8;
enum { C4_FILTER = 1, C4_TABLES = 2 };
template <int L>
__global__ void __launch_bounds__(256, 8) k_c4_wedge_len(Graph g, int2 *wl, const VAcc *vacc, int *counters,
                                                         const int *coff, int ntiles, int sample, int mode) {
    pdl_begin();
    if (call_stopped(counters)) return;
    auto row = [&](int u, int first, int stride) {
        const int4 ru = g.rinfo[u];
        if (ru.y - ru.x > WL_MAXD) return;
        for (int p = ru.x + first; p < ru.y; p += stride) {
            const int4 rv = g.rinfo[g.ncol[p]];
            wl[p] = make_int2(rv.x, wedge_len(g, u, rv));
        }
    };
    const int bound = min(coff[deg_class(WL_LONG) * ntiles], g.n);
    const int ctas = gridDim.x - sample;
    if (sample == 0 && blockIdx.x == 0 && threadIdx.x == 0) counters[CNT_C4_MODE] = mode;
    if ((int)blockIdx.x >= ctas) {   // CTAs of their own for the sample, a vertex of degree below WL_LONG per thread
        const long long at = (long long)(blockIdx.x - ctas) * blockDim.x + threadIdx.x;
        const int u = (int)(at * bound / (sample * (int)blockDim.x));
        long long tri = 0, pairs = 0;
        if (u < bound) {
            const int4 ru = g.rinfo[u];
            const long long d = ru.z - ru.x;
            tri = vacc[u].A1;
            pairs = d * (d - 1);
        }
        tri = warp_sum(tri);
        pairs = warp_sum(pairs);
        if (lane_id() == 0) {
            long long *const sums = reinterpret_cast<long long *>(counters + CNT_CLUSTER);
            add64(sums, tri);
            add64(sums + 1, pairs);
            __threadfence();
            if (atomicAdd(&counters[CNT_SAMPLE_DONE], 1) == sample * ((int)blockDim.x >> 5) - 1) {   // the last warp
                const volatile long long *const all = sums;
                counters[CNT_C4_MODE] = 3 * all[0] > all[1] ? C4_TABLES : C4_FILTER;
            }
        }
        return;
    }
    for (int u = bound + blockIdx.x; u < g.n; u += ctas) row(u, threadIdx.x, blockDim.x);
    const int gh = (blockIdx.x * blockDim.x + threadIdx.x) / L, nh = (ctas * blockDim.x) / L;
    for (int u = gh; u < bound; u += nh) row(u, threadIdx.x & (L - 1), L);
}

// Segment table of in-neighbour chunk cb of root u in the calling warp: the
// wedge prefixes of the rows of v = ncol[b + cb + lane] concatenated. Returns
// the total length; the lane's own v, segment length and offset come back in
// v, len, pre.
__device__ __forceinline__ int wedge_chunk(const Graph &g, int u, int b, int din, int cb, SegTab &T, int &v,
                                           int &len, int &pre) {
    const int p = cb + lane_id();
    int st = 0;
    v = -1;
    len = 0;
    if (p < din) {
        v = g.ncol[b + p];
        const int2 sl = wedge_seg(g, u, din, b + p);
        st = sl.x;
        len = sl.y;
    }
    return seg_build(T, st, len, pre);
}

// Wedge segments of a root's first two chunks of in-neighbours, held in
// registers by the warp (lane p: in-neighbours p and 32 + p) so that its
// walks search no row again.
struct RootChunks {
    int have = 0;          // chunks held: 0, 1 or 2 (warp-uniform)
    int v0 = -1, st0 = 0, len0 = 0, v1 = -1, st1 = 0, len1 = 0;
};

// Segment table of chunk c (in-neighbours 32c ...) of root u, from the
// registers of rc when it holds the chunk, else by searching the rows.
__device__ __forceinline__ int root_chunk(const Graph &g, int u, int b, int din, int c, SegTab &T,
                                          const RootChunks &rc, int &v, int &len, int &pre) {
    if (c < rc.have) {
        v = c == 0 ? rc.v0 : rc.v1;
        len = c == 0 ? rc.len0 : rc.len1;
        return seg_build(T, c == 0 ? rc.st0 : rc.st1, len, pre);
    }
    return wedge_chunk(g, u, b, din, 32 * c, T, v, len, pre);
}

// Walks the wedges of root u (in-neighbours b .. b + din of row u) in the
// calling warp, chunk by chunk of 32 in-neighbours: f(act, q, w) on every
// lane, act meaning that w is a wedge end through the v owned by lane q;
// then done(v) per chunk.
template <class F, class D>
__device__ __forceinline__ void walk_wedges(const Graph &g, int u, int b, int din, SegTab &T, F f, D done,
                                            const RootChunks &rc) {
    for (int c = 0; 32 * c < din; ++c) {
        int v, len, pre;
        const int total = root_chunk(g, u, b, din, c, T, rc, v, len, pre);
        seg_visit32<4>(g.ncol, T, pre, len, total, 0, [&](bool ok, int q, int, int w) { f(ok, q, w); });
        __syncwarp();
        done(v);
        __syncwarp();
    }
}

// The same walk shared by all warps of a CTA: every warp builds the segment
// table of each chunk and takes the windows wid, wid + nw, ... of 32
// elements. With DONE, warp 0 calls done(v) after the CTA finished the chunk.
template <bool DONE, class F, class D>
__device__ __forceinline__ void walk_wedges_cta(const Graph &g, int u, int b, int din, int wid, int nw,
                                                SegTab &T, F f, D done) {
    for (int cb = 0; cb < din; cb += 32) {
        int v, len, pre;
        const int total = wedge_chunk(g, u, b, din, cb, T, v, len, pre);
        seg_visit<4>(g.ncol, T, pre, len, total, wid * 32, nw * 32, [&](bool ok, int q, int, int w) { f(ok, q, w); });
        if (DONE) {
            __syncthreads();
            if (wid == 0) done(v);
            __syncthreads();
        } else {
            __syncwarp();
        }
    }
}

// Probe sequence of the 4-cycle count tables (any size S): first the high
// word of S times the key times 2^32 / golden ratio (Fibonacci hashing; for
// S = 2^k the top k bits of the product), then the same with a second
// multiplier, then linear from there. Keys whose first slots collide part
// ways at the second probe, which keeps the runs, and so a warp's slowest
// insert, short.
__device__ __forceinline__ unsigned fib_slot(int key, unsigned size) {
    return __umulhi(static_cast<unsigned>(key) * 0x9E3779B1u, size);
}
__device__ __forceinline__ unsigned next_probe(unsigned s, unsigned probe, int key, unsigned size) {
    return probe == 0 ? __umulhi(static_cast<unsigned>(key) * 0x85EBCA77u, size) : (s + 1 == size ? 0u : s + 1);
}

// Split table of `size` slots: keys (-1 empty) and counts in two arrays.
struct SplitTab {
    int *hk, *hc;
    unsigned size;
    unsigned short *touched;   // slots filled (CTA groups)
    // counts w; returns the slot if this call inserted w, -1 if w was there
    __device__ __forceinline__ int add(int w) const {
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const int prev = atomicCAS(&hk[s], -1, w);
            if (prev == -1) { atomicAdd(&hc[s], 1); return (int)s; }
            if (prev == w) { atomicAdd(&hc[s], 1); return -1; }
            s = next_probe(s, probe, w, size);
        }
        return -1;
    }
    // Counts w (warp tier); true for the one call whose increment takes
    // w's count from 1 to 2, so that each repeated key is reported once.
    __device__ __forceinline__ bool add_rep(int w) const {
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const int prev = atomicCAS(&hk[s], -1, w);
            if (prev == -1 || prev == w) return atomicAdd(&hc[s], 1) == 1;
            s = next_probe(s, probe, w, size);
        }
        return false;
    }
    __device__ __forceinline__ int get(int w) const {
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const int k = hk[s];
            if (k == w) return hc[s];
            if (k == -1) return 0;
            s = next_probe(s, probe, w, size);
        }
        return 0;
    }
    __device__ __forceinline__ bool empty(int s) const { return hk[s] == -1; }
    __device__ __forceinline__ int key(int s) const { return hk[s]; }
    __device__ __forceinline__ int cnt(int s) const { return hc[s]; }
    __device__ __forceinline__ void clear(int s) const { hk[s] = -1; hc[s] = 0; }
    __device__ __forceinline__ void clear_all(int tid, int nthreads) const {
        for (int i = tid; i < (int)size; i += nthreads) { hk[i] = -1; hc[i] = 0; }
    }
};

// Packed table of `size` slots (a multiple of 4): one word (w << cb) |
// count per slot, EMPTY when free. A count never reaches 2^cb - 1 (the
// caller ensures W < 2^cb - 1), so a full word is never EMPTY.
struct PackedTab {
    unsigned *t;
    unsigned size;
    int cb;
    unsigned short *touched;   // slots filled (CTA groups)
    __device__ __forceinline__ int add(int w) const {
        const unsigned key = static_cast<unsigned>(w);
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const unsigned prev = atomicCAS(&t[s], EMPTY, (key << cb) | 1u);
            if (prev == EMPTY) return (int)s;
            if ((prev >> cb) == key) { atomicAdd(&t[s], 1u); return -1; }
            s = next_probe(s, probe, w, size);
        }
        return -1;
    }
    __device__ __forceinline__ bool add_rep(int w) const {
        const unsigned key = static_cast<unsigned>(w);
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const unsigned prev = atomicCAS(&t[s], EMPTY, (key << cb) | 1u);
            if (prev == EMPTY) return false;
            if ((prev >> cb) == key) return (atomicAdd(&t[s], 1u) & ((1u << cb) - 1)) == 1;
            s = next_probe(s, probe, w, size);
        }
        return false;
    }
    __device__ __forceinline__ int get(int w) const {
        const unsigned key = static_cast<unsigned>(w);
        unsigned s = fib_slot(w, size);
        for (unsigned probe = 0; probe < size; ++probe) {
            const unsigned cur = t[s];
            if (cur == EMPTY) return 0;
            if ((cur >> cb) == key) return (int)(cur & ((1u << cb) - 1));
            s = next_probe(s, probe, w, size);
        }
        return 0;
    }
    __device__ __forceinline__ bool empty(int s) const { return t[s] == EMPTY; }
    __device__ __forceinline__ int key(int s) const { return (int)(t[s] >> cb); }
    __device__ __forceinline__ int cnt(int s) const { return (int)(t[s] & ((1u << cb) - 1)); }
    __device__ __forceinline__ void clear(int s) const { t[s] = EMPTY; }
    __device__ __forceinline__ void clear_all(int tid, int nthreads) const {
        uint4 *t4 = reinterpret_cast<uint4 *>(t);
        for (int i = tid; i < (int)size / 4; i += nthreads) t4[i] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
    }
};

// Counts all wedges of u into the table and credits every 4-cycle rooted at
// u. Every thread of the group (one warp, or a CTA with CTA = true) calls it.
// A repeated key is a 4-cycle, so roots without one skip the credit and
// middle passes. A CTA records the slots it fills in `touched` (flags[0]
// counts them, flags[1] notes a repeated key) and empties only those; a warp
// keeps no list of slots: it uses its whole table for every root, clears all
// of it, and has each repeated key reported by the insert that makes its
// count 2.
// pv holds the per-middle-vertex sums of one chunk (per warp, or shared by
// the CTA).
template <bool CTA, class Tab>
__device__ __forceinline__ void c4_root(const Graph &g, VAcc *vacc, int u, int b, int din,
                                        const Tab &T, int wid, int nw, int tid, int nthreads, SegTab &seg,
                                        long long *pv, int *flags, const RootChunks &rc = RootChunks{},
                                        long long W = 0) {
    const int lane = lane_id();
    auto sync = [] {
        if (CTA) __syncthreads(); else __syncwarp();
    };
    int nrep = 0;   // warp group: repeated keys, the first CW_DUPS of them listed in flags[]
    auto insert = [&](bool act, int, int w) {
        if (!CTA) {
            const bool rep = act && T.add_rep(w);
            const unsigned r = __ballot_sync(FULL, rep);
            if (r) {
                const int at = nrep + __popc(r & lanemask_lt());
                if (rep && at < CW_DUPS) flags[at] = w;
                nrep += __popc(r);
            }
            return;
        }
        const int slot = act ? T.add(w) : -2;
        // new keys of the warp take consecutive `touched` entries
        const unsigned fresh = __ballot_sync(FULL, slot >= 0);
        const unsigned dups = __ballot_sync(FULL, slot == -1);
        if (!(fresh | dups)) return;
        int base = 0;
        if (fresh && lane == __ffs(fresh) - 1) base = atomicAdd(&flags[0], __popc(fresh));
        if (dups && lane == 0) flags[1] = 1;
        if (slot >= 0) {
            base = __shfl_sync(fresh, base, __ffs(fresh) - 1);
            T.touched[base + __popc(fresh & lanemask_lt())] = (unsigned short)slot;
        }
    };
    if (CTA) walk_wedges_cta<false>(g, u, b, din, wid, nw, seg, insert, [](int) {});
    else walk_wedges(g, u, b, din, seg, insert, [](int) {}, rc);
    sync();
    const int nt = CTA ? flags[0] : (int)T.size;   // entries of the list, or slots swept
    bool sweep = CTA ? flags[1] != 0 : false;
    if (!CTA && nrep > 0) {
        // The repeated keys (count >= 2) of a warp's root were reported once
        // each during the walk; up to CW_DUPS of them are listed in flags[],
        // which gives their final counts without sweeping the table (more:
        // a sweep). Each is credited C(c, 2); the middle vertices of key w
        // are N-(u) ∩ N(w), found by searching row w for each in-neighbour
        // (one search per lane and pair), while the pairs number at most
        // W / 4: each search is a short chain of dependent loads, and a root
        // of a small dense graph with tens of repeated keys walks its few
        // windows again sooner. Otherwise: the middle walk below.
        long long su = 0;
        const int nd = nrep;
        if (nd <= CW_DUPS) {
            for (int k = lane; k < nd; k += 32) {
                const int w = flags[k], c = T.get(w);
                flags[CW_DUPS + k] = c;
                su += c2(c);
                add64(&vacc[w].C4, c2(c));
            }
        } else {
            for (int i = lane; i < nt; i += 32) {
                if (T.empty(i)) continue;
                const int c = T.cnt(i);
                if (c >= 2) {
                    su += c2(c);
                    add64(&vacc[T.key(i)].C4, c2(c));
                }
            }
        }
        su = warp_sum(su);
        if (lane == 0) add64(&vacc[u].C4, su);
        __syncwarp();
        if (nd <= CW_DUPS && (long long)nd * din * 4 <= W) {
            // one (key, in-neighbour) pair per lane, all searches independent
            for (int t = lane; t < nd * din; t += 32) {
                const int k = t / din, p = t - k * din;
                const int w = flags[k], c = flags[CW_DUPS + k];
                const int4 rw = g.rinfo[w];
                const int v = g.ncol[b + p];
                if (find_sorted(g.ncol, rw.x, rw.z, v) >= 0) add64(&vacc[v].C4, c - 1);
            }
            __syncwarp();
        } else {
            sweep = true;   // credits done; middle walk only
        }
    }
    if (sweep) {
        if (CTA) {   // (a warp's credits are done)
            long long su = 0;
            for (int i = tid; i < nt; i += nthreads) {
                const int slot = T.touched[i], c = T.cnt(slot);
                if (c >= 2) {
                    su += c2(c);
                    add64(&vacc[T.key(slot)].C4, c2(c));
                }
            }
            su = warp_sum(su);
            if (lane == 0 && su) add64(&vacc[u].C4, su);
        }
        // middle vertices: each wedge through v adds c_w - 1
        if (tid < 32) pv[tid] = 0;
        sync();
        auto middle = [&](bool act, int q, int w) {   // lanes of one v add once
            const int c = act ? T.get(w) : 0;
            add_middle(pv, q, c);
        };
        auto flush = [&](int v) {
            const long long x = pv[lane];
            if (x) add64(&vacc[v].C4, x);
            pv[lane] = 0;
        };
        if (CTA) walk_wedges_cta<true>(g, u, b, din, wid, nw, seg, middle, flush);
        else walk_wedges(g, u, b, din, seg, middle, flush, rc);
        sync();
    }
    if (CTA) {
        for (int i = tid; i < nt; i += nthreads) T.clear(T.touched[i]);
        sync();
        if (tid == 0) {
            flags[0] = 0;
            flags[1] = 0;
        }
    } else {
        T.clear_all(tid, nthreads);
    }
    sync();
}


// ------------------------------- counter layout of the key-tiled tier (below)

constexpr int CK_WORDS = 48 * 1024;   // counter words of a 1024-thread CTA
constexpr int CK_ZONES = 8;

// Counter widths of the zones.
__host__ __device__ constexpr int ck_bits(int zone) {
    return zone == 0 ? 16 : zone == 1 ? 10 : zone == 2 ? 8 : 8 - zone + 1;
}

// Zone z: ids [lo, hi), `per` counters of `bits` bits in a word, stream words
// from `off` on (a multiple of 4). Id w has word off + (hi - 1 - w) / per and
// field (hi - 1 - w) % per. Zones run from the highest ids down.
struct __align__(16) CkZone {
    int lo, hi, off, fmt;
    __device__ __forceinline__ int per() const { return fmt & 0xff; }
    __device__ __forceinline__ int bits() const { return fmt >> 8; }
};

// The zones, from the first id of the class of each zone's lowest degree;
// z[CK_ZONES].off is the length of the stream. One thread.
__device__ __forceinline__ void ck_zones(const int *coff, int ntiles, int n, CkZone *z) {
    const int deg[CK_ZONES] = {1024, 256, 64, 32, 16, 8, 4, 2};
    int hi = n, off = 0;
#pragma unroll
    for (int i = 0; i < CK_ZONES; ++i) {
        CkZone q;
        q.hi = hi;
        q.lo = min(coff[deg_class(deg[i]) * ntiles], hi);
        q.off = off;
        const int bits = ck_bits(i), per = 32 / bits;
        q.fmt = per | bits << 8;
        off += ((hi - q.lo + per - 1) / per + 3) & ~3;
        hi = q.lo;
        z[i] = q;
    }
    z[CK_ZONES].lo = z[CK_ZONES].hi = hi;
    z[CK_ZONES].off = off;
    z[CK_ZONES].fmt = 1;
}

// Wedges from which a root goes to the key-tiled tier. A root there costs
// passes over its in-neighbours and over the counters for every group of
// them, but it has a CTA to itself with no hash: with one group it takes
// roots that the 128-thread tier walks for tens of microseconds (power-law
// graph of 1e5 vertices: call 585 us from 12288 wedges on, 519 from 6144, 477
// from 3072), with many it pays only for the largest (R-MAT 22, six groups:
// 228 ms from 12288 on, 235 from 6144).
__device__ __forceinline__ int ck_min_wedges(const int *coff, int ntiles, int n, int most) {
    CkZone z[CK_ZONES + 1];
    ck_zones(coff, ntiles, n, z);
    const int words = z[CK_ZONES].off;
    return words <= CK_WORDS ? min(most, CM_MAXW) : words <= 4 * CK_WORDS ? min(most, 2 * CM_MAXW) : most;
}

template <int WORDS>
struct __align__(16) C4WarpSmem {
    unsigned t[WORDS];
    SegTab seg;
    long long pv[32];
    int dups[2 * CW_DUPS];   // repeated keys of a root and their counts
};

// Slots of a warp's table of WORDS words (packed words, or split (key,
// count) pairs), and the largest W it takes: 3/4 of the slots.
__host__ __device__ constexpr int cw_slots(bool split, int words) { return split ? words / 2 : words; }
__host__ __device__ constexpr int cw_maxw(bool split, int words) { return cw_slots(split, words) / 4 * 3; }

// ---- roots with few repeated keys, without counting
//
// Most roots of a large sparse graph have no repeated key (G(1e6, mean degree
// 32): 0.03 per root of 256 wedges), and to learn that a root needs no table
// of counts: a blocked Bloom filter does, one atomic per wedge with no probe
// loop (a key clears three bits of one word, and one that finds them clear
// may be a repeat). Which in-neighbours have each of those, and with that the
// exact counts and the middle vertices, then comes from searching their rows
// (few pairs), or from a second walk past a table of the keys alone: a chain
// of searches took 10 us for the largest roots of G(12000, mean degree 15). A
// root with more than CW_DUPS of them goes to a table of counts. The filter
// is all ones when empty, like a table's keys.
// One root of W wedges in a random graph repeats W^2 / 2n keys. Up to 24 of
// them the filter is the better start: with the line at 4, 12, 24 calls on
// G(80000, 40) took 786, 685, 529 us, G(30000, 30) 301, 280, 273, power-law
// graphs of 17000 vertices, whose keys repeat more, 321, 332, 338 (before the
// filter: 849, 324, 500).
__device__ __forceinline__ bool c4_few_repeats(long long W, int n) { return W * W <= 48ll * n; }

// (key, in-neighbour) pairs up to which they are searched, four rounds: G(1e6,
// mean degree 32), whose roots have few, 2820 us a call at 32, 2790 at 64,
// 2754 at 128, 2744 at 256; 8192 small graphs, with many, 12234, 12242, 12269,
// 12335.
constexpr int C4_SEARCH = 128;

// Roots that k_c4_filter leaves, in graphs of up to 2048 vertices a
// multiprocessor: up to C4_FEW_LEFT of them are a few warps' walks in a row
// at the end of the stage, so four warps walk each (k_c4_mid); more have work
// for every warp, and one warp each is the cheaper way (us a call: 300
// power-law graphs of 150 to 1500 vertices 453 with four warps for all, 462
// with the line at 4000, 447 at 8000; one of 2e5 vertices, mean degree 20,
// 1250 with four warps for all, 1235; G(6000, mean degree 30) 175 with the
// line at 1000, 140 from 2000 on).
constexpr int C4_FEW_LEFT = 8192;
__device__ __forceinline__ int c4_mode(const int *counters) {
    return *reinterpret_cast<const volatile int *>(counters + CNT_C4_MODE);
}

template <int LOG>
__device__ __forceinline__ unsigned hash_top(int w) { return (unsigned)w * 0x9E3779B1u >> (32 - LOG); }

__device__ __forceinline__ bool bloom_add(unsigned *t, int log_words, int w) {
    const unsigned h = (unsigned)w * 0x9E3779B1u, b = h << 10;
    const unsigned mask = __funnelshift_l(0u, 1u, b >> 27) | __funnelshift_l(0u, 1u, b >> 22) | __funnelshift_l(0u, 1u, b >> 17);
    return (atomicAnd(&t[h >> (32 - log_words)], ~mask) & mask) == 0;
}

// The wedges of a root of at most 64 in-neighbours (lane: the segments s0 and
// s1 of in-neighbours lane and 32 + lane): eight rows at a time, eight lanes
// and two rows each, f(w[4], pa, pc) with the keys of in-neighbour pa in
// w[0..1] and of pc in w[2..3] (-1: none), by the whole warp.
template <class F>
__device__ __forceinline__ void c4_rows(const int *__restrict__ col, int din, int2 s0, int2 s1, F f) {
    const int sub = lane_id() & 7, q = lane_id() >> 3;
    for (int jb = 0; jb < din; jb += 8) {
        const int2 s = jb < 32 ? s0 : s1;
        const int ja = (jb + q) & 31, jc = (jb + 4 + q) & 31;
        const int xa = __shfl_sync(FULL, s.x, ja), na = __shfl_sync(FULL, s.y, ja);
        const int xc = __shfl_sync(FULL, s.x, jc), nc = __shfl_sync(FULL, s.y, jc);
        const int longest = (int)__reduce_max_sync(FULL, (unsigned)max(na, nc));
        for (int o = sub; o - sub < longest; o += 16) {
            int w[4];
            w[0] = o < na ? __ldg(col + xa + o) : -1;
            w[1] = o + 8 < na ? __ldg(col + xa + o + 8) : -1;
            w[2] = o < nc ? __ldg(col + xc + o) : -1;
            w[3] = o + 8 < nc ? __ldg(col + xc + o + 8) : -1;
            f(w, jb + q, jb + 4 + q);
        }
    }
}

// One root of at most 64 in-neighbours, the warp (segments as in c4_rows).
// False if too many keys may repeat (nothing is credited then).
template <int LOG, class Smem>
__device__ __forceinline__ bool c4_bloom_root(const Graph &g, VAcc *vacc, int u, int b, int din, int2 s0, int2 s1, Smem &S) {
    const int lane = lane_id();
    const int *__restrict__ col = g.ncol;
    int nd = 0;   // keys that may repeat (warp-uniform), the first CW_DUPS of them in S.dups
    c4_rows(col, din, s0, s1, [&](const int (&w)[4], int, int) {
        bool may[4], any = false;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            may[h] = w[h] >= 0 && bloom_add(S.t, LOG, w[h]);
            any |= may[h];
        }
        if (!__any_sync(FULL, any)) return;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const unsigned r = __ballot_sync(FULL, may[h]);
            const int at = nd + __popc(r & lanemask_lt());
            if (may[h] && at < CW_DUPS) S.dups[at] = w[h];
            nd += __popc(r);
        }
    });
    __syncwarp();
#pragma unroll
    for (int i = 0; i < (1 << LOG) / 128; ++i)
        reinterpret_cast<uint4 *>(S.t)[32 * i + lane] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
    if (nd > 0 && nd <= CW_DUPS) {
        // the different ones among them
        const int key = lane < nd ? S.dups[lane] : -1 - lane;
        const unsigned same = __match_any_sync(FULL, key);
        const bool first = lane < nd && lane == __ffs(same) - 1;
        const unsigned firsts = __ballot_sync(FULL, first);
        const int nk = __popc(firsts);
        __syncwarp();
        if (first) S.dups[__popc(firsts & lanemask_lt())] = key;
        unsigned *const common = reinterpret_cast<unsigned *>(S.pv);   // per key, a bit per in-neighbour
        S.pv[lane] = 0;
        __syncwarp();
        if (nk * din <= C4_SEARCH) {
            // one (key, in-neighbour) pair per lane, all searches independent
            for (int t = lane; t < nk * din; t += 32) {
                const int k = t / din, p = t - k * din;
                const int4 rw = g.rinfo[S.dups[k]];
                if (find_sorted(col, rw.x, rw.z, col[b + p]) >= 0) atomicOr(&common[2 * k + (p >> 5)], 1u << (p & 31));
            }
        } else {
            // the rows once more, past a table of the keys (at most 32 in 1 << LOG slots)
            constexpr unsigned MASK = (1u << LOG) - 1;
            unsigned at = 0;
            if (lane < nk) {
                at = hash_top<LOG>(S.dups[lane]);
                while (atomicCAS(&S.t[at], EMPTY, (unsigned)lane) != EMPTY) at = (at + 1) & MASK;
            }
            __syncwarp();
            c4_rows(col, din, s0, s1, [&](const int (&w)[4], int pa, int pc) {
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    const int p = h < 2 ? pa : pc;
                    unsigned x = hash_top<LOG>(w[h]), k;
                    if (w[h] >= 0)
                        for (; (k = S.t[x]) != EMPTY; x = (x + 1) & MASK)
                            if (S.dups[k] == w[h]) {
                                atomicOr(&common[2 * k + (p >> 5)], 1u << (p & 31));
                                break;
                            }
                }
            });
            __syncwarp();
            if (lane < nk) S.t[at] = EMPTY;
        }
        __syncwarp();
        const int c = lane < nk ? __popc(common[2 * lane]) + __popc(common[2 * lane + 1]) : 0;
        if (__any_sync(FULL, c >= 2)) {
            if (c >= 2) add64(&vacc[S.dups[lane]].C4, c2(c));
            const long long su = warp_sum(c2(c));
            if (lane == 0) add64(&vacc[u].C4, su);
            for (int t = lane; t < nk * din; t += 32) {
                const int k = t / din, p = t - k * din;
                const int ck = __popc(common[2 * k]) + __popc(common[2 * k + 1]);
                if (ck >= 2 && (common[2 * k + (p >> 5)] >> (p & 31)) & 1u) add64(&vacc[col[b + p]].C4, ck - 1);
            }
        }
    }
    __syncwarp();
    return nd <= CW_DUPS;
}

// Four roots of at most 8 in-neighbours each (lane 8 q + l: wedge segment s of
// in-neighbour l of root q; its row bounds ru): every lane walks its own
// segment past a filter of 32 words per root. False if a root has too many
// keys that may repeat (nothing is credited then).
template <class Smem>
__device__ __forceinline__ bool c4_bloom_small(const Graph &g, VAcc *vacc, int u, int4 ru, int2 s, Smem &S) {
    const int lane = lane_id(), l = lane & 7, q = lane >> 3;
    const unsigned group = 0xffu << (8 * q);
    const int *__restrict__ col = g.ncol;
    int *const list = S.dups + 16 * q;   // at most 16 keys per root
    int nd = 0;
    const int longest = (int)__reduce_max_sync(FULL, (unsigned)s.y);
    int w = s.y > 0 ? __ldg(col + s.x) : -1;
    for (int o = 0; o < longest; ++o) {
        const int next = o + 1 < s.y ? __ldg(col + s.x + o + 1) : -1;
        const bool may = w >= 0 && bloom_add(S.t + 32 * q, 5, w);
        const unsigned r = __ballot_sync(FULL, may);
        if (r) {
            const int at = nd + __popc(r & group & lanemask_lt());
            if (may && at < 16) list[at] = w;
            nd += __popc(r & group);
        }
        w = next;
    }
    __syncwarp();
    reinterpret_cast<uint4 *>(S.t)[lane] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
    __syncwarp();
    const int most = (int)__reduce_max_sync(FULL, (unsigned)nd);
    if (most > 16) return false;
    const int din = ru.y - ru.x;
    const int v = most > 0 && l < din ? col[ru.x + l] : -1;
    for (int k = 0; k < most; ++k) {   // key k of every root
        const int key = k < nd ? list[k] : -1;
        const bool seen = key >= 0 && ((l < k && list[l] == key) || (l + 8 < k && list[l + 8] == key));
        const bool again = (__ballot_sync(FULL, seen) & group) != 0;
        bool in = false;
        if (key >= 0 && !again && v >= 0) {
            const int4 rw = g.rinfo[key];
            in = find_sorted(col, rw.x, rw.z, v) >= 0;
        }
        const int c = __popc(__ballot_sync(FULL, in) & group);
        if (c < 2) continue;
        if (in) add64(&vacc[v].C4, c - 1);
        if (l < 2) add64(&vacc[l ? key : u].C4, c2(c));
    }
    __syncwarp();
    return true;
}

// Limits of the tiers by wedge count W. A table takes W up to 3/4 of its slots
// (SPLIT: (key, count) pairs, for graphs whose ids leave a packed word too
// few count bits), and a packed count must not reach its field's end.
template <bool SPLIT>
struct C4Limits {
    long long pack, warp, team;   // packed tables, a warp's table, key-tiled from here on
    __device__ __forceinline__ C4Limits(int maxw, int cb, int teamw) {
        pack = (1ll << cb) - 2;
        const long long cap = SPLIT ? maxw : (maxw < pack ? maxw : pack);   // W the warp tiers take
        constexpr int most = cw_maxw(SPLIT, SPLIT ? CWB_WORDS : CW_WORDS);
        warp = cap < most ? cap : most;
        team = teamw;
    }
};

// The wedge segments of a root's in-neighbours lane and 32 + lane (din <= 64;
// s0 is loaded) and its wedge count W, for any din.
__device__ __forceinline__ long long c4_wedges(const Graph &g, int b, int din, int2 s0, int2 &s1) {
    const int lane = lane_id();
    s1 = make_int2(0, 0);
    if (din <= 64) {
        if (32 + lane < din) s1 = g.wl[b + 32 + lane];
        return __reduce_add_sync(FULL, (unsigned)(s0.y + s1.y));   // W <= m < 2^31
    }
    long long W = 0;
    if (din <= WL_MAXD) {
        for (int p = lane; p < din; p += 32) W += g.wl[b + p].y;
    } else {
        // more in-neighbours than the wedge-segment table covers: the
        // key-tiled tier, which takes any root, without searching every row
        // for W here (one warp for a hub's rows would be the kernel's tail);
        // its order takes the in-neighbours' degree sum, at least W, in W's
        // place
#pragma unroll 8
        for (int p = lane; p < din; p += 32) {
            const int4 rv = g.rinfo[g.ncol[b + p]];
            W += rv.z - rv.x;
        }
    }
    return warp_sum(W);
}

// Queues a root for another kernel: k_c4_warp_left (`warp`: that is the next
// one), or a wider tier's.
template <bool SPLIT>
__device__ __forceinline__ void c4_queue_root(const Graph &g, int *lists, int *counters, int u, int din, long long W, bool warp,
                                              const C4Limits<SPLIT> &lim) {
    if (lane_id() != 0) return;
    int which, list;   // queue counter and list slot (lists + list * n)
    if (din > WL_MAXD) { which = CNT_C4_TEAM; list = 4; }
    else if (warp && W <= lim.warp) { which = CNT_C4_LEFT; list = CW_LEFT_LIST; }
    else if (W > lim.team) { which = CNT_C4_TEAM; list = 4; }
    else if (W <= 2 * CM_MAXW && W <= lim.pack) { which = CNT_C4_MIDP; list = 5; }
    else if (W <= CM_MAXW) { which = CNT_C4_MID; list = 2; }
    else { which = CNT_C4_CTA; list = 3; }
    const int at = atomicAdd(&counters[which], 1);
    lists[(size_t)list * g.n + at] = u;
    if (which == CNT_C4_TEAM)   // the order of the key-tiled tier
        lists[(size_t)g.n + at] = (int)(W < 0x7fffffffll ? W : 0x7fffffffll);
}

// The roots i = first, first + nw, ... < count of a warp, f(u, row bounds,
// wedge segment of in-neighbour `lane`), in a software pipeline: row bounds
// are loaded two roots ahead, the first 32 segments one root ahead.
template <class R, class F>
__device__ __forceinline__ void c4_roots(const Graph &g, int first, int nw, int count, R root, F f) {
    const int lane = lane_id();
    const int4 Z = make_int4(0, 0, 0, 0);
    const int2 Z2 = make_int2(0, 0);
    int i = first;
    int u = i < count ? root(i) : 0;
    int un = i + nw < count ? root(i + nw) : 0;
    int4 ru = i < count ? g.rinfo[u] : Z;
    int4 ru1 = i + nw < count ? g.rinfo[un] : Z;
    int2 s0 = (i < count && lane < ru.y - ru.x && ru.y - ru.x <= 64) ? g.wl[ru.x + lane] : Z2;
    for (; i < count; i += nw) {
        const int i2 = i + 2 * nw;
        const int u2 = i2 < count ? root(i2) : 0;
        const int4 ru2 = i2 < count ? g.rinfo[u2] : Z;
        const int2 s1 = (i + nw < count && lane < ru1.y - ru1.x && ru1.y - ru1.x <= 64) ? g.wl[ru1.x + lane] : Z2;
        f(u, ru, s0);
        u = un;
        un = u2;
        ru = ru1;
        ru1 = ru2;
        s0 = s1;
    }
}

// One warp per root, with a count table. In small graphs k_c4_warp takes
// every vertex as a root and queues those above its limit for the wider
// tiers; in others k_c4_filter is the first kernel, and k_c4_warp_left
// (QUEUE) takes the smaller roots that it could not finish, or, where the
// filter does not run, every vertex (`count` of them). Packed tables
// have 6 KB (8 CTAs per SM); ids that need split tables have 8 KB, since those
// take half the wedges in the same space, and the 4-warp tier the rest (8192
// small graphs: 442 + 2607 us with 6 KB, 717 + 2157 with 8 KB).
template <bool SPLIT, bool QUEUE, class Smem>
__device__ __forceinline__ void c4_warp_body(Smem *sm_all, const Graph &g, VAcc *vacc, int *lists, int *counters, int maxw, int cb,
                                             int teamw, int count) {
    constexpr int WORDS = SPLIT ? CWB_WORDS : CW_WORDS;
    constexpr int TS = cw_slots(SPLIT, WORDS);
    Smem &S = sm_all[threadIdx.x >> 5];
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const C4Limits<SPLIT> lim(maxw, cb, teamw);
    const int *const left = lists + (size_t)CW_LEFT_LIST * g.n;
    int *const sk = reinterpret_cast<int *>(S.t), *const sc = sk + TS;   // split keys, counts
    if (SPLIT) SplitTab{sk, sc, (unsigned)TS, nullptr}.clear_all(lane, 32);
    else PackedTab{S.t, (unsigned)TS, cb, nullptr}.clear_all(lane, 32);
    __syncwarp();
    c4_roots(
        g, gw, nw, count, [&](int i) { return QUEUE ? left[i] : i; },
        [&](int u, const int4 &ru, int2 s0) {
            const int b = ru.x, din = ru.y - ru.x;
            if (din < 2) return;
            int2 s1;
            const long long W = c4_wedges(g, b, din, s0, s1);
            const bool hub = din > WL_MAXD;
            if (W < 2 && !hub) return;
            if (!QUEUE && (W > lim.warp || hub)) {
                c4_queue_root(g, lists, counters, u, din, W, false, lim);
                return;
            }
            RootChunks rc;
            if (din <= 64) {   // both chunks' segments stay in registers
                rc.have = din > 32 ? 2 : 1;
                rc.st0 = s0.x, rc.len0 = s0.y, rc.st1 = s1.x, rc.len1 = s1.y;
                rc.v0 = lane < din ? g.ncol[b + lane] : -1;   // for the middle walk's credits
                rc.v1 = 32 + lane < din ? g.ncol[b + 32 + lane] : -1;
            }
            // every root takes the whole table: at the low load this leaves
            // (W / 1536 on the 6 KB table) a warp's slowest insert needs fewer
            // probes, which paid more than the larger clear and sweep cost
            if constexpr (SPLIT) {
                const SplitTab T{sk, sc, (unsigned)TS, nullptr};
                c4_root<false>(g, vacc, u, b, din, T, 0, 1, lane, 32, S.seg, S.pv, S.dups, rc, W);
            } else {
                const PackedTab T{S.t, (unsigned)TS, cb, nullptr};
                c4_root<false>(g, vacc, u, b, din, T, 0, 1, lane, 32, S.seg, S.pv, S.dups, rc, W);
            }
        });
}

// 8 CTAs of 4 warps per SM: 6 KB tables and at most 64 registers a thread.
template <bool SPLIT>
__global__ void __launch_bounds__(CW_WARPS * 32, SPLIT ? 6 : 8) k_c4_warp(Graph g, VAcc *vacc, int *lists, int *counters,
                                                                          int maxw, int cb, int teamw, const int *coff,
                                                                          int ntiles) {
    pdl_begin();
    __shared__ C4WarpSmem<SPLIT ? CWB_WORDS : CW_WORDS> sm[CW_WARPS];
    if (call_stopped(counters)) return;
    c4_warp_body<SPLIT, false>(sm, g, vacc, lists, counters, maxw, cb, ck_min_wedges(coff, ntiles, g.n, teamw), g.n);
}

template <bool SPLIT>
__global__ void __launch_bounds__(CW_WARPS * 32, SPLIT ? 6 : 8) k_c4_warp_left(Graph g, VAcc *vacc, int *lists,
                                                                               int *counters, int maxw, int cb, int few,
                                                                               int teamw, const int *coff, int ntiles) {
    pdl_begin();
    __shared__ C4WarpSmem<SPLIT ? CWB_WORDS : CW_WORDS> sm[CW_WARPS];
    const int mode = c4_mode(counters), left = counters[CNT_C4_LEFT];
    if (mode == C4_FILTER && left <= few) {   // k_c4_mid's, behind its own
        int *const midp = lists + 5 * (size_t)g.n + counters[CNT_C4_MIDP];
        const int first = blockIdx.x * blockDim.x + threadIdx.x;
        for (int i = first; i < left; i += gridDim.x * blockDim.x) midp[i] = lists[(size_t)CW_LEFT_LIST * g.n + i];
        if (first == 0) counters[CNT_C4_MIDP_LEFT] = left;
    } else if (mode == C4_FILTER) c4_warp_body<SPLIT, true>(sm, g, vacc, lists, counters, maxw, cb, 0, left);
    else if (mode == C4_TABLES)
        c4_warp_body<SPLIT, false>(sm, g, vacc, lists, counters, maxw, cb, ck_min_wedges(coff, ntiles, g.n, teamw), g.n);
}

// The first kernel of large graphs: every vertex as a root, the filter only.
// Without the table's code it takes 48 registers and 4.5 KB a warp, 40 warps
// per SM instead of 32 (40 registers and 48 warps spill: 1.33 ms against 1.04
// on G(1e6, mean degree 32), where the tables of three kernels took 1.79 ms;
// G(3e6, mean degree 6) 0.37 ms against 0.76).
// It is bound by the latency of row bounds -> segments -> rows and by issue,
// about 60 instructions per 32 wedges.
constexpr int CF_WARPS = 8;
constexpr int CF_LOG = 10;
// W that the filter takes, for tables of up to maxw: 2048 at the default of
// 1536. That is two keys per word of the filter, of which about 8 may be
// falsely taken for repeats.
__device__ __forceinline__ int cf_maxw(int maxw) { return maxw * 4 / 3; }

struct __align__(16) C4FilterSmem {
    unsigned t[1 << CF_LOG];
    long long pv[32];
    int dups[2 * CW_DUPS];
};

template <bool SPLIT>
__global__ void __launch_bounds__(CF_WARPS * 32, 5) k_c4_filter(Graph g, VAcc *vacc, int *lists, int *counters, int maxw,
                                                                int cb, int teamw, const int *coff, int ntiles) {
    pdl_begin();
    if (c4_mode(counters) != C4_FILTER) return;
    extern __shared__ __align__(16) unsigned char dsm[];
    C4FilterSmem &S = reinterpret_cast<C4FilterSmem *>(dsm)[threadIdx.x >> 5];
    const int lane = lane_id();
    const int gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    const C4Limits<SPLIT> lim(maxw, cb, ck_min_wedges(coff, ntiles, g.n, teamw));
    const long long most = min((long long)cf_maxw(maxw), lim.team);
    for (int i = lane; i < (1 << CF_LOG) / 4; i += 32) reinterpret_cast<uint4 *>(S.t)[i] = make_uint4(EMPTY, EMPTY, EMPTY, EMPTY);
    __syncwarp();
    auto do_root = [&](int u, const int4 &ru, int2 s0) {
        const int b = ru.x, din = ru.y - ru.x;
        if (din < 2) return;
        int2 s1;
        const long long W = c4_wedges(g, b, din, s0, s1);
        if (W < 2 && din <= WL_MAXD) return;
        if (din <= 64 && W <= most && c4_few_repeats(W, g.n) && c4_bloom_root<CF_LOG>(g, vacc, u, b, din, s0, s1, S)) return;
        c4_queue_root(g, lists, counters, u, din, W, true, lim);
    };
    // ids of low degree: four roots at a time, eight lanes each
    const int2 Z2 = make_int2(0, 0);
    const int low = most >= 8 * SMALL_ROW ? low_degree_ids(g.n, nw, coff, ntiles) : 0;
    for (long long u0 = 4ll * gw; u0 < low; u0 += 4ll * nw) {
        const int u = (int)u0 + (lane >> 3), l = lane & 7;
        int4 ru = make_int4(0, 0, 0, 0);
        if (u < low) ru = g.rinfo[u];
        const int din = ru.y - ru.x;
        if (!__any_sync(FULL, din > 8)) {
            const int2 s = l < din ? g.wl[ru.x + l] : Z2;
            if (!__any_sync(FULL, s.y > SMALL_ROW) && c4_bloom_small(g, vacc, u, ru, s, S)) continue;
        }
        for (int q = 0; q < 4; ++q) {
            const int x = __shfl_sync(FULL, ru.x, 8 * q), y = __shfl_sync(FULL, ru.y, 8 * q);
            do_root((int)u0 + q, make_int4(x, y, 0, 0), lane < y - x && y - x <= 64 ? g.wl[x + lane] : Z2);
        }
    }
    c4_roots(g, low + gw, nw, g.n, [](int i) { return i; }, do_root);
}

// Roots from a queue, one CTA each. The table (SLOTS split slots, or
// 2 x SLOTS packed ones) lives in dynamic shared memory and is emptied once
// per CTA.
template <int THREADS, int SLOTS, int MAXW, bool PACKED>
__device__ __forceinline__ void c4_queue(const Graph &g, VAcc *vacc, const int *list, int count, int *next,
                                         int cb) {
    extern __shared__ __align__(16) unsigned char dsm[];
    constexpr int NW = THREADS / 32;
    constexpr int NT = PACKED ? 2 * MAXW : MAXW;   // touched capacity: every key of a root
    unsigned *words = reinterpret_cast<unsigned *>(dsm);            // 2 x SLOTS words
    unsigned short *touched = reinterpret_cast<unsigned short *>(words + 2 * SLOTS);
    SegTab *segs = reinterpret_cast<SegTab *>(touched + NT);         // one per warp
    long long *pv = reinterpret_cast<long long *>(segs + NW);        // 32, shared by the CTA
    int *flags = reinterpret_cast<int *>(pv + 32);                  // new keys, repeated key
    const int wid = threadIdx.x >> 5;
    SegTab &seg = segs[wid];
    if (PACKED) {
        for (int i = threadIdx.x; i < 2 * SLOTS; i += THREADS) words[i] = EMPTY;
    } else {
        for (int i = threadIdx.x; i < SLOTS; i += THREADS) { words[i] = EMPTY; words[SLOTS + i] = 0; }
    }
    if (threadIdx.x == 0) { flags[0] = 0; flags[1] = 0; }
    __syncthreads();
    for (int h = cta_next(next); h < count; h = cta_next(next)) {
        const int u = list[h];
        const int4 ru = g.rinfo[u];
        if (PACKED) {
            const PackedTab T{words, 2 * SLOTS, cb, touched};
            c4_root<true>(g, vacc, u, ru.x, ru.y - ru.x, T, wid, NW, threadIdx.x, THREADS, seg, pv, flags);
        } else {
            const SplitTab T{reinterpret_cast<int *>(words), reinterpret_cast<int *>(words + SLOTS), SLOTS, touched};
            c4_root<true>(g, vacc, u, ru.x, ru.y - ru.x, T, wid, NW, threadIdx.x, THREADS, seg, pv, flags);
        }
    }
}

constexpr size_t cq_smem(int threads, int slots, int maxw) {
    // 2 x slots words, 2 x maxw 16-bit touched entries, segments, pv, flags
    return (size_t)2 * slots * 4 + (size_t)2 * maxw * 2 + (size_t)(threads / 32) * sizeof(SegTab) + 32 * 8 + 16;
}
constexpr size_t CM_SMEM = cq_smem(CM_THREADS, CM_SLOTS, CM_MAXW);
constexpr size_t CC_SMEM = cq_smem(CC_THREADS, CC_SLOTS, CC_MAXW);

// Both 128-thread queues in one launch: the packed one (W <= 6144 with
// enough count bits), then the split one (W <= 3072).
__global__ void __launch_bounds__(CM_THREADS) k_c4_mid(Graph g, VAcc *vacc, const int *lists, int *counters,
                                                       int cb) {
    pdl_begin();
    const int np = counters[CNT_C4_MIDP] + counters[CNT_C4_MIDP_LEFT], nm = counters[CNT_C4_MID];   // (0 in a stopped call)
    if (np == 0 && nm == 0) return;
    c4_queue<CM_THREADS, CM_SLOTS, CM_MAXW, true>(g, vacc, lists + 5 * (size_t)g.n, np, counters + CNT_C4_MIDP_NEXT, cb);
    c4_queue<CM_THREADS, CM_SLOTS, CM_MAXW, false>(g, vacc, lists + 2 * (size_t)g.n, nm, counters + CNT_C4_MID_NEXT, cb);
}

__global__ void __launch_bounds__(CC_THREADS) k_c4_cta(Graph g, VAcc *vacc, const int *lists, int *counters,
                                                       int cb) {
    pdl_begin();
    if (call_stopped(counters)) return;
    c4_queue<CC_THREADS, CC_SLOTS, CC_MAXW, false>(g, vacc, lists + 3 * (size_t)g.n, counters[CNT_C4_CTA],
                                                   counters + CNT_C4_CTA_NEXT, cb);
}

// ------------------------------------------------------ key-tiled tier
//
// Roots with more wedges than the hash tiers take (W > teamw): one CTA per
// root, largest roots first. The keys w of a root u are the vertices below
// u; their counters are packed words in shared memory, indexed by w.
//
// Counter stream. A count c_uw is at most the degree of w, and ids are
// ordered by degree class, so an id range has a fixed counter width (zones,
// ck_zones: 2 bits for degrees 2-3, 3 for 4-7, ... 10 for 256-1023, 16
// above; a root whose counts could pass 16 bits takes the last zone with
// 32-bit counters, c4_wide_top). Vertices of degree 0 and 1 are on no cycle
// and have no counter. All counters form one stream of words, from the
// highest id down; a group is the part of it that fits the shared memory.
//
// The layout is the same for every root, so each column entry's counter
// (byte address in its group, shift, width) is computed once (`enc`), as are
// the position in every row where each group starts (`index`, group by
// group over the vertices) and the position of every root in its
// in-neighbours' rows (`ends`): k_c4_tiled_plan. They live in the
// triangle-count region, which nothing reads after the hash tiers.
//
// A root takes group after group: it counts its wedges that end in the
// group (the entries of row v in the group's id range and below u are a
// contiguous run), walks them again adding c - 1 per wedge to the middle
// vertex, then sweeps the counters, crediting C(c, 2) to every key and to u,
// and clears them. A walk takes the runs in batches of one per thread
// (loaded one batch ahead): a run of at most CK_TINY entries is walked by
// its thread; the others are listed in shared memory with the prefix sums of
// their windows of 32 entries, and every warp takes an equal share of the
// windows. A window lies in one run: a warp finds the runs of 32 windows at
// once (one window per lane, into a shared list) and then spends a load, two
// shifts and an atomic on each window, CK_UNROLL of them in flight.
//
// Measured (GB300, the tier's time): R-MAT 22 364 -> 114 ms, R-MAT 18
// 5.34 -> 1.83 ms, R-MAT 14 0.34 -> 0.12 ms, G(1501, 0.5) 1.34 -> 0.48 ms,
// against tiles of 104448 16-bit counters whose runs were concatenated and
// looked up entry by entry (63 and 88 instructions per 32 wedges in the two
// walks). It is bound by shared memory now: on R-MAT 21 the LSU data pipe is
// 68% busy (3.4 wavefronts per 32 random counter updates) and 60% of the
// sectors hit L2. Two 512-thread CTAs per SM with half the counters took
// twice the time (every group passes over all in-neighbours).
constexpr int CK_TINY = 4;
constexpr int CK_NARROW_MAXD = 65534;               // in-degree up to which 16-bit counters cannot overflow
constexpr int CK_SMALL_N = 12288;                   // graphs whose 16-bit counters fit 24 KB: 256-thread CTAs
constexpr int CK_MAX_GROUPS = 64;                   // groups up to which there may be an index
constexpr int CK_ENDS_MAXD = 8192;                  // in-degree of a root up to which `ends` holds its positions
constexpr int CK_UNROLL = 16;                       // windows a warp has in flight (R-MAT 22: 125 ms with 8)
constexpr size_t ck_smem(int threads, int words) {
    // counters; per thread: run start, length, window prefix, vertex and a window; warp totals, zones, scalars
    return (size_t)words * 4 + (size_t)threads * 24 + (size_t)(threads / 32) * 8 + (CK_ZONES + 1) * 16 + 32;
}
static_assert(ck_smem(1024, CK_WORDS) <= 227 * 1024, "k_c4_tiled shared memory");

// Lowest id with a counter before stream word e.
__device__ __forceinline__ int ck_low_id(const CkZone *z, long long e) {
    int lo = z[0].hi;
    for (int i = 0; i < CK_ZONES && z[i].off < e; ++i)
        lo = (int)max((long long)z[i].lo, z[i].hi - (e - z[i].off) * z[i].per());
    return lo;
}

// Where the plan's arrays lie in the triangle-count region (2 m ints): enc
// (m ints), ends (m 16-bit offsets from the split of the in-neighbour's
// row; an out-degree is at most sqrt(1.25 m) < 2^16), index (groups x n
// ints, when there is room).
struct CkPlan {
    int *enc;
    unsigned short *ends;
    int *index;
    int groups;
    bool indexed;
};
__device__ __forceinline__ CkPlan ck_plan(int *region, const CkZone *z, int words, int n, int m) {
    CkPlan P;
    P.enc = region;
    P.ends = reinterpret_cast<unsigned short *>(region + m);
    P.index = region + m + (m + 1) / 2;
    P.groups = (z[CK_ZONES].off + words - 1) / words;
    P.indexed = P.groups <= CK_MAX_GROUPS && (long long)P.groups * n <= m / 2;
    return P;
}

// CTA 0: root order of the key-tiled tier: the queued roots (list 4, their
// wedge counts in list 1) sorted by decreasing wedge count (64 buckets, two
// per octave) into list 0. Their in-degrees sum to more than m / 2 only in a
// CSR that is not symmetric, which is reported. Every other CTA: enc, ends and
// index.
__global__ void __launch_bounds__(1024) k_c4_tiled_plan(Graph g, int *lists, int *counters, const int *coff, int ntiles,
                                                        int words, int *region, int *status) {
    pdl_begin();
    __shared__ int hist[64], base[64];
    __shared__ long long degrees;
    __shared__ CkZone z[CK_ZONES + 1];
    __shared__ int glo[CK_MAX_GROUPS];
    if (call_stopped(counters)) return;
    const int nt = counters[CNT_C4_TEAM];
    if (nt == 0) return;
    const int *roots = lists + 4 * (size_t)g.n, *wts = lists + (size_t)g.n;
    if (blockIdx.x > 0) {
        if (threadIdx.x == 0) ck_zones(coff, ntiles, g.n, z);
        __syncthreads();
        const CkPlan P = ck_plan(region, z, words, g.n, g.m);
        if ((int)threadIdx.x < min(P.groups, CK_MAX_GROUPS))
            glo[threadIdx.x] = ck_low_id(z, (long long)(threadIdx.x + 1) * words);
        __syncthreads();
        const int first = z[CK_ZONES].lo;   // rows below have degree 0 or 1
        const int b = blockIdx.x - 1;
        const long long t0 = b * (long long)blockDim.x + threadIdx.x, stride = (long long)(gridDim.x - 1) * blockDim.x;
        for (long long p = t0; p < g.m; p += stride) {
            const int w = g.ncol[p];
            int i = 0;
            while (i < CK_ZONES && w < z[i].lo) ++i;
            if (i == CK_ZONES) {   // no counter, and below every run of a sorted row
                P.enc[p] = 0;
                continue;
            }
            const CkZone q = z[i];
            const unsigned k = (unsigned)(q.hi - 1 - w), per = (unsigned)q.per(), word = k / per;
            const unsigned at = (unsigned)q.off + word, local = at - at / (unsigned)words * (unsigned)words;
            P.enc[p] = (int)(local << 12 | (unsigned)(32 - q.bits()) << 5 | (k - word * per) * (unsigned)q.bits());
        }
        if (P.indexed)
            for (int i = 0; i < P.groups; ++i) {
                const int key = glo[i];
                for (long long v = first + t0; v < g.n; v += stride) {
                    const int4 rv = g.rinfo[v];
                    P.index[(size_t)i * g.n + v] = lower_bound(g.ncol, rv.x, rv.z, key);
                }
            }
        for (int r = b * 4 + (threadIdx.x >> 8); r < nt; r += (gridDim.x - 1) * 4) {   // 256 threads per root
            const int u = roots[r];
            const int4 ru = g.rinfo[u];
            if (ru.y - ru.x > CK_ENDS_MAXD) continue;
            for (int p = ru.x + (threadIdx.x & 255); p < ru.y; p += 256) {
                const int4 rv = g.rinfo[g.ncol[p]];
                P.ends[p] = (unsigned short)min(lower_bound(g.ncol, rv.y, rv.z, u) - rv.y, 65535);
            }
        }
        return;
    }
    int *sorted = lists;
    auto bucket = [](int w) {
        const int e = 31 - __clz(max(w, 1));
        const int half = e > 0 ? (w >> (e - 1)) & 1 : 0;
        return 63 - min(63, 2 * e + half);
    };
    if (threadIdx.x < 64) hist[threadIdx.x] = 0;
    if (threadIdx.x == 0) degrees = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < nt; i += blockDim.x) atomicAdd(&hist[bucket(wts[i])], 1);
    __syncthreads();
    if (threadIdx.x < 32) {   // exclusive scan of 64 buckets, two per lane
        const int a = hist[2 * threadIdx.x], b = hist[2 * threadIdx.x + 1];
        const int ex = warp_inclusive_scan(a + b) - (a + b);
        base[2 * threadIdx.x] = ex;
        base[2 * threadIdx.x + 1] = ex + a;
    }
    __syncthreads();
    long long din = 0;
    for (int i = threadIdx.x; i < nt; i += blockDim.x) {
        const int u = roots[i];
        sorted[atomicAdd(&base[bucket(wts[i])], 1)] = u;
        const int4 ru = g.rinfo[u];
        din += ru.y - ru.x;
    }
    din = warp_sum(din);
    if (lane_id() == 0) add64(&degrees, din);
    __syncthreads();
    if (threadIdx.x == 0 && degrees > g.m / 2) set_status(status, ST_ENOTSIMPLE);
}

// What a CTA keeps in shared memory.
struct CkShared {
    unsigned char *cnt;        // a group's counters, and four words that stay 0
    int *st, *len, *win, *v;   // a batch's listed runs: start, length, first window, vertex
    int2 *wnd;                 // the warp's 32 windows: first entry, entries
    int *wwin, *wrun;          // windows and listed runs of every warp's part of the batch
    CkZone *z;
    int *any, *job;
    long long *twice;          // sum of c - 1 over the root's wedges
    // adds one to / reads the counter of a column entry (see k_c4_tiled_plan:
    // byte address << 10 | (32 - bits) << 5 | shift; shifts wrap at 32)
    __device__ __forceinline__ void add(unsigned e) const {
        atomicAdd(reinterpret_cast<unsigned *>(cnt + (e >> 10)), __funnelshift_l(0u, 1u, e));
    }
    __device__ __forceinline__ unsigned get(unsigned e) const {
        const unsigned x = *reinterpret_cast<const unsigned *>(cnt + (e >> 10));
        const unsigned r = e >> 5;
        return __funnelshift_r(__funnelshift_l(0u, x, r - e), 0u, r);
    }
};

// Credits C(c, 2) to every key with c >= 2 of the group's stream words
// [max(gw0, from), to), zone by zone from Z on, and clears the words. Most
// words of the narrow zones hold no count above 1: four words are tested at
// once, and only the fields that pass are visited; a word of the wide zones
// has at most four fields, each taken with constant shifts.
template <int THREADS, int Z>
__device__ __forceinline__ void ck_sweep(const CkShared &S, VAcc *vacc, int gw0, int from, int to) {
    constexpr int BITS = ck_bits(Z), PER = 32 / BITS;
    constexpr unsigned FIELD = (1u << BITS) - 1u;
    constexpr unsigned GE2 = [] {   // the bits that are set in some field of 2 or more
        unsigned m = 0;
        for (int f = 0; f < PER; ++f) m |= (FIELD - 1u) << (f * BITS);
        return m;
    }();
    const CkZone z = S.z[Z];
    const int ws = max(max(z.off, gw0), from), we = min(S.z[Z + 1].off, to);
    for (int s = ws + 4 * (int)threadIdx.x; s < we; s += 4 * THREADS) {
        uint4 *const at = reinterpret_cast<uint4 *>(S.cnt + 4 * (size_t)(s - gw0));
        const uint4 x4 = *at;
        const unsigned some = x4.x | x4.y | x4.z | x4.w;
        if (!some) continue;
        *at = make_uint4(0, 0, 0, 0);
        if (!(some & GE2)) continue;
        const unsigned xs[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            unsigned m = xs[h] & GE2;
            if (!m) continue;
            const int w = z.hi - 1 - (s + h - z.off) * PER;   // key of field 0, the others descend from it
            VAcc *const p = vacc + w;
            if constexpr (PER <= 4) {
#pragma unroll
                for (int f = 0; f < PER; ++f) {
                    const unsigned c = (xs[h] >> (f * BITS)) & FIELD;   // below 2^16: c (c - 1) fits 32 bits
                    if (c >= 2 && w - f >= z.lo) add64(&p[-f].C4, (long long)(c * (c - 1u) / 2u));
                }
            } else {
                while (m) {
                    const int f = (31 - __clz(m)) / BITS;
                    m &= ~(FIELD << (f * BITS));
                    const unsigned c = (xs[h] >> (f * BITS)) & FIELD;
                    if (w - f >= z.lo) add64(&p[-f].C4, (long long)(c * (c - 1u) / 2u));
                }
            }
        }
    }
    if constexpr (Z + 1 < CK_ZONES) ck_sweep<THREADS, Z + 1>(S, vacc, gw0, from, to);
}

// One root, the whole CTA: the keys below ulim (u, or for a root with
// c4_wide_top the first id of zone 0).
template <int THREADS>
__device__ __forceinline__ void c4_tiled_root(const Graph &g, VAcc *vacc, int u, int ulim, int words, const CkPlan &P,
                                              const CkShared &S) {
    constexpr int NW = THREADS / 32, U = CK_UNROLL;
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    const int *__restrict__ col = g.ncol;
    const int *__restrict__ enc = P.enc, *__restrict__ encl = P.enc + lane;
    const unsigned none = (unsigned)words << 12;
    const int *__restrict__ index = P.index;
    const int4 ru = g.rinfo[u];
    const int b = ru.x, din = ru.y - ru.x;
    const int first = S.z[CK_ZONES].lo;
    long long su = 0;
    if (ulim <= first) return;
    int lim_word = 0;   // the stream word of id ulim - 1, the first one the root may use
    for (int i = 0; i < CK_ZONES; ++i)
        if (ulim - 1 >= S.z[i].lo) {
            lim_word = S.z[i].off + (max(S.z[i].hi - ulim, 0)) / S.z[i].per();
            break;
        }
    const int g0 = lim_word / words;
    for (int gi = g0; gi < P.groups; ++gi) {
        const int glo = P.indexed ? 0 : ck_low_id(S.z, (long long)(gi + 1) * words);
        const int ghi = P.indexed || gi == g0 ? ulim : ck_low_id(S.z, (long long)gi * words);
        auto vertex = [&](int e) { return e < din ? col[b + e] : -1; };
        auto run = [&](int e, int v) {   // {start, end} of the run of in-neighbour e, v
            if (v < first) return make_int2(0, 0);   // none, or a row of one entry
            if (P.indexed) {
                const int x = index[(size_t)gi * g.n + v];
                if (gi > g0) return make_int2(x, index[(size_t)(gi - 1) * g.n + v]);
                const int4 rv = g.rinfo[v];
                if (ulim < u) return make_int2(x, lower_bound(col, x, rv.z, ulim));
                return make_int2(x, din <= CK_ENDS_MAXD ? rv.y + (int)P.ends[b + e] : lower_bound(col, rv.y, rv.z, u));
            }
            const int4 rv = g.rinfo[v];
            const int x = lower_bound(col, rv.x, rv.z, glo);
            return make_int2(x, lower_bound(col, x, rv.z, ghi));
        };
        // One walk over the group's runs. MID: sum c - 1 per run into the
        // middle vertices; else count.
        auto walk = [&](auto mid) {
            constexpr bool MID = decltype(mid)::value;
            bool any = false;
            int v = vertex((int)threadIdx.x);
            int2 r = run((int)threadIdx.x, v);
            int vn = vertex(THREADS + (int)threadIdx.x);
            for (int e0 = 0; e0 < din; e0 += THREADS) {
                const int e = e0 + (int)threadIdx.x;
                const int len = r.y - r.x;
                const bool list = len > CK_TINY;
                // list the batch's longer runs with their first windows
                const int nwin = list ? (len + 31) >> 5 : 0;
                const unsigned bal = __ballot_sync(FULL, list);
                const int incl = warp_inclusive_scan(nwin);
                if (lane == 31) {
                    S.wwin[wid] = incl;
                    S.wrun[wid] = __popc(bal);
                }
                __syncthreads();   // and the batch before is done with the list
                const int tw = lane < NW ? S.wwin[lane] : 0, tr = lane < NW ? S.wrun[lane] : 0;
                const int iw = warp_inclusive_scan(tw), ir = warp_inclusive_scan(tr);
                const int total = __shfl_sync(FULL, iw, 31), nlist = __shfl_sync(FULL, ir, 31);
                const int w0 = __shfl_sync(FULL, iw - tw, wid), q0 = __shfl_sync(FULL, ir - tr, wid);
                if (list) {
                    const int q = q0 + __popc(bal & lanemask_lt());
                    S.st[q] = r.x;
                    S.len[q] = len;
                    S.win[q] = w0 + incl - nwin;
                    S.v[q] = v;
                }
                if (len > 0) any = true;
                if (len > 0 && !list) {
                    unsigned a = 0;
                    for (int q = r.x; q < r.y; ++q) {
                        const unsigned c = (unsigned)__ldg(enc + q);
                        if (MID) a += S.get(c) - 1u; else S.add(c);
                    }
                    if (MID && a) {
                        add64(&vacc[v].C4, a);
                        su += a;
                    }
                }
                __syncthreads();
                // the next batch's runs, in flight during this one
                v = vn;
                r = run(e + THREADS, v);
                vn = vertex(e + 2 * THREADS);
                // this warp's share of the windows, [x, y)
                const int x = (int)((long long)total * wid / NW);
                const int y = (int)((long long)total * (wid + 1) / NW);
                if (x >= y) continue;
                int q = 0, above = nlist;   // the run that holds window x
                while (above - q > 1) {
                    const int m = (q + above) >> 1;
                    if (S.win[m] <= x) q = m; else above = m;
                }
                for (int x0 = x; x0 < y; x0 += 32) {   // 32 windows
                    const int xl = x0 + lane;
                    if (q + 1 < nlist && S.win[q + 1] <= x0) ++q;   // the run of window x0
                    int j = q, ln = 0;   // the run of this lane's window: a run has at least one, so below q + 32
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (j + step < nlist && S.win[j + step] <= xl) j += step;
                    if (xl < y) {
                        const int o = (xl - S.win[j]) * 32;
                        ln = min(32, S.len[j] - o);
                        S.wnd[lane] = make_int2(S.st[j] + o, ln);
                    } else {
                        S.wnd[lane] = make_int2(0, 0);
                    }
                    __syncwarp();
                    const int cnt = min(32, y - x0);
                    unsigned sum = 0;   // of the lane's window
                    for (int h0 = 0; h0 < cnt; h0 += U) {
                        // lanes past a window's end hold `none`, the entry of a counter that stays 0
                        unsigned c[U];
#pragma unroll
                        for (int h = 0; h < U; h += 2) {
                            const int4 d = *reinterpret_cast<const int4 *>(S.wnd + h0 + h);
                            c[h] = c[h + 1] = none;
                            if (lane < d.y) c[h] = (unsigned)__ldg(encl + d.x);
                            if (lane < d.w) c[h + 1] = (unsigned)__ldg(encl + d.z);
                        }
#pragma unroll
                        for (int h = 0; h < U; ++h) {
                            if (MID) {
                                const unsigned t = __reduce_add_sync(FULL, S.get(c[h]));
                                if (lane == h0 + h) sum = t;
                            } else if (c[h] != none) {
                                S.add(c[h]);
                            }
                        }
                    }
                    if (MID) {
                        sum -= (unsigned)ln;   // (32 counts of at most 65535; 32 such windows fit run_add too)
                        su += sum;
                        run_add(&vacc[S.v[j]].C4, j, sum);
                    }
                    q = __shfl_sync(FULL, j, 31);
                    __syncwarp();
                }
            }
            return any;
        };
        if (walk(std::false_type{})) *S.any = 1;   // 1. count
        __syncthreads();
        const bool live = *S.any != 0;
        if (live) {
            walk(std::true_type{});                // 2. middle vertices: c - 1 per wedge
            __syncthreads();
            if (threadIdx.x == 0) *S.any = 0;
            // 3. C(c, 2) to every key with c >= 2; clear
            const int gw0 = gi * words;
            ck_sweep<THREADS, 0>(S, vacc, gw0, lim_word & ~3, gw0 + words);
        }
        __syncthreads();
    }
    su = warp_sum(su);   // of all warps: sum of c - 1 over the wedges = twice the sum of C(c, 2) over the keys
    if (lane == 0 && su) add64(S.twice, su);
    __syncthreads();
    if (threadIdx.x == 0 && *S.twice) {
        add64(&vacc[u].C4, *S.twice / 2);
        *S.twice = 0;
    }
}

// The keys of zone 0 (degree 1024 and more) for a root u with so many
// in-neighbours that a count could pass 16 bits: 32-bit counters, `words` ids
// at a time, runs found by search, one warp per run. Such a root has 65535
// in-neighbours or more; a graph has few of them.
template <int THREADS>
__device__ __forceinline__ void c4_wide_top(const Graph &g, VAcc *vacc, int u, int words, const CkShared &S) {
    constexpr int NW = THREADS / 32;
    const int lane = lane_id(), wid = threadIdx.x >> 5;
    const int *__restrict__ col = g.ncol;
    const int4 ru = g.rinfo[u];
    unsigned *const cnt = reinterpret_cast<unsigned *>(S.cnt);
    long long su = 0;
    for (int lo = S.z[0].lo; lo < u; lo += words) {
        const int nk = min(words, u - lo);
        auto walk = [&](auto mid) {
            constexpr bool MID = decltype(mid)::value;
            for (int p0 = ru.x + 32 * wid; p0 < ru.y; p0 += 32 * NW) {
                const int v = p0 + lane < ru.y ? col[p0 + lane] : -1;
                int st = 0, ln = 0;
                if (v >= 0) {
                    const int4 rv = g.rinfo[v];
                    st = lower_bound(col, rv.x, rv.z, lo);
                    ln = lower_bound(col, st, rv.z, lo + nk) - st;
                }
                unsigned acc = 0;   // below W <= m
                for (unsigned m = __ballot_sync(FULL, ln > 0); m; m &= m - 1) {
                    const int j = __ffs(m) - 1, js = __shfl_sync(FULL, st, j), jl = __shfl_sync(FULL, ln, j);
                    unsigned a = 0;
                    for (int o = lane; o < jl; o += 32) {
                        const unsigned k = (unsigned)(__ldg(col + js + o) - lo);
                        if (k >= (unsigned)nk) continue;   // never, for sorted rows
                        if (MID) a += cnt[k] - 1u; else atomicAdd(&cnt[k], 1u);
                    }
                    if (MID) {
                        a = __reduce_add_sync(FULL, a);
                        if (lane == j) acc = a;
                    }
                }
                if (MID && acc) add64(&vacc[v].C4, acc);
            }
            __syncthreads();
        };
        walk(std::false_type{});
        walk(std::true_type{});
        for (int k = threadIdx.x; k < nk; k += THREADS) {
            const long long cc = c2((long long)cnt[k]);
            cnt[k] = 0;
            if (cc) add64(&vacc[lo + k].C4, cc);
            su += cc;
        }
        __syncthreads();
    }
    su = warp_sum(su);
    if (lane == 0 && su) add64(&vacc[u].C4, su);
}

// Roots from the work queue. Every access stays in range for any CSR with
// sorted rows or not: runs lie within their rows, and every entry of `enc` is
// a counter of the CTA.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 4 : 1)
    k_c4_tiled(Graph g, VAcc *vacc, const int *lists, int *counters, const int *coff, int ntiles, int words, int *region) {
    pdl_begin();
    extern __shared__ __align__(16) unsigned char dsm[];
    CkShared S;
    S.cnt = dsm;
    S.z = reinterpret_cast<CkZone *>(dsm + 4 * (size_t)words + 16);
    S.st = reinterpret_cast<int *>(S.z + CK_ZONES + 1);   // (16-byte aligned, like S.wnd)
    S.len = S.st + THREADS;
    S.win = S.len + THREADS;
    S.v = S.win + THREADS;
    S.wnd = reinterpret_cast<int2 *>(S.v + THREADS) + (threadIdx.x & ~31u);
    S.wwin = S.v + 3 * THREADS;
    S.wrun = S.wwin + THREADS / 32;
    S.any = S.wrun + THREADS / 32;
    S.job = S.any + 1;
    S.twice = reinterpret_cast<long long *>(S.any + 2);
    if (call_stopped(counters)) return;
    const int nt = counters[CNT_C4_TEAM];
    if (nt == 0) return;
    const int *sorted = lists;
    for (int i = threadIdx.x; i <= words / 4; i += THREADS) reinterpret_cast<uint4 *>(S.cnt)[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        ck_zones(coff, ntiles, g.n, S.z);
        *S.any = 0;
        *S.twice = 0;
    }
    __syncthreads();
    const CkPlan P = ck_plan(region, S.z, words, g.n, g.m);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) *S.job = atomicAdd(&counters[CNT_C4_TILED_NEXT], 1);
        __syncthreads();
        const int j = *S.job;
        if (j >= nt) break;
        const int u = sorted[j];
        const int4 ru = g.rinfo[u];
        const bool wide = ru.y - ru.x > CK_NARROW_MAXD;
        if (wide) c4_wide_top<THREADS>(g, vacc, u, words, S);
        c4_tiled_root<THREADS>(g, vacc, u, wide ? min(u, S.z[0].lo) : u, words, P, S);
    }
}

// Count bits of a packed table for ids below n: the key takes bits(n - 1).
static int packed_count_bits(int n) {
    unsigned top = n > 1 ? (unsigned)(n - 1) : 1u;
    int kb = 0;
    while (top) { ++kb; top >>= 1; }
    return 32 - kb;
}

void launch_cycle4(Work &w, cudaStream_t st) {
    // the wedge segments take the region of the triangle counts, dead after the aggregate stage
    int2 *wl = reinterpret_cast<int2 *>(w.tcnt);
    Graph g{w.n, w.m, w.rinfo, w.ncol, wl};
    int maxw = w.tune[TUNE_C4_WARP_MAXW] < CW_MAXW ? w.tune[TUNE_C4_WARP_MAXW] : CW_MAXW;
    // Batches of graphs of under 150 vertices on average: their roots have many
    // repeated keys and short walks, so all go to a warp's table at once (1756
    // graphs of 18 to 144 vertices: 315 us a call; 359 with the filter first;
    // 357 graphs of 18 to 180: 138, 160).
    const bool tiny = w.graphs > 1 && w.n / w.graphs < 150 && w.n > w.num_sms * 32;
    const bool filter = w.n > w.num_sms * 32 && !tiny;
    // Batches of random graphs in which the average root (d^2 / 3 wedges at
    // mean degree d, over the n / graphs keys of its graph) repeats eight keys
    // and more: the tables at once too. Larger single graphs of that kind are
    // better off with the filter, whose rule knows their size (us a call,
    // filter first / tables at once: 100 graphs G(700, 0.03), 15 repeats,
    // 408 / 377; 200 graphs G(300, 0.1), 150, 597 / 548; 1000 graphs
    // G(300, 0.05), 9, 943 / 932; 8192 power-law graphs, 0.2, 11966 / 13446;
    // one G(8000, mean degree 40), 18, 192 / 209).
    const double mean = (double)w.m / w.n;
    const bool repeats = w.graphs > 1 && mean * mean * mean * mean / 9 >= 2.0 * 8 * w.n / w.graphs;
    const int sample = filter && !repeats && w.m >= 12ll * w.n ? SAMPLE_CTAS : 0;
    launch_pdl((long long)w.m < 16ll * w.n ? k_c4_wedge_len<8> : k_c4_wedge_len<16>, w.num_sms * 8 + sample, 256, 0, st, g, wl,
               w.vacc, w.counters, w.coff, w.ntiles, sample, repeats ? C4_TABLES : C4_FILTER);
    after_launch(st, K_C4_WEDGE_LEN);
    const int cb = packed_count_bits(w.n);
    // a packed word holds counts up to 2^cb - 2; with many vertices (large
    // graphs, batches) that is below what the warp tier takes, and the warp
    // tier counts in split tables instead
    const bool packed = (1ll << cb) - 2 >= maxw;
    const int few = packed && w.n <= w.num_sms * 2048 ? C4_FEW_LEFT : 0;
    const int teamw = w.tune[TUNE_C4_TEAM_MINW];
    static const int occ_w = resident_ctas((const void *)k_c4_warp<false>, CW_WARPS * 32, 0);
    static const int occ_ws = resident_ctas((const void *)k_c4_warp<true>, CW_WARPS * 32, 0);
    static const int occ_l = resident_ctas((const void *)k_c4_warp_left<false>, CW_WARPS * 32, 0);
    static const int occ_ls = resident_ctas((const void *)k_c4_warp_left<true>, CW_WARPS * 32, 0);
    constexpr size_t CF_SMEM = CF_WARPS * sizeof(C4FilterSmem);
    static const int occ_f = resident_ctas((const void *)k_c4_filter<false>, CF_WARPS * 32, CF_SMEM);
    // More roots than resident warps: the filter first, then the table for
    // what it leaves. Below, every warp has one root, and nearly all (W above
    // CW_SMALL_MAXW) go to the 4-warp tier at once, where the slowest walk is
    // shorter: with the filter in front, G(400, mean degree 20) took 67 us a
    // call instead of 63, G(2000, 20) 75 instead of 71. From 16 vertices a
    // multiprocessor on the 4-warp tier has several roots for each of its CTAs,
    // and the line is higher (at 32 / 128 wedges: G(4800, 16) 104 / 99 us a
    // call, a ring of 4800 vertices of degree 16 with 10% rewired 111 / 100;
    // G(400, 20) 63 / 64, G(1000, 20) 67 / 68).
    if (filter) {
        launch_pdl(packed ? k_c4_filter<false> : k_c4_filter<true>, w.num_sms * min(w.tune[TUNE_GRID_C4], occ_f),
                   CF_WARPS * 32, CF_SMEM, st, g, w.vacc, w.lists, w.counters, maxw, cb, teamw, w.coff, w.ntiles);
        after_launch(st, K_C4_FILTER);
        launch_pdl(packed ? k_c4_warp_left<false> : k_c4_warp_left<true>, w.num_sms * (packed ? occ_l : occ_ls),
                   CW_WARPS * 32, 0, st, g, w.vacc, w.lists, w.counters, maxw, cb, few, teamw, w.coff, w.ntiles);
        after_launch(st, K_C4_WARP_LEFT);
    } else {
        launch_pdl(packed ? k_c4_warp<false> : k_c4_warp<true>,
                   w.num_sms * min(w.tune[TUNE_GRID_C4], packed ? occ_w : occ_ws), CW_WARPS * 32, 0, st, g, w.vacc, w.lists,
                   w.counters, tiny ? maxw : min(maxw, w.n > w.num_sms * 16 ? CW_FEW_MAXW : CW_SMALL_MAXW), cb, teamw,
                   w.coff, w.ntiles);
        after_launch(st, K_C4_WARP);
    }
    static const int occ_m = resident_ctas((const void *)k_c4_mid, CM_THREADS, CM_SMEM);
    static const int occ_c = resident_ctas((const void *)k_c4_cta, CC_THREADS, CC_SMEM);
    launch_pdl(k_c4_mid, w.num_sms * occ_m, CM_THREADS, CM_SMEM, st, g, w.vacc, w.lists, w.counters, cb);
    after_launch(st, K_C4_MID);
    // (a graph whose counters surely are one group has no root between the 128-thread tier and the key-tiled one)
    if (w.n / 2 + 4 * CK_ZONES > CK_WORDS) {
        launch_pdl(k_c4_cta, w.num_sms * occ_c, CC_THREADS, CC_SMEM, st, g, w.vacc, w.lists, w.counters, cb);
        after_launch(st, K_C4_CTA);
    }
    const bool small = w.n <= CK_SMALL_N;
    const int words = small ? (w.n / 2 + 4 * CK_ZONES + 4) & ~3 : CK_WORDS;
    launch_pdl(k_c4_tiled_plan, 1 + min(2 * w.num_sms, w.m / 4096 + 1), 1024, 0, st, g, w.lists, w.counters, w.coff, w.ntiles, words,
               w.tcnt, w.status);
    after_launch(st, K_C4_PLAN);
    if (small) {
        const size_t smem = ck_smem(256, words);
        const int occ = (int)min((size_t)4, (size_t)(227 * 1024) / (smem + 1024));
        launch_pdl(k_c4_tiled<256>, w.num_sms * occ, 256, smem, st, g, w.vacc, w.lists, w.counters, w.coff, w.ntiles, words,
                   w.tcnt);
    } else {
        launch_pdl(k_c4_tiled<1024>, w.num_sms, 1024, ck_smem(1024, words), st, g, w.vacc, w.lists, w.counters, w.coff,
                   w.ntiles, words, w.tcnt);
    }
    after_launch(st, K_C4_TILED);
}

void configure_cycle4() {
    // the warp tiers need nearly all of an SM's shared memory for full residency
    for (auto k : {(const void *)k_c4_warp<false>, (const void *)k_c4_warp<true>, (const void *)k_c4_warp_left<false>, (const void *)k_c4_warp_left<true>,
                   (const void *)k_c4_filter<false>, (const void *)k_c4_filter<true>})
        cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    cudaFuncSetAttribute(k_c4_mid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CM_SMEM);
    cudaFuncSetAttribute(k_c4_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CC_SMEM);
    cudaFuncSetAttribute(k_c4_tiled<256>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ck_smem(256, CK_SMALL_N / 2 + 64));
    cudaFuncSetAttribute(k_c4_tiled<256>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    cudaFuncSetAttribute(k_c4_tiled<1024>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    cudaFuncSetAttribute(k_c4_tiled<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ck_smem(1024, CK_WORDS));
}

}  // namespace niorca
