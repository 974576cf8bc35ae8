// lexbfs_csr.cu — LexBFS by partition refinement on CSR graphs (sparse), in
// panels of up to 32 pivots, one CTA per graph.
//
// Method: Section 4.2 (Habib, McConnell, Paul and Viennot's partition
// refinement): visit the first vertex x of the first class, then replace every
// class C by C ∩ N_x placed before C \ N_x.  Its O(N + M) form moves only the
// neighbours of x.
//
// One step at a time is a chain of dependent L2 loads (row, classes, links:
// 1.9 us per vertex on GB300 at 65,536 vertices and degree 21).  As in the dense
// search (lexbfs_dense.cuh) the next vertices in partition order depend only on
// the edges among them, so a panel takes up to 32 of them, the window:
//   1. the threads gather the window's rows, one entry each, and build every
//      neighbour's key (bit j = adjacent to window vertex j) in a hash table in
//      shared memory; the first to meet a neighbour lists it with its class;
//   2. the window's own keys give the visiting order (panel_in_order, or
//      panel_solve when few are visited in window order);
//   3. the neighbours met, sorted by (class, label, id), leave their classes:
//      each run of equal (class, label) becomes a new class, placed before the
//      old one.
//
// State.  A class is a segment of an arena of vertices, in id order; a member is
// live while cls[] still names the class, so leaving a class costs one store.
// New segments are cut from the arena's end; when it is full the live ones are
// packed (7 n entries, so a packing follows at least 5 n moves).  Classes are in
// a doubly linked list, top first; the next pointers of the first ids live in
// shared memory, because following them is the one serial chain left.  The
// class of the vertices without a numbered neighbour (id n) ends the list and
// is never stored: its members are the v with cls[v] = n, in id order.
// The first classes of the list are taken out of it ahead of time into the
// front, an array of up to 128 vertices in partition order in shared memory
// (warp 0 does that while the other warps gather the window's rows); classes in
// the front are split there.  A class too large for the front is entered 32
// members at a time; what a panel leaves of those goes back.
// Rows longer than the hash table takes (kMaxEntries) make a panel of one
// pivot, whose neighbours are sorted by (class, row position) in the workspace.
// parent[y]: the last pivot of the last panel that met y, p(y) of the
// perfect-elimination check (Section 5.2).
#include <algorithm>

#include "kernels.h"
#include "lexbfs_dense.cuh"

namespace cg {

namespace {

constexpr int kNumberedCls = -2;
constexpr int kFrontCls = -3;
constexpr int kHead = -4;              // predecessor of the first class
constexpr unsigned kFull = 0xFFFFFFFFu;

constexpr int kCsrArrays = 11;         // the state's size in blocks of n + 1 ints, without the long rows' arrays
constexpr int kCsrThreads = 1024;
constexpr int kMaxEntries = 2048;      // row entries of one panel
constexpr int kHashSize = 4096;        // at least kMaxEntries + 2 kFrontCap
constexpr int kFrontCap = 128;
constexpr int kFrontLow = 64;          // the front is filled up to this many vertices beyond the window
constexpr int kNextSmem = 30 * 1024;   // next pointers kept in shared memory
constexpr int kScanStop = 128;         // a scan that has found a member looks at this many more slots

// State in the workspace.
struct CsrState {
    CG_ARR(int) cls;                        // [n] class of each vertex (n: no numbered neighbour yet)
    CG_ARR(int) cnext;                      // [n] next class, ids >= next_smem
    CG_ARR(int4) rec;                       // [n + 1] per class: segment start, end, live members, previous class
    CG_ARR(int) freel;                      // [n] free class ids
    CG_ARR(int) subid;                      // [n] long row: new class by sorted index
    CG_ARR(unsigned long long) skey;        // [next pow2 >= n] long row: (class << 32 | row position)
    CG_ARR(int) arena;                      // [cap]
    unsigned cap;
};

__host__ __device__ inline int64_t pow2_at_least(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

__device__ inline CsrState csr_state_carve(int *base, int64_t n, int64_t max_deg) {
    CsrState s;
    int *p = base;
    const int64_t stride = ((n + 1 + 31) / 32) * 32;
    const int64_t md = max_deg > 1 ? max_deg : 1, ds = ((md + 31) / 32) * 32;
    s.rec = cg_arr(reinterpret_cast<int4 *>(p), n + 1, kChkCsrRec); p += 4 * stride;   // 16-byte aligned
    s.skey = cg_arr(reinterpret_cast<unsigned long long *>(p), pow2_at_least(md), kChkCsrSkey);
    p += 2 * pow2_at_least(md);
    s.cls = cg_arr(p, n, kChkCsrCls); p += stride;
    s.cnext = cg_arr(p, n, kChkCsrNext); p += stride;
    s.freel = cg_arr(p, n, kChkCsrFree); p += stride;
    s.subid = cg_arr(p, n, kChkCsrSub); p += stride;
    const int64_t cap = (kCsrArrays - 8) * stride + 4 * ds;
    s.cap = (unsigned)(cap < 0xFFFFFFFFll ? cap : 0xFFFFFFFFll);
    s.arena = cg_arr(p, s.cap, kChkCsrArena);
    return s;
}

__host__ inline size_t csr_state_stride_bytes(int64_t n, int64_t max_deg) {
    const int64_t stride = ((n + 1 + 31) / 32) * 32;
    const int64_t ds = ((std::max<int64_t>(max_deg, 1) + 31) / 32) * 32;
    return (size_t)(kCsrArrays * stride + 4 * ds) * sizeof(int) +
           (size_t)pow2_at_least(std::max<int64_t>(max_deg, 1)) * sizeof(unsigned long long);
}

struct Front {                         // vertices in partition order
    int64_t beg[kFrontCap];            // row
    int deg[kFrontCap];
    int v[kFrontCap];
    int par[kFrontCap];                // last pivot that met it
};

struct CsrShared {
    unsigned long long key[kMaxEntries];    // moved vertices: class << 32 | inverted label
    unsigned long long key2[kMaxEntries];   // listed: class << 32 | hash slot; then moved, sorted
    int y[kMaxEntries];
    int y2[kMaxEntries];
    int sub[kMaxEntries];                   // new class by sorted index
    int hkey[kHashSize];                    // vertex (-1: free)
    uint32_t hmask[kHashSize];              // its key
    uint8_t hfront[kHashSize];              // it came to the front in this panel
    Front front[2];
    int fslot[kFrontCap];                   // hash slot
    unsigned fat[kFrontCap];                // slot in the arena (large class in the front)
    uint32_t fck[kFrontCap];                // inverted label of this panel
    uint32_t nck[kFrontCap];                // the same and the old class's start, by new position
    int ncs[kFrontCap];
    uint32_t fstart[kFrontCap / 32];        // bit p: a class starts at p
    int flen;
    int pcls, pmore;                        // the front is a part of this class (-1: whole classes); there is more of it
    int head_next;                          // first class of the list
    int free_top;
    int unl_size, unl_cur;                  // vertices without a numbered neighbour: how many, none below this id
    unsigned atop;                          // end of the arena's used part
    int lcount, m;
    int r;
    uint32_t pivmask;
    uint32_t ub;
    int piv[32];
    uint32_t bit[32];
    uint32_t tab[8][16];
    int scan[32];
    int next[1];                            // [next_smem]
};

__global__ void csr_init_kernel(int *ws, int64_t n, int64_t max_deg, int32_t *parent) {
    CsrState s = csr_state_carve(ws, n, max_deg);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        s.cls[v] = (int)n;
        s.freel[v] = (int)(n - 1 - v);   // taken from the end: low ids first
        if (parent) parent[v] = -1;
        if (v == 0) s.rec[n] = make_int4(0, 0, 0, kHead);
    }
}

// Sorts key[0..p), p > tile_n a power of two, in global memory (bitonic, all
// threads of the CTA): the passes with a stride below tile_n pair keys inside one aligned tile of tile_n keys, so they
// run on a shared-memory copy of each tile (the first log2 of them for every k
// up to the tile size, the rest after each k's global passes).
__device__ void cta_sort_keys_tiled(unsigned long long *key, int64_t p, unsigned long long *tile, int tile_n) {
    const int T = blockDim.x;
    auto tile_passes = [&](int64_t t0, int64_t k_lo, int64_t k_hi, int64_t j_first) {
        for (int li = threadIdx.x; li < tile_n; li += T) tile[li] = key[t0 + li];
        __syncthreads();
        for (int64_t k = k_lo; k <= k_hi; k <<= 1) {
            for (int64_t j = (k == k_lo ? j_first : (k >> 1)); j > 0; j >>= 1) {
                for (int li = threadIdx.x; li < tile_n; li += T) {
                    const int l = li ^ (int)j;
                    if (l > li) {
                        const unsigned long long a = tile[li], b = tile[l];
                        if ((a > b) == (((t0 + li) & k) == 0)) {
                            tile[li] = b;
                            tile[l] = a;
                        }
                    }
                }
                __syncthreads();
            }
        }
        for (int li = threadIdx.x; li < tile_n; li += T) key[t0 + li] = tile[li];
        __syncthreads();
    };
    for (int64_t t0 = 0; t0 < p; t0 += tile_n) tile_passes(t0, 2, tile_n, 1);   // k = 2 .. tile size
    for (int64_t k = 2 * (int64_t)tile_n; k <= p; k <<= 1) {
        for (int64_t j = k >> 1; j >= tile_n; j >>= 1) {
            for (int64_t i = threadIdx.x; i < p; i += T) {
                const int64_t l = i ^ j;
                if (l > i) {
                    const unsigned long long a = key[i], b = key[l];
                    if ((a > b) == ((i & k) == 0)) {
                        key[i] = b;
                        key[l] = a;
                    }
                }
            }
            __syncthreads();
        }
        for (int64_t t0 = 0; t0 < p; t0 += tile_n) tile_passes(t0, k, k, tile_n >> 1);
    }
}

struct CsrGraph {
    int n;
    int next_smem;                          // classes whose next pointer is in shared memory
    const int64_t *__restrict__ row_ptr;
    const int32_t *__restrict__ col;
    int32_t *parent;
};

__device__ __forceinline__ int get_next(const CsrState &s, const CsrShared *sh, const CsrGraph &g, int c) {
    return c < g.next_smem ? sh->next[c] : s.cnext[c];
}
__device__ __forceinline__ void set_next(const CsrState &s, CsrShared *sh, const CsrGraph &g, int c, int to) {
    if (c == kHead) sh->head_next = to;
    else if (c < g.next_smem) sh->next[c] = to;
    else s.cnext[c] = to;
}

// y's slot of the hash table, taken if it was not there.  At most kMaxEntries +
// 2 kFrontCap vertices meet the table's kHashSize slots, so a free one is found.
__device__ __forceinline__ int hash_slot(CsrShared *sh, int y, bool *fresh) {
    unsigned h = ((unsigned)y * 2654435761u) >> 20;   // 12 bits: kHashSize
    *fresh = false;
    for (int k = 0; k < kHashSize; ++k) {
        const int old = atomicCAS(&sh->hkey[h], -1, y);
        if (old == -1) *fresh = true;
        if (old == -1 || old == y) break;
        h = (h + 1) & (kHashSize - 1);
    }
    return (int)h;
}

__device__ __forceinline__ int warp_inclusive(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// The lane whose share of a row of shares contains item e (incl: the lanes'
// inclusive sums; 31 when e is beyond all of them).
__device__ __forceinline__ int warp_owner(unsigned incl, unsigned e) {
    int p = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
        if (__shfl_sync(kFull, incl, p + st - 1) <= e) p += st;
    return p;
}

// Puts v at position p of the front.
__device__ __forceinline__ void front_put(CsrShared *sh, Front *f, const CsrGraph &g, int p, int v, int par) {
    const int64_t b = g.row_ptr[v], e = g.row_ptr[v + 1];
    f->v[p] = v;
    f->par[p] = par;
    f->beg[p] = b;
    f->deg[p] = (int)(e - b);
}

// Warp 0: takes the next classes of the list into the front f, which holds
// `have` vertices, until `want` more are in it; an empty front takes up to 32
// members of a class that does not fit.
__device__ void front_fill(const CsrState &s, CsrShared *sh, const CsrGraph &g, Front *f, int have, int want) {
    const int lane = threadIdx.x & 31;
    const int room = kFrontCap - have;
    const int top = sh->head_next;
    int len = have, pcls = -1, pmore = 0;
    int4 r0 = make_int4(sh->unl_cur, g.n, sh->unl_size, 0);
    if (top != g.n) {
        // the next classes' ids: lane k the k-th
        int id = top, mine = g.n, cnt = 0, after = g.n;
        const int lim = min(32, want);
        for (; cnt < lim && id != g.n; ++cnt) {
            if (lane == cnt) mine = id;
            id = get_next(s, sh, g, id);
        }
        after = id;
        const int4 rc = lane < cnt ? s.rec[mine] : make_int4(0, 0, 0, 0);
        const int sz = min(rc.z, kFrontCap + 1), incl = warp_inclusive(sz);
        const bool take = lane < cnt && incl <= room && incl - sz < want;
        const int ntake = __popc(__ballot_sync(kFull, take));   // a prefix of the lanes
        if (ntake > 0) {
            const unsigned len_k = take ? (unsigned)rc.y - (unsigned)rc.x : 0u;
            unsigned slots = len_k;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned u = __shfl_up_sync(kFull, slots, o);
                if (lane >= o) slots += u;
            }
            const unsigned total = __shfl_sync(kFull, slots, 31);
            constexpr int U = 2;
            for (unsigned b = 0; b < total; b += 32 * U) {
                int v[U], own[U], pv[U];
                bool live[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned e = b + 32 * u + lane;
                    own[u] = warp_owner(slots, e);
                    const unsigned at = (unsigned)__shfl_sync(kFull, rc.x, own[u]) + e -
                                        __shfl_sync(kFull, slots - len_k, own[u]);
                    v[u] = e < total ? s.arena[at] : -1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int c = __shfl_sync(kFull, mine, own[u]);
                    live[u] = v[u] >= 0 && s.cls[v[u]] == c;
                    pv[u] = live[u] && g.parent ? g.parent[v[u]] : -1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int first = have + __shfl_sync(kFull, incl - sz, own[u]);
                    const unsigned lm = __ballot_sync(kFull, live[u]);
                    const int p = len + __popc(lm & lanes_below(lane));
                    if (live[u] && p < kFrontCap) {
                        front_put(sh, f, g, p, v[u], pv[u]);
                        s.cls[v[u]] = kFrontCls;
                        if (p == first) atomicOr(&sh->fstart[p >> 5], 1u << (p & 31));
                        bool fresh;
                        const int h = hash_slot(sh, v[u], &fresh);
                        sh->fslot[p] = h;
                        sh->hfront[h] = 1;
                    }
                    len = min(len + __popc(lm), kFrontCap);
                }
            }
            const int nx = ntake < cnt ? __shfl_sync(kFull, mine, ntake) : after;
            if (take) s.freel[sh->free_top + lane] = mine;
            __syncwarp();
            if (lane == 0) {
                sh->free_top += ntake;
                sh->head_next = nx;
                s.rec[nx].w = kHead;
                sh->flen = len;
                sh->pcls = -1;
            }
            __syncwarp();
            return;
        }
        if (have > 0) return;
        r0.x = __shfl_sync(kFull, rc.x, 0);
        r0.y = __shfl_sync(kFull, rc.y, 0);
        r0.z = __shfl_sync(kFull, rc.z, 0);
    }
    if (have > 0 || r0.z <= 0) return;
    // the first members of class `top`, which stays in the list
    constexpr int U = 4;
    unsigned found_at = 0u;
    const unsigned end = (unsigned)r0.y;
    for (unsigned b = (unsigned)r0.x; b < end && len < 32; b += 32 * U) {
        if (len > 0 && b - found_at >= (unsigned)kScanStop) break;
        int v[U];
        bool live[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned e = b + 32 * u + lane;
            v[u] = e < end ? (top == g.n ? (int)e : s.arena[e]) : -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) live[u] = v[u] >= 0 && s.cls[v[u]] == top;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const unsigned lm = __ballot_sync(kFull, live[u]);
            const int p = len + __popc(lm & lanes_below(lane));
            if (live[u] && p < 32) {
                front_put(sh, f, g, p, v[u], g.parent ? g.parent[v[u]] : -1);
                s.cls[v[u]] = kFrontCls;
                sh->fat[p] = b + 32 * u + lane;
            }
            if (len == 0 && lm) found_at = b;
            len = min(len + __popc(lm), 32);
        }
    }
    pcls = top;
    pmore = r0.z > len;
    if (lane == 0) {
        sh->flen = len;
        sh->pcls = pcls;
        sh->pmore = pmore;
        sh->fstart[0] = 1u;
    }
    __syncwarp();
}

// Packs the arena's live segments (all threads).
__device__ void arena_pack(const CsrState &s, CsrShared *sh, const CsrGraph &g) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const unsigned top = sh->atop;
    unsigned out = 0u;
    for (unsigned b = 0; b < top; b += kCsrThreads) {
        const unsigned a = b + t;
        int v = -1;
        if (a < top) {
            v = s.arena[a];
            const int c = s.cls[v];
            bool live = c >= 0 && c < g.n;
            if (live) {
                const int4 rc = s.rec[c];
                live = (unsigned)rc.x <= a && a < (unsigned)rc.y;
            }
            if (!live) v = -1;
        }
        const unsigned lm = __ballot_sync(kFull, v >= 0);
        if (lane == 0) sh->scan[warp] = __popc(lm);
        __syncthreads();   // the chunk is read before it is written
        const int wc = sh->scan[lane];
        const int before = __reduce_add_sync(kFull, lane < warp ? wc : 0), all = __reduce_add_sync(kFull, wc);
        if (v >= 0) s.arena[out + before + __popc(lm & lanes_below(lane))] = v;
        out += all;
        __syncthreads();
    }
    for (unsigned a = t; a < out; a += kCsrThreads) {
        const int c = s.cls[s.arena[a]];
        const int cp = a > 0 ? s.cls[s.arena[a - 1]] : -1;
        if (c != cp) {
            s.rec[c].x = (int)a;
            if (cp >= 0) s.rec[cp].y = (int)a;
        }
        if (a + 1 == out) s.rec[c].y = (int)out;
    }
    if (t == 0) sh->atop = out;
    __syncthreads();
}

// Sorted moved vertices, of a panel (shared memory) or of a long row (workspace).
template <bool LONG>
struct Moved {
    const unsigned long long *key;
    const int *y;
    const int32_t *row;
    int m;
    // equal for members of one new class, the old class in the high half
    __device__ __forceinline__ unsigned long long group(int k) const { return LONG ? key[k] >> 32 << 32 : key[k]; }
    __device__ __forceinline__ int cls(int k) const { return (int)(key[k] >> 32); }
    __device__ __forceinline__ int vertex(int k) const { return LONG ? row[key[k] & 0xFFFFFFFFu] : y[k]; }
    // the first index after k / the first index at or before k of the run of equal `what`
    template <typename F>
    __device__ __forceinline__ int run_end(int k, F what) const {
        const auto x = what(k);
        int lo = k, st = 1;   // lo is in the run
        while (lo + st < m && what(lo + st) == x) lo += st, st *= 2;
        for (; st > 0; st >>= 1)
            if (lo + st < m && what(lo + st) == x) lo += st;
        return lo + 1;
    }
    template <typename F>
    __device__ __forceinline__ int run_start(int k, F what) const {
        const auto x = what(k);
        int hi = k, st = 1;
        while (hi - st >= 0 && what(hi - st) == x) hi -= st, st *= 2;
        for (; st > 0; st >>= 1)
            if (hi - st >= 0 && what(hi - st) == x) hi -= st;
        return hi;
    }
};

// The moved vertices into their new classes: ids and the list's outer links,
// then segments, members and inner links.  The last new class of a class that
// moved whole keeps its id, place and links.
template <bool LONG>
__device__ __forceinline__ void move_ids(const CsrState &s, CsrShared *sh, const CsrGraph &g, const Moved<LONG> &mv,
                                         int *sub) {
    auto grp = [&](int k) { return mv.group(k); };
    auto cl = [&](int k) { return mv.cls(k); };
    for (int k = threadIdx.x; k < mv.m; k += kCsrThreads) {
        if (k > 0 && mv.group(k - 1) == mv.group(k)) continue;
        const int c = mv.cls(k);
        const bool first = k == 0 || mv.cls(k - 1) != c;
        const int4 rc = s.rec[c];
        const int e = mv.run_end(k, grp);
        const bool last = e >= mv.m || mv.cls(e) != c;
        int id = -1;
        if (last) {
            const int mc = e - mv.run_start(k, cl);
            if (c == g.n) sh->unl_size -= mc;
            else if (mc == rc.z) id = c;
            else s.rec[c].z = rc.z - mc;
        }
        if (id < 0) id = s.freel[atomicSub(&sh->free_top, 1) - 1];
        sub[k] = id;
        if (first && id != c) {
            s.rec[id].w = rc.w;
            set_next(s, sh, g, rc.w, id);
        }
    }
}
template <bool LONG>
__device__ __forceinline__ void move_members(const CsrState &s, CsrShared *sh, const CsrGraph &g,
                                             const Moved<LONG> &mv, const int *sub) {
    auto grp = [&](int k) { return mv.group(k); };
    const unsigned base = sh->atop;
    for (int k = threadIdx.x; k < mv.m; k += kCsrThreads) {
        const int sf = mv.run_start(k, grp), id = sub[sf], y = mv.vertex(k);
        s.arena[base + k] = y;
        s.cls[y] = id;
        if (g.parent) g.parent[y] = sh->piv[LONG ? 0 : 32 - __ffs(~(uint32_t)mv.key[k])];
        if (k != sf) continue;
        const int c = mv.cls(k), e = mv.run_end(k, grp);
        const bool last = e >= mv.m || mv.cls(e) != c;
        s.rec[id].x = (int)(base + k);
        s.rec[id].y = (int)(base + e);
        s.rec[id].z = e - k;
        if (id != c) {   // (the kept id is the class's last)
            const int nid = last ? c : sub[e];
            set_next(s, sh, g, id, nid);
            s.rec[nid].w = id;
        }
    }
}

__global__ void __launch_bounds__(kCsrThreads) lexbfs_csr_kernel(int *ws, int64_t max_deg, CsrGraph g, int64_t nnz,
                                                                 int32_t *__restrict__ order, int32_t *__restrict__ pos) {
    extern __shared__ __align__(16) unsigned char smem[];
    CsrShared *sh = reinterpret_cast<CsrShared *>(smem);
    const int n = g.n, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const CsrState s = csr_state_carve(ws, n, max_deg);
    // Every row is read once, when its vertex is in a window, so its first read
    // would be a DRAM miss: pull row_ptr and col into L2 (bulk prefetch, no
    // completion wait) while the search starts.
    prefetch_range_l2<kCsrThreads>(g.row_ptr, (size_t)(n + 1) * sizeof(int64_t));
    prefetch_range_l2<kCsrThreads>(g.col, (size_t)nnz * sizeof(int32_t));
    auto clear_hash = [&]() {
        for (int k = t; k < kHashSize; k += kCsrThreads) {
            sh->hkey[k] = -1;
            sh->hmask[k] = 0u;
            sh->hfront[k] = 0;
        }
    };
    clear_hash();
    if (t < kFrontCap / 32) sh->fstart[t] = 0u;
    if (t == 0) {
        sh->flen = 0;
        sh->pcls = -1;
        sh->pmore = 0;
        sh->head_next = n;
        sh->free_top = n;
        sh->unl_size = n;
        sh->unl_cur = 0;
        sh->atop = 0u;
        sh->lcount = 0;
        sh->m = 0;
        sh->ub = 0u;
    }
    __syncthreads();

    int i = 0;     // numbered vertices
    int cur = 0;   // the front at hand
    const int fp = t - (kCsrThreads - kFrontCap);   // the last threads: position in the front
    while (i < n) {
        Front *f = &sh->front[cur], *nf = &sh->front[cur ^ 1];
        if (sh->flen == 0) {
            __syncthreads();
            if (warp == 0) front_fill(s, sh, g, f, 0, kFrontLow);
            __syncthreads();
            if (sh->flen == 0) break;   // not on a well-formed graph
        }
        int fl = sh->flen;
        int pcls = sh->pcls;
        // ---- the window: as many of the front's first 32 as kMaxEntries row entries allow
        const int wmax = min(32, fl);
        const int64_t beg = lane < wmax ? f->beg[lane] : 0;
        const int deg = lane < wmax ? f->deg[lane] : 0;
        const int vk = lane < wmax ? f->v[lane] : 0;
        const unsigned einc = (unsigned)warp_inclusive(min(deg, kMaxEntries + 1));
        int w2 = __popc(__ballot_sync(kFull, lane < wmax && einc <= (unsigned)kMaxEntries));
        const bool long_row = w2 == 0;
        if (long_row) w2 = 1;
        const int entries = long_row ? 0 : (int)__shfl_sync(kFull, einc, w2 - 1);
        __syncthreads();   // everyone has read the front's length

        uint32_t adj = 0u;
        if (!long_row) {
            if (warp == 0) {
                if (pcls < 0 && fl - w2 < kFrontLow && sh->head_next != n)
                    front_fill(s, sh, g, f, fl, kFrontLow + w2 - fl);
            } else {
                if (fp >= 0 && fp < fl) {
                    bool fresh;
                    sh->fslot[fp] = hash_slot(sh, f->v[fp], &fresh);
                }
                constexpr int U = (kMaxEntries + kCsrThreads - 33) / (kCsrThreads - 32);
                constexpr int kStep = kCsrThreads - 32;
                int y[U], c[U], own[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int e = t - 32 + u * kStep;
                    y[u] = -1;
                    own[u] = 0;
                    if (e - lane < entries) {
                        own[u] = warp_owner(einc, (unsigned)e);
                        const int64_t at = __shfl_sync(kFull, beg, own[u]) +
                                           (e - (int)__shfl_sync(kFull, einc - (unsigned)deg, own[u]));
                        if (e < entries) y[u] = g.col[at];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) c[u] = y[u] >= 0 ? s.cls[y[u]] : kNumberedCls;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (t - 32 - lane + u * kStep >= entries) break;
                    bool list = false;
                    int h = 0;
                    if (c[u] != kNumberedCls) {
                        bool fresh;
                        h = hash_slot(sh, y[u], &fresh);
                        atomicOr(&sh->hmask[h], 1u << own[u]);
                        list = fresh && c[u] >= 0;
                    }
                    const unsigned lm = __ballot_sync(kFull, list);
                    int at = 0;
                    if (lane == 0 && lm) at = atomicAdd(&sh->lcount, __popc(lm));
                    at = __shfl_sync(kFull, at, 0) + __popc(lm & lanes_below(lane));
                    if (list && at < kMaxEntries) {
                        sh->key2[at] = (unsigned long long)(unsigned)c[u] << 32 | (unsigned)h;
                        sh->y2[at] = y[u];
                    }
                }
            }
            __syncthreads();
            fl = sh->flen;
            adj = lane < w2 ? sh->hmask[sh->fslot[lane]] & ~(1u << lane) : 0u;
        } else if (pcls >= 0) {   // a long row in a large class: the others go back
            if (fp >= 1 && fp < fl) s.cls[f->v[fp]] = pcls;
            __syncthreads();
            if (t == 0) {
                sh->pmore = sh->pmore || fl > 1;
                sh->flen = 1;
            }
            __syncthreads();
            fl = 1;
        }
        // key of the front's vertex p (long row: searched in the pivot's row)
        auto front_key = [&](int p) -> uint32_t {
            if (!long_row) return sh->hmask[sh->fslot[p]];
            const int32_t *row = g.col + f->beg[0];
            const int v = f->v[p];
            int lo = 0, hi = f->deg[0];
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (row[mid] < v) lo = mid + 1; else hi = mid;
            }
            return lo < f->deg[0] && row[lo] == v ? 1u : 0u;
        };

        // ---- the pivots: window vertices 0..r-1 in order, or what warp 0 finds
        const uint32_t starts = sh->fstart[0] & low_bits(w2);
        const bool outside = pcls >= 0 && sh->pmore;   // members of the window's class beyond the front
        const bool straddle = w2 < fl ? w2 == 32 ? !(sh->fstart[1] & 1u) : !((sh->fstart[0] >> w2) & 1u) : outside;
        uint32_t ub = 0u;
        if (straddle && !long_row) {
            if (outside) ub = kFull;
            else {   // the class's members in the front beyond the window
                int ce = fl;
                for (int w = w2 >> 5; w < kFrontCap / 32 && 32 * w < ce; ++w) {
                    const uint32_t b = sh->fstart[w] & (w == (w2 >> 5) ? kFull << (w2 & 31) : kFull);
                    if (b) ce = min(ce, 32 * w + __ffs(b) - 1);
                }
                for (int p = w2 + lane; p < ce; p += 32) ub |= sh->hmask[sh->fslot[p]];
                ub = __reduce_or_sync(kFull, ub);
            }
        }
        int mypos = -1, la = -1;   // warp 0
        bool order_fails = false;
        int r = long_row ? 1 : panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
        bool ident = true;
        if (r < w2 && r < kPanelFew) {   // too few (the same in every warp)
            if (!order_fails && outside) {
                __syncthreads();
                uint32_t any = 0u;
                for (int k = t; k < sh->lcount; k += kCsrThreads)
                    if ((int)(sh->key2[k] >> 32) == pcls) any |= sh->hmask[(unsigned)sh->key2[k]];
                if (fp >= w2 && fp < fl) any |= sh->hmask[sh->fslot[fp]];
                any = __reduce_or_sync(kFull, any);
                if (lane == 0 && any) atomicOr(&sh->ub, any);
                __syncthreads();
                ub = sh->ub;
                r = panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
            }
            ident = !(order_fails && r < kPanelFew);
        }
        uint32_t pm = low_bits(r);
        if (warp == 0) {
            if (ident) {
                mypos = lane < r ? lane : -1;
                const uint32_t before = adj & lanes_below(lane);
                la = before ? 31 - __clz(before) : -1;
            } else {
                r = panel_solve(lane, w2, starts, straddle, adj, ub, &mypos, &la);
            }
            const uint32_t taken = __ballot_sync(kFull, mypos >= 0);
            if (mypos >= 0) sh->piv[mypos] = vk;
            sh->bit[lane] = mypos >= 0 ? 0x80000000u >> mypos : 0u;
            __syncwarp();
            if (mypos >= 0) {
                order[i + mypos] = vk;
                if (pos) pos[vk] = i + mypos;
                if (g.parent) g.parent[vk] = la >= 0 ? sh->piv[la] : f->par[lane];
                s.cls[vk] = kNumberedCls;
            }
            if (lane == 0) {
                sh->r = r;
                sh->pivmask = taken;
                if (pcls >= 0) {   // the large class loses the pivots from its head
                    const int left = __ffs(~taken) - 1;   // -1: none of 32
                    const unsigned to = left >= 0 && left < fl ? sh->fat[left] : sh->fat[fl - 1] + 1u;
                    if (pcls == n) {
                        sh->unl_size -= r;
                        sh->unl_cur = (int)to;
                    } else {
                        const int sz = s.rec[pcls].z - r;
                        s.rec[pcls].z = sz;
                        s.rec[pcls].x = (int)to;
                        if (sz == 0) {
                            const int nx = get_next(s, sh, g, pcls);
                            sh->head_next = nx;
                            s.rec[nx].w = kHead;
                            s.freel[sh->free_top++] = pcls;
                        }
                    }
                }
            }
        }
        if (!ident) {
            __syncthreads();
            r = sh->r;
            pm = sh->pivmask;
            if (t < 128) {
                uint32_t v = 0u;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if ((t >> b) & 1) v |= sh->bit[((t >> 4) << 2) + b];
                sh->tab[t >> 4][t & 15] = v;
            }
            __syncthreads();
        }
        // a key's bits in pivot order, the first pivot's highest
        auto pivot_key = [&](uint32_t k) -> uint32_t {
            if (ident) return __brev(k);
            uint32_t v = 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) v |= sh->tab[b][(k >> (4 * b)) & 15u];
            return v;
        };

        // ---- the moved vertices of the listed classes; the front's labels
        auto append = [&](bool keep, int c, uint32_t pk, int y) {
            const unsigned lm = __ballot_sync(kFull, keep);
            int at = 0;
            if (lane == 0 && lm) at = atomicAdd(&sh->m, __popc(lm));
            at = __shfl_sync(kFull, at, 0) + __popc(lm & lanes_below(lane));
            if (keep && at < kMaxEntries) {
                sh->key[at] = (unsigned long long)(unsigned)c << 32 | (unsigned)~pk;
                sh->y[at] = y;
            }
        };
        if (!long_row) {
            const int lc = sh->lcount;
            for (int k0 = warp * 32; k0 < lc; k0 += kCsrThreads) {
                const int k = k0 + lane;
                unsigned long long e = 0ull;
                uint32_t mk = 0u;
                if (k < lc) {
                    e = sh->key2[k];
                    if (!sh->hfront[(unsigned)e]) mk = sh->hmask[(unsigned)e] & pm;
                }
                append(mk != 0u, (int)(e >> 32), pivot_key(mk), k < lc ? sh->y2[k] : 0);
            }
        }
        if (fp >= lane) {   // the front's warps
            const bool left = fp < fl && !(fp < 32 && ((pm >> fp) & 1u));
            uint32_t k = left ? front_key(fp) & pm : 0u;
            if (pcls >= 0) {   // the rest of a large class goes back (a long row left none)
                if (left && k == 0u) s.cls[f->v[fp]] = pcls;
                append(k != 0u, pcls, pivot_key(k), left ? f->v[fp] : 0);
            } else if (left) {
                const uint32_t pk = pivot_key(k);
                sh->fck[fp] = ~pk;
                if (k) f->par[fp] = ident ? f->v[31 - __clz(k)] : sh->piv[32 - __ffs(pk)];
            }
        }
        if (long_row) {
            const int64_t rb = f->beg[0];
            const int d = f->deg[0];
            const int64_t p2 = pow2_at_least(d);
            __syncthreads();   // the pivot's cls
            for (int64_t k = t; k < p2; k += kCsrThreads) {
                unsigned long long e = ~0ull;
                if (k < d) {
                    const int c = s.cls[g.col[rb + k]];
                    if (c >= 0) e = (unsigned long long)(unsigned)c << 32 | (unsigned long long)k;
                }
                s.skey[k] = e;
                const unsigned lm = __ballot_sync(kFull, e != ~0ull);   // p2 is a multiple of the CTA
                if (lm && lane == 0) atomicAdd(&sh->m, __popc(lm));
            }
        }
        __syncthreads();
        const int m = sh->m;

        // ---- sorted by (class, label, id)
        const unsigned long long *skey = sh->key2;
        const int *sy = sh->y2;
        if (long_row) {
            cta_sort_keys_tiled(s.skey, pow2_at_least(f->deg[0]), sh->key, kMaxEntries);   // deg > kMaxEntries
        } else if (m <= 512) {   // ranks by counting, as many lanes per vertex as there are
            const int lg = m <= 32 ? 5 : m <= 64 ? 4 : m <= 128 ? 3 : m <= 256 ? 2 : 1;
            const int e = t >> lg, step = 1 << lg;
            if ((warp * 32) >> lg < m) {
                const unsigned long long ke = e < m ? sh->key[e] : 0ull;
                const int ye = e < m ? sh->y[e] : 0;
                int rank = 0;
#pragma unroll 4
                for (int k = t & (step - 1); k < m; k += step) {
                    const unsigned long long kk = sh->key[k];
                    rank += kk < ke || (kk == ke && sh->y[k] < ye) ? 1 : 0;
                }
                for (int o = 1; o < step; o <<= 1) rank += __shfl_xor_sync(kFull, rank, o);
                if (e < m && (t & (step - 1)) == 0) {
                    sh->key2[rank] = ke;
                    sh->y2[rank] = ye;
                }
            }
        } else {
            int p2 = 1024;
            if (m > 1024) p2 = 2048;
            for (int e = m + t; e < p2; e += kCsrThreads) {
                sh->key[e] = ~0ull;
                sh->y[e] = 0;
            }
            __syncthreads();
            for (int k = 2; k <= p2; k <<= 1)
                for (int j = k >> 1; j > 0; j >>= 1) {
                    const int e = t;
                    if (e < p2 / 2) {
                        const int lo = ((e & ~(j - 1)) << 1) | (e & (j - 1)), hi = lo | j;
                        const unsigned long long a = sh->key[lo], b = sh->key[hi];
                        const int ya = sh->y[lo], yb = sh->y[hi];
                        if ((a > b || (a == b && ya > yb)) == ((lo & k) == 0)) {
                            sh->key[lo] = b;
                            sh->key[hi] = a;
                            sh->y[lo] = yb;
                            sh->y[hi] = ya;
                        }
                    }
                    __syncthreads();
                }
            skey = sh->key;
            sy = sh->y;
        }
        // ---- the front after the panel: each class's members by label
        const int fl2 = pcls >= 0 ? 0 : fl - r;
        if (pcls < 0 && fp >= 0 && fp < fl && !(fp < 32 && ((pm >> fp) & 1u))) {
            int cs = 0, ce = fl;
            for (int w = fp >> 5; w >= 0; --w) {
                const uint32_t b = sh->fstart[w] & (w == (fp >> 5) ? low_bits((fp & 31) + 1) : kFull);
                if (b) {
                    cs = 32 * w + 31 - __clz(b);
                    break;
                }
            }
            for (int w = fp >> 5; w < kFrontCap / 32; ++w) {
                const uint32_t b = sh->fstart[w] & (w == (fp >> 5) ? 0xFFFFFFFEu << (fp & 31) : kFull);
                if (b) {
                    ce = min(ce, 32 * w + __ffs(b) - 1);
                    break;
                }
            }
            int np = cs - __popc(pm & low_bits(cs));
            const uint32_t ck = sh->fck[fp];
            for (int q = cs; q < ce; ++q) {
                if (q < 32 && ((pm >> q) & 1u)) continue;
                const uint32_t cq = sh->fck[q];
                np += cq < ck || (cq == ck && q < fp) ? 1 : 0;
            }
            nf->v[np] = f->v[fp];
            nf->par[np] = f->par[fp];
            nf->beg[np] = f->beg[fp];
            nf->deg[np] = f->deg[fp];
            sh->nck[np] = ck;
            sh->ncs[np] = cs;
        }
        __syncthreads();

        // ---- new classes
        if (fp >= lane) {
            const bool st = fp < fl2 &&
                            (fp == 0 || sh->ncs[fp] != sh->ncs[fp - 1] || sh->nck[fp] != sh->nck[fp - 1]);
            const uint32_t b = __ballot_sync(kFull, st);
            if (lane == 0) sh->fstart[fp >> 5] = b;
        }
        // nothing in the list but vertices that had no numbered neighbour: what the panel met goes to the front
        const bool to_front = !long_row && m > 0 && fl2 + m <= kFrontCap && sh->head_next == n;
        const Moved<false> mv{skey, sy, nullptr, m};
        const Moved<true> ml{s.skey, nullptr, g.col + f->beg[0], m};
        if (!to_front) {
            if (long_row) move_ids(s, sh, g, ml, (int *)s.subid);
            else move_ids(s, sh, g, mv, sh->sub);
        }
        clear_hash();
        __syncthreads();
        if (to_front) {
            if (t < m) {
                const int p = fl2 + t, y = sy[t];
                front_put(sh, nf, g, p, y, sh->piv[32 - __ffs(~(uint32_t)skey[t])]);
                s.cls[y] = kFrontCls;
                if (t == 0 || skey[t] != skey[t - 1]) atomicOr(&sh->fstart[p >> 5], 1u << (p & 31));
            }
        } else if (m > 0) {
            if (s.cap - sh->atop < (unsigned)m) arena_pack(s, sh, g);   // the same for all threads
            if (long_row) move_members(s, sh, g, ml, (int *)s.subid);
            else move_members(s, sh, g, mv, sh->sub);
        }
        __syncthreads();
        if (t == 0) {
            sh->flen = fl2 + (to_front ? m : 0);
            sh->pcls = -1;
            sh->pmore = 0;
            if (to_front) sh->unl_size -= m;
            else sh->atop += (unsigned)m;
            sh->lcount = 0;
            sh->m = 0;
            sh->ub = 0u;
        }
        i += r;
        cur ^= 1;
        __syncthreads();
    }
}

}  // namespace

size_t lexbfs_csr_workspace_bytes(int64_t n, int64_t max_deg) { return csr_state_stride_bytes(n, max_deg) + 256; }

int lexbfs_csr_launch(int n, int64_t max_deg, const int64_t *row_ptr, const int32_t *col, int64_t nnz, int32_t *order,
                      int32_t *pos, int32_t *parent, void *ws, int num_sms, cudaStream_t stream) {
    if (n <= 0) return CG_OK;
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), (int64_t)num_sms * 4));
    csr_init_kernel<<<blocks, 256, 0, stream>>>(static_cast<int *>(ws), n, max_deg, parent);
    CG_LAUNCH_CHECK("csr_init_kernel");
    static_assert(sizeof(CsrShared) + kNextSmem * sizeof(int) <= 227 * 1024, "shared memory of one CTA");
    const CsrGraph g{n, std::min(n, kNextSmem), row_ptr, col, parent};
    const size_t smem = sizeof(CsrShared) + (size_t)g.next_smem * sizeof(int);
    CG_CUDA_TRY(cudaFuncSetAttribute(lexbfs_csr_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    lexbfs_csr_kernel<<<1, kCsrThreads, smem, stream>>>(static_cast<int *>(ws), max_deg, g, nnz, order, pos);
    CG_LAUNCH_CHECK("lexbfs_csr_kernel");
    CG_DEBUG_CHECK(stream, "lexbfs_csr_kernel");
    return CG_OK;
}

}  // namespace cg
