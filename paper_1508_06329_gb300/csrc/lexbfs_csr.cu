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
// On narrow graphs (paths, matchings, small components, interval graphs of small
// degree) the next vertex is known only after the one before, and a window numbers
// two to ten.  When the windows do not pay, the front goes back to the list and warp
// 0 takes pivots one by one, a lane per vertex that has met one (csr_steps); windows
// are tried again from time to time.
//
// State.  A class is a segment of an arena of vertices, in id order; a member is
// live while cls[] still names the class, so leaving a class costs one store.
// New segments are cut from the arena's end; when it is full the live ones are
// packed (3 n entries and 4 for every one of the longest row, so a packing
// follows at least 2 n moves).  Classes are in
// a doubly linked list, top first; the next pointers of the first ids live in
// shared memory, because following them is the one serial chain left.  The
// class of the vertices without a numbered neighbour (id n) ends the list and
// is never stored: its members are the v with cls[v] = n, in id order.
// The first classes of the list are taken out of it ahead of time into the
// front, an array of up to 128 vertices in partition order in shared memory
// (warp 0 does that while the other warps, the workers, gather, order and sort);
// classes in the front are split there.  A class too large for the front is entered 32
// members at a time; what a panel leaves of those goes back.
// Rows longer than the hash table takes (kMaxEntries) make a panel of one
// pivot, whose neighbours are sorted by (class, row position) in the workspace;
// those without a numbered neighbour need no sort.
// parent[y]: the last pivot of the last panel that met y, p(y) of the
// perfect-elimination check (Section 5.2).
//
// Measured on GB300 (whole test, one step per vertex -> panels): 65,536 vertices
// of degree 21 120.5 -> 25.7 ms, 262,143 506 -> 122 ms, 5,000 8.0 -> 2.8 ms, 20,000
// of degree 5 28.0 -> 8.5 ms.  A panel of 30 pivots takes about 12 us: gathering
// 2, the order 1.7, sorting 3, new classes 4.5, the front and barriers the rest;
// all of it latency (barriers, dependent loads from L2, instruction fetch).
// Narrow, 65,536 vertices (windows alone in brackets): path 91 -> 53 ms (279),
// matching 74 -> 40 (308), disjoint K4 70 -> 42 (164), K10 66 -> 51 (70), random
// of degree 1 70 -> 37 (135).
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
// 65,536 / 5,000 vertices of degree 21: 26.4 / 2.8 ms with 1,024 threads, 27.9 / 3.6 with 512, 33.8 / 5.5 with 256
constexpr int kCsrThreads = 1024;
constexpr int kCsrWorkers = kCsrThreads - 32;   // all but warp 0, which fills the front
constexpr int kMaxEntries = 2048;      // row entries of one panel
constexpr int kHashSize = 4096;        // at least kMaxEntries + kFrontCap
constexpr int kFrontCap = 128;
constexpr int kFrontLow = 64;          // the front is filled up to this many vertices beyond the window
constexpr int kNextSmem = 30 * 1024;   // next pointers kept in shared memory
// Windows give way to steps when they have numbered this many vertices less than kStepsBelow each: a window's panel
// costs 8 to 12 us, a step 0.65 to 0.9.
constexpr int kCsrStepsLost = 36;
constexpr int kScanStop = 128;                // a scan that has found a member looks at this many more slots

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
#pragma unroll 1
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
    // (a long row's digit counts lie in the first two arrays)
    unsigned long long key[kMaxEntries];    // moved vertices: class << 32 | inverted label
    unsigned long long key2[kMaxEntries];   // listed: class << 32 | hash slot; then moved, sorted
    int hkey[kHashSize];                    // vertex (-1: free)
    uint32_t hmask[kHashSize];              // its key
    int y[kMaxEntries];
    int y2[kMaxEntries];
    int sub[kMaxEntries];                   // new class by sorted index
    uint32_t gstart[kMaxEntries / 32];      // bit k: the sorted index k is the first of its new class
    uint32_t cstart[kMaxEntries / 32];      // and of its old class
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
    int unl_id;                             // long row: the new class of the vertices without a numbered neighbour
    int next[1];                            // [next_smem]
};

__global__ void csr_init_kernel(int *ws, int64_t n, int64_t max_deg, int32_t *parent) {
    CsrState s = csr_state_carve(ws, n, max_deg);
#pragma unroll 1
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        s.cls[v] = (int)n;
        s.freel[v] = (int)(n - 1 - v);   // taken from the end: low ids first
        if (parent) parent[v] = -1;
        if (v == 0) s.rec[n] = make_int4(0, 0, 0, kHead);
    }
}

// Sorts the moved vertices key/y[0..m) by (key, y) into key2/y2, m <= kMaxEntries:
// every warp sorts 32 in registers, then a vertex's rank is its place in its run
// plus the vertices before it in every other run, found by bisection, two runs
// at a time.  (About 300 are moved on the sparse chordal graphs: 15,000 cycles by
// comparing all with all.)  One barrier of the workers; the caller has the ones
// around.
__device__ void panel_sort_moved(CsrShared *sh, int m) {
    constexpr int T = kCsrWorkers;
    const int t = threadIdx.x - 32, lane = t & 31, warp = warp_index() - 1;
    const int runs = (m + 31) >> 5;
#pragma unroll 1
    for (int b = warp; b < runs; b += T / 32) {
        const int e = 32 * b + lane;
        unsigned long long k = e < m ? sh->key[e] : ~0ull;
        int y = e < m ? sh->y[e] : 0x7FFFFFFF;
#pragma unroll 1
        for (int s = 2; s <= 32; s <<= 1)
#pragma unroll 1
            for (int j = s >> 1; j > 0; j >>= 1) {
                const unsigned long long ok = __shfl_xor_sync(kFull, k, j);
                const int oy = __shfl_xor_sync(kFull, y, j);
                const bool greater = k > ok || (k == ok && y > oy);
                if (greater == (((lane & s) == 0) == ((lane & j) == 0))) {
                    k = ok;
                    y = oy;
                }
            }
        sh->key[e] = k;
        sh->y[e] = y;
    }
    named_barrier(1, kCsrWorkers);
    int lg = 4;   // lanes per vertex
    while (lg > 0 && (32 * runs << lg) > T) --lg;
    const int step = 1 << lg;
#pragma unroll 1
    for (int e = t >> lg; e < 32 * runs; e += T) {   // whole warps: a warp's elements are of one run
        const unsigned long long k = sh->key[e];
        const int y = sh->y[e], own = e >> 5;
        int rank = 0;
#pragma unroll 1
        for (int b0 = t & (step - 1); b0 < runs; b0 += 2 * step) {
            int lo[2] = {0, 0};
            auto before = [&](int b, int i) {   // element i of run b is before this one
                const unsigned long long x = sh->key[32 * b + i];
                return x < k || (x == k && sh->y[32 * b + i] < y);
            };
#pragma unroll
            for (int st = 16; st > 0; st >>= 1)
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (before(min(b0 + u * step, runs - 1), lo[u] + st - 1)) lo[u] += st;
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int b = b0 + u * step;
                if (b < runs && b != own) rank += lo[u] + (before(b, lo[u]) ? 1 : 0);
            }
        }
#pragma unroll 1
        for (int o = 1; o < step; o <<= 1) rank += __shfl_xor_sync(kFull, rank, o);
        rank += e & 31;
        if ((t & (step - 1)) == 0 && rank < m) {
            sh->key2[rank] = k;
            sh->y2[rank] = y;
        }
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
// kFrontCap vertices meet the table's kHashSize slots, so a free one is found.
__device__ __forceinline__ int hash_slot(CsrShared *sh, int y, bool *fresh) {
    unsigned h = ((unsigned)y * 2654435761u) >> 20;   // 12 bits: kHashSize
    *fresh = false;
#pragma unroll 1
    for (int k = 0; k < kHashSize; ++k) {
        const int old = atomicCAS(&sh->hkey[h], -1, y);
        if (old == -1) *fresh = true;
        if (old == -1 || old == y) break;
        h = (h + 1) & (kHashSize - 1);
    }
    return (int)h;
}

// y's key, 0 when it is not in the table.
__device__ __forceinline__ uint32_t hash_key(const CsrShared *sh, int y) {
    unsigned h = ((unsigned)y * 2654435761u) >> 20;
#pragma unroll 1
    for (int k = 0; k < kHashSize; ++k) {
        const int x = sh->hkey[h];
        if (x == y) return sh->hmask[h];
        if (x == -1) break;
        h = (h + 1) & (kHashSize - 1);
    }
    return 0u;
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

// A long row's vertices in the order of (class, row position): kept[k] is the
// class of the row's k-th vertex (-1: none of them), m how many there are.  A
// radix sort by class, eight bits a pass, each warp over its own part of the
// row, between the buffers b1 and b2; returns the one with the result, keys
// (class << 32 | row position).  (25,000 vertices: 15,000 cycles; a bitonic
// network on 8,192 keys at a time in shared memory took 500,000.)
__device__ const unsigned long long *sort_long_row(CsrShared *sh, const int *kept, int d, int m, int n,
                                                   unsigned long long *b1, unsigned long long *b2) {
    constexpr int NW = kCsrThreads / 32;
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    uint32_t(*hist)[256] = reinterpret_cast<uint32_t(*)[256]>(sh->key);   // [NW][256]: key and key2
    unsigned long long *src = b2, *dst = b1;
#pragma unroll 1
    for (int shift = 0; shift == 0 || (shift < 32 && ((n - 1) >> shift) > 0); shift += 8) {
        const int len = shift ? m : d, part = (len + kCsrThreads - 1) / kCsrThreads * 32;
        const int lo = min(warp * part, len), hi = min(lo + part, len);
        auto load = [&](int k) -> unsigned long long {   // ~0: none
            if (k >= hi) return ~0ull;
            if (shift) return src[k];
            const int c = kept[k];
            return c < 0 ? ~0ull : (unsigned long long)(unsigned)c << 32 | (unsigned)k;
        };
        auto digit = [&](unsigned long long x) -> unsigned {
            return x == ~0ull ? 256u : (unsigned)(x >> (32 + shift)) & 255u;
        };
        for (int k = t; k < NW * 256; k += kCsrThreads) hist[k >> 8][k & 255] = 0u;
        __syncthreads();
        unsigned long long ahead = load(lo + lane);
#pragma unroll 1
        for (int k0 = lo; k0 < hi; k0 += 32) {
            const unsigned g = digit(ahead);
            ahead = load(k0 + 32 + lane);
            const uint32_t same = __match_any_sync(kFull, g);
            if (g < 256u && (same & lanes_below(lane)) == 0u) hist[warp][g] += __popc(same);
            __syncwarp();
        }
        __syncthreads();
        // where each warp's share of each digit begins: thread t sums warps [w0, w0 + PER) of one digit
        constexpr int PER = NW * 256 / kCsrThreads;
        const int g = t / (NW / PER), w0 = t % (NW / PER) * PER;
        int mine = 0;
        for (int w = 0; w < PER; ++w) mine += hist[w0 + w][g];
        const int incl = warp_inclusive(mine);
        if (lane == 31) sh->scan[warp] = incl;
        __syncthreads();
        const int wc = lane < NW ? sh->scan[lane] : 0;
        int at = __reduce_add_sync(kFull, lane < warp ? wc : 0) + incl - mine;
        for (int w = 0; w < PER; ++w) {
            const int x = hist[w0 + w][g];
            hist[w0 + w][g] = at;
            at += x;
        }
        __syncthreads();
        ahead = load(lo + lane);
#pragma unroll 1
        for (int k0 = lo; k0 < hi; k0 += 32) {
            const unsigned long long x = ahead;
            const unsigned h = digit(x);
            ahead = load(k0 + 32 + lane);
            const uint32_t same = __match_any_sync(kFull, h), below = same & lanes_below(lane);
            const uint32_t base = h < 256u ? hist[warp][h] : 0u;
            __syncwarp();
            if (h < 256u) {
                dst[base + __popc(below)] = x;
                if (below == 0u) hist[warp][h] = base + __popc(same);
            }
            __syncwarp();
        }
        __syncthreads();
        unsigned long long *const u = src;
        src = dst;
        dst = u;
    }
    return src;
}

// Puts v, whose row is col[b, e), at position p of the front.
__device__ __forceinline__ void front_put(Front *f, int p, int v, int par, int64_t b, int64_t e) {
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
#pragma unroll 1
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
            constexpr int U = 4;   // slots per lane at once, so that their loads overlap
#pragma unroll 1
            for (unsigned b = 0; b < total; b += 32 * U) {
                int v[U], own[U], c[U], pv[U];
                int64_t rb[U], re[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned e = b + 32 * u + lane;
                    own[u] = warp_owner(slots, e);
                    const unsigned at = (unsigned)__shfl_sync(kFull, rc.x, own[u]) + e -
                                        __shfl_sync(kFull, slots - len_k, own[u]);
                    v[u] = e < total ? s.arena[at] : -1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {   // (also for slots whose vertex has left)
                    const int x = max(v[u], 0);
                    c[u] = v[u] >= 0 ? s.cls[x] : kNumberedCls;
                    rb[u] = g.row_ptr[x];
                    re[u] = g.row_ptr[x + 1];
                    pv[u] = g.parent ? g.parent[x] : -1;
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (b + 32 * u >= total) break;
                    const bool live = c[u] == __shfl_sync(kFull, mine, own[u]);
                    const int first = have + __shfl_sync(kFull, incl - sz, own[u]);
                    const unsigned lm = __ballot_sync(kFull, live);
                    const int p = len + __popc(lm & lanes_below(lane));
                    if (live && p < kFrontCap) {
                        front_put(f, p, v[u], pv[u], rb[u], re[u]);
                        s.cls[v[u]] = kFrontCls;
                        if (p == first) atomicOr(&sh->fstart[p >> 5], 1u << (p & 31));
                    }
                    len = min(len + __popc(lm), kFrontCap);
                }
            }
            const int nx = ntake < cnt ? __shfl_sync(kFull, mine, ntake) : after;
            if (take) {
                s.freel[sh->free_top + lane] = mine;
                s.rec[mine].z = -1;   // what the panel lists of it stays in the front
            }
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
#pragma unroll 1
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
                front_put(f, p, v[u], g.parent ? g.parent[v[u]] : -1, g.row_ptr[v[u]], g.row_ptr[v[u] + 1]);
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
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    const unsigned top = sh->atop;
    unsigned out = 0u;
#pragma unroll 1
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
        const int wc = lane < kCsrThreads / 32 ? sh->scan[lane] : 0;
        const int before = __reduce_add_sync(kFull, lane < warp ? wc : 0), all = __reduce_add_sync(kFull, wc);
        if (v >= 0) s.arena[out + before + __popc(lm & lanes_below(lane))] = v;
        out += all;
        __syncthreads();
    }
#pragma unroll 1
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

// Sorted moved vertices: of a panel, in shared memory with the first indices of
// the new and the old classes as masks, or of a long row, in the workspace (all
// members of an old class make one new class).
template <bool LONG>
struct Moved {
    const CsrShared *sh;
    const unsigned long long *key;
    const int32_t *row;
    int m;
    const uint32_t *bits;   // long row: bit k: k is the first of its class (null: not kept)
    const int *last;        // and the last of these up to the end of a word
    __device__ __forceinline__ int cls(int k) const { return (int)(key[k] >> 32); }
    __device__ __forceinline__ int vertex(int k) const { return LONG ? row[key[k] & 0xFFFFFFFFu] : sh->y2[k]; }
    __device__ __forceinline__ bool first(int k) const {   // of its old class
        if (LONG && !bits) return k == 0 || cls(k - 1) != cls(k);
        return ((LONG ? bits : sh->cstart)[k >> 5] >> (k & 31)) & 1u;
    }
    __device__ __forceinline__ bool group_first(int k) const {   // of its new class
        return LONG ? first(k) : (sh->gstart[k >> 5] >> (k & 31)) & 1u;
    }
    // the first index of k's new class; of its old one; the first index after its new one
    __device__ __forceinline__ int group_start(int k) const { return LONG ? key_start(k) : bit_at_or_before(sh->gstart, k); }
    __device__ __forceinline__ int class_start(int k) const { return LONG ? key_start(k) : bit_at_or_before(sh->cstart, k); }
    __device__ __forceinline__ int group_end(int k) const {
        if (LONG && bits) {   // the first word beyond k's with another last start
            int w = k >> 5, hi = (m - 1) >> 5;
            const uint32_t b = bits[w] & (0xFFFFFFFEu << (k & 31));
            if (b) return 32 * w + __ffs(b) - 1;
            const int own = last[w];
            if (last[hi] == own) return m;
#pragma unroll 1
            while (hi - w > 1) {
                const int mid = (w + hi) >> 1;
                if (last[mid] == own) w = mid; else hi = mid;
            }
            return 32 * hi + __ffs(bits[hi]) - 1;
        }
        if (LONG) {
            const int c = cls(k);
            int lo = k, st = 1;   // lo is in the class
#pragma unroll 1
            while (lo + st < m && cls(lo + st) == c) lo += st, st *= 2;
#pragma unroll 1
            for (; st > 0; st >>= 1)
                if (lo + st < m && cls(lo + st) == c) lo += st;
            return lo + 1;
        }
        int w = k >> 5;
        uint32_t b = sh->gstart[w] & (0xFFFFFFFEu << (k & 31));
#pragma unroll 1
        while (!b && 32 * ++w < m) b = sh->gstart[w];
        return b ? 32 * w + __ffs(b) - 1 : m;
    }
    __device__ __forceinline__ int key_start(int k) const {
        if (bits) {   // (bit 0 is set)
            const uint32_t b = bits[k >> 5] & low_bits((k & 31) + 1);
            return b ? (k & ~31) + 31 - __clz(b) : last[(k >> 5) - 1];
        }
        const int c = cls(k);
        int hi = k, st = 1;
#pragma unroll 1
        while (hi - st >= 0 && cls(hi - st) == c) hi -= st, st *= 2;
#pragma unroll 1
        for (; st > 0; st >>= 1)
            if (hi - st >= 0 && cls(hi - st) == c) hi -= st;
        return hi;
    }
    __device__ __forceinline__ int bit_at_or_before(const uint32_t *bits, int k) const {   // (bit 0 is set)
        int w = k >> 5;
        uint32_t b = bits[w] & low_bits((k & 31) + 1);
#pragma unroll 1
        while (!b && w > 0) b = bits[--w];
        return 32 * w + 31 - __clz(b);
    }
};

// The moved vertices into their new classes: ids and the list's outer links,
// then segments, members and inner links.  The last new class of a class that
// moved whole keeps its id, place and links.
template <bool LONG>
__device__ __forceinline__ void move_ids(const CsrState &s, CsrShared *sh, const CsrGraph &g, const Moved<LONG> &mv,
                                         int *sub) {
#pragma unroll 1
    for (int k = threadIdx.x; k < mv.m; k += kCsrThreads) {
        if (!mv.group_first(k)) continue;
        const int c = mv.cls(k);
        const bool first = mv.first(k);
        const int4 rc = s.rec[c];
        if (rc.z < 0) {   // the class came to the front in this panel
            sub[k] = -1;
            continue;
        }
        const int e = mv.group_end(k);
        const bool last = e >= mv.m || mv.first(e);
        int id = -1;
        if (last) {
            const int mc = e - mv.class_start(k);
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
                                             const Moved<LONG> &mv, const int *sub, unsigned base) {
#pragma unroll 1
    for (int k = threadIdx.x; k < mv.m; k += kCsrThreads) {
        const int sf = mv.group_start(k), id = sub[sf], y = mv.vertex(k);
        s.arena[base + k] = y;
        if (id < 0) continue;
        s.cls[y] = id;
        if (g.parent) g.parent[y] = sh->piv[LONG ? 0 : 32 - __ffs(~(uint32_t)mv.key[k])];
        if (k != sf) continue;
        const int c = mv.cls(k), e = mv.group_end(k);
        const bool last = e >= mv.m || mv.first(e);
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

// The front's classes go back to the head of the list (warp 0).
__device__ void front_to_list(const CsrState &s, CsrShared *sh, const CsrGraph &g, const Front *f) {
    const int lane = threadIdx.x & 31, fl = sh->flen;
    const int head = sh->head_next, ftop = sh->free_top;
    const unsigned atop = sh->atop;
    __syncwarp();
    int before = 0;   // classes that start in the masks' earlier words
#pragma unroll 1
    for (int p0 = 0; p0 < fl; p0 += 32) {
        const int p = p0 + lane;
        const uint32_t starts = sh->fstart[p0 >> 5] & low_bits(fl - p0);
        const int k = before + __popc(starts & low_bits(lane + 1)) - 1;
        if (p < fl) {
            const int id = s.freel[ftop - 1 - k], v = f->v[p];
            s.arena[atop + p] = v;
            s.cls[v] = id;
            if (g.parent) g.parent[v] = f->par[p];
            if ((starts >> lane) & 1u) {
                int e = fl;   // the next class's start
#pragma unroll 1
                for (int w = p0 >> 5; 32 * w < fl; ++w) {
                    const uint32_t b = sh->fstart[w] & (w == (p0 >> 5) ? 0xFFFFFFFEu << lane : kFull);
                    if (b) {
                        e = min(e, 32 * w + __ffs(b) - 1);
                        break;
                    }
                }
                const int next = e < fl ? s.freel[ftop - 2 - k] : head;
                s.rec[id] = make_int4((int)(atop + p), (int)(atop + e), e - p, k > 0 ? s.freel[ftop - k] : kHead);
                set_next(s, sh, g, id, next);
                if (e == fl) s.rec[head].w = id;
                if (k == 0) sh->head_next = id;
            }
        }
        before += __popc(starts);
        __syncwarp();
    }
    if (lane == 0) {
        sh->free_top = ftop - before;
        sh->atop = atop + (unsigned)fl;
        sh->flen = 0;
    }
    if (lane < kFrontCap / 32) sh->fstart[lane] = 0u;
    __syncwarp();
}

// Panels of up to 32 pivots one by one, by warp 0 alone, on the list (the front is
// empty): for narrow graphs, whose next vertices the window does not hold.  A lane
// per vertex that has met a pivot and is not numbered yet: its class, its label in
// this panel, its row.  A step reads the pivot's row (at most 32 entries) and the
// classes and rows of the neighbours (two dependent L2 loads); the next pivot is
// the lane of the class at hand with the largest label, or that class's first
// member that has not been met.  At the panel's end the lanes move to their new
// classes as after a window.  Ends early before a pivot with a longer row or one
// that meets more vertices than lanes are free.  Leaves the number of pivots in sh->r.
__device__ void csr_steps(const CsrState &s, CsrShared *sh, const CsrGraph &g, int i, int32_t *__restrict__ order,
                          int32_t *__restrict__ pos, int panels) {
    const int n = g.n, lane = threadIdx.x & 31;
    int total = 0;
    bool stop = false;
#pragma unroll 1
    for (; panels > 0 && !stop && i + total < n && s.cap - sh->atop >= 32u; --panels) {
        int y = -1, cy = -1, dy = 0;    // the lane's vertex, its class, its row
        int64_t by = 0;
        uint32_t ky = 0u;               // its label in pivot order, the first pivot highest
        int c = sh->head_next, z = 0;   // the class at hand, its live members
        unsigned q = 0u, end = 0u;      // its slots from q on
        int mv = -1, md = 0;            // the lane's member in q .. q + 31 (live, not met when it was looked at), its row
        int64_t mb = 0;
        auto members = [&]() {
            const unsigned e = q + lane;
            mv = e < end ? (c == n ? (int)e : s.arena[e]) : -1;
            const int x = max(mv, 0);
            const int cl = s.cls[x];
            mb = g.row_ptr[x];
            md = (int)(g.row_ptr[x + 1] - mb);
            if (cl != c) mv = -1;
        };
        auto enter = [&]() {
            const int4 rc = c == n ? make_int4(sh->unl_cur, n, sh->unl_size, 0) : s.rec[c];
            q = (unsigned)rc.x;
            end = (unsigned)rc.y;
            z = rc.z;
            members();
        };
        auto leave = [&]() {   // the class at hand is used up
            const int nx = get_next(s, sh, g, c);
            __syncwarp();
            if (lane == 0) {
                s.freel[sh->free_top++] = c;
                sh->head_next = nx;
                s.rec[nx].w = kHead;
            }
            __syncwarp();
            c = nx;
        };
        enter();
        int r = 0;
#pragma unroll 1
        for (;;) {
            // ---- the next pivot
            int x = -1, deg = 0;
            int64_t beg = 0;
            uint32_t label;
#pragma unroll 1
            for (;;) {
                label = __reduce_max_sync(kFull, y >= 0 && cy == c ? ky : 0u);
                if (label) {
                    x = (int)__reduce_min_sync(kFull, y >= 0 && cy == c && ky == label ? (unsigned)y : kNoVertex);
                    const int l = __ffs(__ballot_sync(kFull, y == x)) - 1;
                    beg = __shfl_sync(kFull, by, l);
                    deg = __shfl_sync(kFull, dy, l);
                    break;
                }
                uint32_t ok = z > 0 ? __ballot_sync(kFull, mv >= 0) : 0u;
#pragma unroll 1
                while (ok) {
                    const int l = __ffs(ok) - 1, v = __shfl_sync(kFull, mv, l);
                    if (!__ballot_sync(kFull, y == v)) {
                        x = v;
                        beg = __shfl_sync(kFull, mb, l);
                        deg = __shfl_sync(kFull, md, l);
                        break;
                    }
                    if (lane == l) mv = -1;   // met
                    ok &= ok - 1u;
                }
                if (ok) break;
                if (z > 0 && q + 32 < end) {
                    q += 32;
                    members();
                    continue;
                }
                if (c == n) break;   // (not on a well-formed graph)
                leave();
                enter();
            }
            // ---- its row
            if (x < 0 || deg > 32) {
                stop = true;
                break;
            }
            const int w = lane < deg ? g.col[beg + lane] : -1, wx = max(w, 0);
            const int cw = s.cls[wx];
            const int64_t bw = g.row_ptr[wx];
            const int dw = (int)(g.row_ptr[wx + 1] - bw);
            bool adj = false, known = w < 0;
#pragma unroll 1
            for (int k = 0; k < deg; ++k) {
                const bool is = y == __shfl_sync(kFull, w, k);
                adj |= is;
                if (__ballot_sync(kFull, is) && lane == k) known = true;
            }
            const bool fresh = !known && cw != kNumberedCls && w != x;
            const uint32_t met = __ballot_sync(kFull, fresh), room = __ballot_sync(kFull, y < 0 || y == x);
            if (__popc(met) > __popc(room)) {
                stop = true;
                break;
            }
            if (lane == 0) {
                sh->piv[r] = x;
                sh->scan[r] = label ? sh->piv[32 - __ffs((int)label)] : -2;   // (-2: what met it before this panel)
                s.cls[x] = kNumberedCls;
            }
            if (y == x) y = -1;
            if (mv == x) mv = -1;
            --z;
            const uint32_t bit = 0x80000000u >> r;
            if (y >= 0 && adj) ky |= bit;
            if (fresh) {
                const int k = __popc(met & lanes_below(lane));
                sh->y[k] = w;
                sh->sub[k] = cw;
                sh->key[k] = (unsigned long long)bw;
                sh->key2[k] = (unsigned long long)(unsigned)dw;
            }
            __syncwarp();
            const int k = __popc(room & lanes_below(lane));
            if (((room >> lane) & 1u) && k < __popc(met)) {
                y = sh->y[k];
                cy = sh->sub[k];
                by = (int64_t)sh->key[k];
                dy = (int)sh->key2[k];
                ky = bit;
            }
            __syncwarp();
            ++r;
            if (r == 32 || i + total + r == n) break;
        }
        // ---- what is left of the class at hand; the results
        if (c == n) {
            if (lane == 0) {
                sh->unl_cur = (int)q;
                sh->unl_size = z;
            }
        } else if (z == 0) {
            leave();
        } else if (lane == 0) {
            s.rec[c].x = (int)q;
            s.rec[c].z = z;
        }
        if (lane < r) {
            const int v = sh->piv[lane], p = sh->scan[lane];
            order[i + total + lane] = v;
            if (pos) pos[v] = i + total + lane;
            if (g.parent && p != -2) g.parent[v] = p;
        }
        __syncwarp();
        // ---- the vertices met, by (class, label, id), to their new classes
        const uint32_t on = __ballot_sync(kFull, y >= 0);
        const int m = __popc(on);
        if (m > 0) {
            const unsigned long long mine = (unsigned long long)(unsigned)cy << 32 | (unsigned)~ky;
            int rank = 0;
#pragma unroll 1
            for (uint32_t b = on; b; b &= b - 1u) {
                const int l = __ffs(b) - 1;
                const unsigned long long o = __shfl_sync(kFull, mine, l);
                const int oy = __shfl_sync(kFull, y, l);
                rank += o < mine || (o == mine && oy < y) ? 1 : 0;
            }
            if (y >= 0) {
                sh->key2[rank] = mine;
                sh->y2[rank] = y;
            }
            __syncwarp();
            const unsigned long long o = lane < m ? sh->key2[lane] : 0ull, po = lane > 0 && lane < m ? sh->key2[lane - 1] : 0ull;
            const uint32_t gb = __ballot_sync(kFull, lane < m && (lane == 0 || o != po));
            const uint32_t cb = __ballot_sync(kFull, lane < m && (lane == 0 || o >> 32 != po >> 32));
            if (lane == 0) {
                sh->gstart[0] = gb;
                sh->cstart[0] = cb;
            }
            __syncwarp();
            const Moved<false> moved{sh, sh->key2, nullptr, m, nullptr, nullptr};
            move_ids(s, sh, g, moved, sh->sub);
            __syncwarp();
            move_members(s, sh, g, moved, sh->sub, sh->atop);
            __syncwarp();
            if (lane == 0) sh->atop += (unsigned)m;
            __syncwarp();
        }
        total += r;
    }
    if (lane == 0) sh->r = total;
    __syncwarp();
}

__global__ void __launch_bounds__(kCsrThreads) lexbfs_csr_kernel(int *ws, int64_t max_deg, CsrGraph g, int64_t nnz,
                                                                 int32_t *__restrict__ order, int32_t *__restrict__ pos) {
    extern __shared__ __align__(16) unsigned char smem[];
    CsrShared *sh = reinterpret_cast<CsrShared *>(smem);
    const int n = g.n, t = threadIdx.x, lane = t & 31, warp = warp_index();
    const CsrState s = csr_state_carve(ws, n, max_deg);
    // Every row is read once, when its vertex is in a window, so its first read
    // would be a DRAM miss: pull row_ptr and col into L2 (bulk prefetch, no
    // completion wait) while the search starts.
    prefetch_range_l2<kCsrThreads>(g.row_ptr, (size_t)(n + 1) * sizeof(int64_t));
    prefetch_range_l2<kCsrThreads>(g.col, (size_t)nnz * sizeof(int32_t));
    auto clear_hash = [&]() {
#pragma unroll 1
        for (int k = t; k < kHashSize; k += kCsrThreads) {
            sh->hkey[k] = -1;
            sh->hmask[k] = 0u;
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
    const bool front_warp = warp >= (kCsrThreads - kFrontCap) / 32;
    // pivots that windows have fallen short of kStepsBelow each; panels of steps that follow the next time
    int lost = 0, span = 1;
    while (i < n) {
        Front *f = &sh->front[cur], *nf = &sh->front[cur ^ 1];
        if (lost > kCsrStepsLost) {
            const bool pack = s.cap - sh->atop < (unsigned)(kFrontCap + 32 * span);
            __syncthreads();   // everyone has read the arena's end
            if (pack) arena_pack(s, sh, g);
            if (warp == 0) {
                const bool room = s.cap - sh->atop >= (unsigned)kFrontCap;
                __syncwarp();
                if (lane == 0) sh->r = 0;
                if (room) {
                    front_to_list(s, sh, g, f);
                    csr_steps(s, sh, g, i, order, pos, span);
                }
            }
            __syncthreads();
            const int r = sh->r;
            i += r;
            // the next window that does not pay is the last one, unless the steps did not pay either
            lost = r < kStepsBelow ? 0 : kCsrStepsLost;
            span = min(2 * span, kStepsMost);
            __syncthreads();
            continue;
        }
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

        // the classes' members in the front: [start, end) of the one at position p
        auto front_class = [&](int p, int *cs, int *ce, int len) {
            *cs = 0;
            *ce = len;
#pragma unroll 1
            for (int w = p >> 5; w >= 0; --w) {
                const uint32_t b = sh->fstart[w] & (w == (p >> 5) ? low_bits((p & 31) + 1) : kFull);
                if (b) {
                    *cs = 32 * w + 31 - __clz(b);
                    break;
                }
            }
#pragma unroll 1
            for (int w = p >> 5; w < kFrontCap / 32; ++w) {
                const uint32_t b = sh->fstart[w] & (w == (p >> 5) ? 0xFFFFFFFEu << (p & 31) : kFull);
                if (b) {
                    *ce = min(*ce, 32 * w + __ffs(b) - 1);
                    break;
                }
            }
        };
        int r = 1;
        uint32_t pm = 1u;
        bool ident = true;
        // a key's bits in pivot order, the first pivot's highest
        auto pivot_key = [&](uint32_t k) -> uint32_t {
            if (ident) return __brev(k);
            uint32_t v = 0u;
#pragma unroll
            for (int b = 0; b < 8; ++b) v |= sh->tab[b][(k >> (4 * b)) & 15u];
            return v;
        };
        if (warp == 0) {
            // ---- the front is filled for the next panel while the workers do this one's keys, order and sort
            if (!long_row && pcls < 0 && fl - w2 < kFrontLow && sh->head_next != n)
                front_fill(s, sh, g, f, fl, kFrontLow + w2 - fl);
        } else {
            const int wt = t - 32;
            uint32_t adj = 0u;
            if (!long_row) {
                // ---- keys: an entry of the window's rows per thread
                if (fp >= 0 && fp < fl) {
                    bool fresh;
                    sh->fslot[fp] = hash_slot(sh, f->v[fp], &fresh);
                }
                constexpr int U = (kMaxEntries + kCsrWorkers - 1) / kCsrWorkers;
                int y[U], c[U], own[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int e = wt + u * kCsrWorkers;
                    y[u] = -1;
                    own[u] = 0;
                    if ((warp - 1) * 32 + u * kCsrWorkers < entries) {
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
                    if ((warp - 1) * 32 + u * kCsrWorkers >= entries) break;
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
                        prefetch_l1(&s.rec[c[u]]);   // what move_ids reads
                        prefetch_l1(&s.freel[max(sh->free_top - 1 - at, 0)]);
                    }
                }
                named_barrier(1, kCsrWorkers);
                adj = lane < w2 ? sh->hmask[sh->fslot[lane]] & ~(1u << lane) : 0u;
            } else if (pcls >= 0) {   // a long row in a large class: the others go back
                if (fp >= 1 && fp < fl) s.cls[f->v[fp]] = pcls;
                if (t == 32) sh->pmore = sh->pmore || fl > 1;
                named_barrier(1, kCsrWorkers);
                fl = 1;
            }

            // ---- the pivots: window vertices 0..r-1 in order, or what warp 1 finds
            const uint32_t starts = sh->fstart[0] & low_bits(w2);
            const bool outside = pcls >= 0 && sh->pmore;   // members of the window's class beyond the front
            const bool straddle = w2 < fl ? w2 == 32 ? !(sh->fstart[1] & 1u) : !((sh->fstart[0] >> w2) & 1u) : outside;
            uint32_t ub = 0u;
            if (straddle && !long_row) {
                if (outside) ub = kFull;
                else {   // the class's members in the front beyond the window
                    int cs, ce;
                    front_class(w2, &cs, &ce, fl);
#pragma unroll 1
                    for (int p = w2 + lane; p < ce; p += 32) ub |= sh->hmask[sh->fslot[p]];
                    ub = __reduce_or_sync(kFull, ub);
                }
            }
            int mypos = -1, la = -1;   // warp 1
            if (!long_row) {
                bool order_fails = false;
                r = panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
                if (r < w2 && r < kPanelFew) {   // too few (the same in every warp)
                    if (!order_fails && outside) {
                        named_barrier(1, kCsrWorkers);
                        uint32_t any = 0u;
#pragma unroll 1
                        for (int k = wt; k < sh->lcount; k += kCsrWorkers)
                            if ((int)(sh->key2[k] >> 32) == pcls) any |= sh->hmask[(unsigned)sh->key2[k]];
                        if (fp >= w2 && fp < fl) any |= sh->hmask[sh->fslot[fp]];
                        any = __reduce_or_sync(kFull, any);
                        if (lane == 0 && any) atomicOr(&sh->ub, any);
                        named_barrier(1, kCsrWorkers);
                        ub = sh->ub;
                        r = panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
                    }
                    ident = !(order_fails && r < kPanelFew);
                }
            }
            pm = low_bits(r);
            if (warp == 1) {
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
                named_barrier(1, kCsrWorkers);
                pm = sh->pivmask;
                if (wt < 128) {
                    uint32_t v = 0u;
#pragma unroll
                    for (int b = 0; b < 4; ++b)
                        if ((wt >> b) & 1) v |= sh->bit[((wt >> 4) << 2) + b];
                    sh->tab[wt >> 4][wt & 15] = v;
                }
                named_barrier(1, kCsrWorkers);
            }

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
#pragma unroll 1
                for (int k0 = (warp - 1) * 32; k0 < lc; k0 += kCsrWorkers) {
                    const int k = k0 + lane;
                    unsigned long long e = 0ull;
                    uint32_t mk = 0u;
                    if (k < lc) {
                        e = sh->key2[k];
                        mk = sh->hmask[(unsigned)e] & pm;
                        if (mk && s.rec[(int)(e >> 32)].z == 1) {   // a class of one: it keeps its place
                            if (g.parent) g.parent[sh->y2[k]] = ident ? f->v[31 - __clz(mk)] : sh->piv[32 - __ffs(pivot_key(mk))];
                            mk = 0u;
                        }
                    }
                    append(mk != 0u, (int)(e >> 32), pivot_key(mk), k < lc ? sh->y2[k] : 0);
                }
            }
            if (front_warp && pcls >= 0) {   // the front's warps: the rest of a large class goes back (a long row left none)
                const bool left = fp < fl && !(fp < 32 && ((pm >> fp) & 1u));
                const uint32_t k = left ? sh->hmask[sh->fslot[fp]] & pm : 0u;
                if (left && k == 0u) s.cls[f->v[fp]] = pcls;
                append(k != 0u, pcls, pivot_key(k), left ? f->v[fp] : 0);
            }
            if (!long_row) {
                named_barrier(1, kCsrWorkers);
                panel_sort_moved(sh, sh->m);   // by (class, label, id)
            }
        }
        __syncthreads();
        r = sh->r;
        pm = sh->pivmask;
        if (warp == 0) ident = false;   // (no labels needed)
        int m = sh->m, unl = 0;
        if (pcls < 0) fl = sh->flen;
        const int fl2 = pcls >= 0 ? 0 : fl - r;

        // ---- the front after the panel: each class's members by label (the last warps)
        if (front_warp) {
            const bool left = pcls < 0 && fp < fl && !(fp < 32 && ((pm >> fp) & 1u));
            uint32_t ck = 0u;
            if (left) {
                const int v = f->v[fp];
                uint32_t k;
                if (long_row) {   // searched in the pivot's row
                    const int32_t *row = g.col + f->beg[0];
                    int lo = 0, hi = f->deg[0];
#pragma unroll 1
                    while (lo < hi) {
                        const int mid = (lo + hi) >> 1;
                        if (row[mid] < v) lo = mid + 1; else hi = mid;
                    }
                    k = lo < f->deg[0] && row[lo] == v ? 1u : 0u;
                } else {
                    k = hash_key(sh, v) & pm;
                }
                const uint32_t pk = pivot_key(k);
                ck = ~pk;
                sh->fck[fp] = ck;
                if (k) f->par[fp] = sh->piv[32 - __ffs(pk)];
            }
            named_barrier(2, kFrontCap);
            if (left) {
                int cs, ce;
                front_class(fp, &cs, &ce, fl);
                int np = cs - __popc(pm & low_bits(cs));
#pragma unroll 1
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
            named_barrier(2, kFrontCap);
            const bool st = fp < fl2 &&
                            (fp == 0 || sh->ncs[fp] != sh->ncs[fp - 1] || sh->nck[fp] != sh->nck[fp - 1]);
            const uint32_t b = __ballot_sync(kFull, st);
            if (lane == 0) sh->fstart[fp >> 5] = b;
        }

        // a class of one vertex: moving it changes nothing but its last adjacent pivot
        auto single = [&](int c) -> bool { return s.rec[c].z == 1; };
        // ---- a long row: the vertices without a numbered neighbour come in id order already, the others are sorted
        // by (class, row position), in shared memory when they fit
        const unsigned long long *lkey = nullptr;
        if (long_row) {
            const int64_t rb = f->beg[0];
            const int d = f->deg[0];
            int *kept = s.subid;   // the class of the row's k-th vertex when it is to be sorted
#pragma unroll 1
            for (int k0 = 32 * warp; k0 < d; k0 += kCsrThreads) {
                const int k = k0 + lane;
                const int y = k < d ? g.col[rb + k] : 0;
                int c = k < d ? s.cls[y] : kNumberedCls;
                if (c >= 0 && c != n && single(c)) {
                    if (g.parent) g.parent[y] = f->v[0];
                    c = kNumberedCls;
                }
                const unsigned um = __ballot_sync(kFull, c == n), lm = __ballot_sync(kFull, c >= 0 && c != n);
                if (lane == 0 && um) atomicAdd(&sh->lcount, __popc(um));
                if (lane == 0 && lm) atomicAdd(&sh->m, __popc(lm));
                if (k < d) kept[k] = c != n ? c : kNumberedCls;
            }
            __syncthreads();
            m = sh->m;
            unl = sh->lcount;
            // the new members' place at the arena's end, and a buffer after it
            if ((int64_t)s.cap - sh->atop < 3 * ((int64_t)m + unl) + 2) {   // the same for all threads
                __syncthreads();
                arena_pack(s, sh, g);
            }
            int *const after = (int *)s.arena + sh->atop + (unsigned)(m + unl);
            lkey = sort_long_row(sh, kept, d, m, n,
                                 reinterpret_cast<unsigned long long *>((reinterpret_cast<uintptr_t>(after) + 7) & ~uintptr_t(7)),
                                 (unsigned long long *)s.skey);
        }

        // ---- new classes
        // nothing in the list but vertices that had no numbered neighbour: what the panel met goes to the front
        const bool to_front = !long_row && m > 0 && fl2 + m <= kFrontCap && sh->head_next == n &&
                              (int)(sh->key2[0] >> 32) == n;
        const Moved<false> mv{sh, sh->key2, nullptr, m, nullptr, nullptr};
        uint32_t *lbits = reinterpret_cast<uint32_t *>(sh->y);   // y, y2 and sub
        int *llast = reinterpret_cast<int *>(sh->key);           // key and key2
        static_assert(sizeof(sh->key) + sizeof(sh->key2) >= 3 * kMaxEntries * sizeof(int), "a word of starts per int");
        const bool keep_bits = long_row && m <= 3 * 32 * kMaxEntries;
        const Moved<true> ml{sh, lkey, g.col + f->beg[0], m, keep_bits ? lbits : nullptr, llast};
        if (keep_bits) {
#pragma unroll 1
            for (int k0 = 32 * warp; k0 < m; k0 += kCsrThreads) {
                const int k = k0 + lane;
                const uint32_t cb =
                    __ballot_sync(kFull, k < m && (k == 0 || lkey[max(k - 1, 0)] >> 32 != lkey[k] >> 32));
                if (lane == 0) lbits[k0 >> 5] = cb;
            }
            __syncthreads();
            // the last start up to each word's end, so that no member walks back through its class (a row of
            // 65,000 members of one class: 6 ms by walking)
            const int nw = (m + 31) >> 5, per = (nw + kCsrThreads - 1) / kCsrThreads;
            const int a = min(t * per, nw), b = min(a + per, nw);
            int own = -1;
#pragma unroll 1
            for (int w = a; w < b; ++w)
                if (lbits[w]) own = 32 * w + 31 - __clz(lbits[w]);
            int incl = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl = max(incl, u);
            }
            if (lane == 31) sh->scan[warp] = incl;
            __syncthreads();
            int at = __shfl_up_sync(kFull, incl, 1);
            if (lane == 0) at = -1;
            at = max(at, __reduce_max_sync(kFull, lane < warp ? sh->scan[lane] : -1));
#pragma unroll 1
            for (int w = a; w < b; ++w) {
                if (lbits[w]) at = 32 * w + 31 - __clz(lbits[w]);
                llast[w] = at;
            }
        }
        if (!long_row && !to_front)
#pragma unroll 1
            for (int k0 = 32 * warp; k0 < m; k0 += kCsrThreads) {
                const int k = k0 + lane;
                const unsigned long long x = k < m ? sh->key2[k] : 0ull, px = k > 0 && k < m ? sh->key2[k - 1] : 0ull;
                const uint32_t gb = __ballot_sync(kFull, k < m && (k == 0 || x != px));
                const uint32_t cb = __ballot_sync(kFull, k < m && (k == 0 || x >> 32 != px >> 32));
                if (lane == 0) {
                    sh->gstart[k0 >> 5] = gb;
                    sh->cstart[k0 >> 5] = cb;
                }
            }
        __syncthreads();
        if (!to_front) {
            if (long_row) move_ids(s, sh, g, ml, (int *)s.subid);
            else move_ids(s, sh, g, mv, sh->sub);
        }
        if (t == 0 && unl > 0) {   // the new class before the last one
            const int id = s.freel[atomicSub(&sh->free_top, 1) - 1], before = s.rec[n].w;
            s.rec[id].w = before;
            set_next(s, sh, g, before, id);
            set_next(s, sh, g, id, n);
            s.rec[n].w = id;
            sh->unl_size -= unl;
            sh->unl_id = id;
        }
        unsigned atop = sh->atop;
        clear_hash();
        __syncthreads();
        if (t == 0) {   // (what the threads still need of these they hold)
            sh->flen = fl2 + (to_front ? m : 0);
            sh->pcls = -1;
            sh->pmore = 0;
            sh->lcount = 0;
            sh->m = 0;
            sh->ub = 0u;
            if (to_front) sh->unl_size -= m;
        }
        if (to_front) {
            if (t < m) {
                const int p = fl2 + t, y = sh->y2[t];
                const unsigned long long k = sh->key2[t];
                front_put(nf, p, y, sh->piv[32 - __ffs(~(uint32_t)k)], g.row_ptr[y], g.row_ptr[y + 1]);
                s.cls[y] = kFrontCls;
                if (t == 0 || k != sh->key2[t - 1]) atomicOr(&sh->fstart[p >> 5], 1u << (p & 31));
            }
        } else if (m + unl > 0) {
            if (s.cap - atop < (unsigned)(m + unl)) {   // the same for all threads (a long row has its room)
                arena_pack(s, sh, g);
                atop = sh->atop;
                __syncthreads();
            }
            if (t == 0) sh->atop = atop + (unsigned)(m + unl);
            if (long_row) move_members(s, sh, g, ml, (int *)s.subid, atop);
            else move_members(s, sh, g, mv, sh->sub, atop);
            if (unl > 0) {   // those without a numbered neighbour, in row order
                const int64_t rb = f->beg[0];
                const int d = f->deg[0], id = sh->unl_id, x = f->v[0];
                const unsigned out = atop + (unsigned)m;
                unsigned done = 0u;
#pragma unroll 1
                for (int k0 = 0; k0 < d; k0 += kCsrThreads) {
                    const int k = k0 + t, y = k < d ? g.col[rb + k] : -1;
                    const bool in = k < d && s.cls[y] == n;
                    const unsigned lm = __ballot_sync(kFull, in);
                    if (lane == 0) sh->scan[warp] = __popc(lm);
                    __syncthreads();
                    const int wc = lane < kCsrThreads / 32 ? sh->scan[lane] : 0;
                    const int ahead = __reduce_add_sync(kFull, lane < warp ? wc : 0);
                    if (in) {
                        s.arena[out + done + ahead + __popc(lm & lanes_below(lane))] = y;
                        s.cls[y] = id;
                        if (g.parent) g.parent[y] = x;
                    }
                    done += __reduce_add_sync(kFull, wc);
                    __syncthreads();
                }
                if (t == 0) {
                    s.rec[id].x = (int)out;
                    s.rec[id].y = (int)(out + unl);
                    s.rec[id].z = unl;
                }
            }
        }
        if (!long_row) lost = max(lost + kStepsBelow - r, 0);
        if (r >= kStepsBelow) span = 1;
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
