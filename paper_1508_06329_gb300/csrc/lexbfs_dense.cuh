// lexbfs_dense.cuh — LexBFS by partition refinement in panels of up to 32
// pivots, one CTA per graph.
//
// Method (Section 4.2 of the paper; its GPU form in Section 6.1): the
// unnumbered vertices are partitioned into classes ordered top first.  Each
// step visits the first vertex x of the first class, then replaces every class
// C by C ∩ N_x followed by C \ N_x.  Within a class vertices are kept in id
// order, so the visited vertex is the lowest id of the top class.
//
// One step at a time costs a row load, two CTA barriers and a pass over the
// row per vertex (1.74 us per step at n = 16,384 on GB300, all of it latency
// and issue).  But the steps of the classes in front do not need the rest of
// the partition: every member of a class is visited before any member of a
// later class, and the order of the members of the first classes depends only
// on the edges among them.  So a panel takes the next (at most) 32 vertices in
// partition order, the window:
//   1. the threads read the window's rows, a word of all 32 rows per thread,
//      and transpose the 32 x 32 bits in registers: vertex y's key, bit j =
//      adjacent to window vertex j;
//   2. the window vertices' own keys are the window's adjacency: every warp
//      finds how many of them are visited in window order, in one comparison
//      per lane (panel_in_order).  That is nearly always all of them; when it
//      is fewer than kPanelFew, warp 0 runs LexBFS on the window, one lane per
//      vertex (panel_solve);
//   3. the classes whose members' keys differ are split: members in decreasing
//      order of the key read in pivot order (the lexicographic order of the
//      labels these r steps append), ids ascending among equals.
// A window's last class may continue beyond it.  Then a pivot from its part in
// the window is only taken while no member outside can have a larger label:
// while its appended label is all ones, or, when that gives few pivots (large
// independent sets), at least the OR of the outside members' keys; members
// outside have larger ids, so equality suffices.  A panel numbers 26..32
// vertices on broad graphs: subtree-intersection and random graphs, trees, grids.
//
// On narrow graphs the next vertex is known only after the one before (paths,
// cycles, matchings, small components, interval graphs of small degree): it is
// seldom in the window, and a panel numbers two to ten.  When the windows do not
// pay, warp 0 takes pivots one by one, a row load and no split pass each
// (panel_steps), 32 to a panel, and windows are tried again from time to time.
//
// Measured on GB300 (whole test; one step per vertex -> this): the pair of
// n = 16,384 graphs at density 0.1 28.3 -> 4.2 ms (7.7 us per panel of 31),
// G(10,000, 0.5) 49.4 -> 1.9 ms, n = 41,003 104 -> 33 ms, 4,096 graphs of
// 16..2,048 vertices 3.8 -> 1.25 ms, one graph of 1,000 vertices 913 -> 175 us.
// Narrow (windows alone in brackets): path of 1,000 vertices 1.02 -> 0.72 ms
// (3.4), 16,384 24.7 -> 16.6 (143), 41,003 95 -> 70 (1,200); disjoint K4, 16,384
// 19.1 -> 14.2 (51); 600 graphs of 64..1,024 vertices of disjoint K4, the one kind
// that one step per vertex did faster, with its rows in shared memory, 0.96 -> 1.03
// (3.2).
// What bounds a panel is latency and issue: the rows' L2 loads and their
// transpose (a third), the passes over positions, the barriers, and instruction
// fetch (code that runs once per panel is rolled where it can be).
//
// State: perm[] holds the vertices by position (numbered ones in front, then
// class after class, ascending ids inside a class), and the class boundaries
// are a bitmask over positions.  A class that does not split is not touched,
// so a panel without splits costs steps 1, 2 and one pass over the positions
// that compares neighbouring keys.  Splits: members with key 0 keep their
// order and move to the end of the class (prefix counts), the others are
// sorted by (class, key, order), by counting when the classes' moved parts are
// small, else with a bitonic network.  More than cap of them (the first steps
// on a dense random graph): the panel is cut to its first pivot, whose one-bit
// keys need no sort.
//
// Parents: p(y) of the perfect-elimination check (Section 5.2), y's neighbour
// with the largest order index below its own, is the last pivot whose bit is
// set in y's label.  Members of a class share their label, so while a class is
// unnumbered ppos[its first position] holds that pivot (-1: none); a pivot's
// own parent is the last adjacent pivot of its panel or else that value.
// emask: E_b, the vertices numbered before position 32 b, one mask row per 32
// positions for the staged check.
#pragma once
#include "common.cuh"

namespace cg {

constexpr unsigned kNoVertex = 0xFFFFFFFFu;

// Where the per-vertex arrays live.  A vertex's key is gathered once per panel
// in position order, so the keys stay in shared memory as long as they fit;
// perm is only read in order, so it moves to the workspace first.
constexpr int kStateSmem = 0;       // perm and keys in shared memory, 16-bit ids
constexpr int kStatePermGlobal = 1; // perm in the workspace, keys in shared memory, 16-bit ids
constexpr int kStateGlobal = 2;     // perm and keys in the workspace, 32-bit ids

template <int STATE>
struct PanelId { using type = uint16_t; };
template <>
struct PanelId<kStateGlobal> { using type = uint32_t; };

struct PanelScalars {
    uint4 row4[8];          // four times the window vertices (every warp writes the same ones)
    int piv[32];            // the panel's pivots in order
    int par[32];            // their parents
    uint32_t bit[32];       // window vertex j's bit in pivot order (0: not a pivot)
    uint32_t tab[8][16];    // nibble tables of the same permutation
    int scan[3][32];
    int r;                  // pivots of the panel
    uint32_t pivmask;       // window vertices that are pivots
    int ident;              // the pivots are window vertices 0..r-1 in order
    int cend;               // end of the class that goes on beyond the window
    uint32_t ub;            // OR of the keys of its members beyond the window
    int set_start;          // position whose boundary bit the commit set (-1: none)
    int any;                // some class has members with different keys
    int nz_max;             // the most moved members in one split class
    int next_graph;
};
constexpr size_t kPanelScalarBytes = (sizeof(PanelScalars) + 15) & ~size_t(15);

constexpr int kPanelWordArrays = 9;
constexpr int kPanelCount = 1024;   // moved members of one class sorted by counting up to this many
constexpr int kPanelFew = 16;   // pivots below which a panel is worth extending by slower rules
constexpr int kSortCapMax = 4096;
constexpr int kPanelSettled = 64;      // panel_steps: nothing is left to split
// Windows give way to steps when they have numbered panel_lost_limit vertices less than kStepsBelow each.  A
// window's panel costs 3.3 us at n = 1,000 and 13 at 16,384 when it splits a large class, a step 0.6 to 0.9 us; the
// limit keeps the first windows of broad graphs (a few pivots each until the classes are many) out of it.
constexpr int kStepsBelow = 12;
__device__ __forceinline__ int panel_lost_limit(int n) { return min(36, 8 + n / 8); }
// Windows with a vertex of more neighbours in the window than this are of a dense graph: a step would meet too many.
constexpr unsigned kStepsDegree = 16;
// Panels of steps before a window is tried again (a try costs a few steps) are 1, 4, then this many.
constexpr int kStepsMost = 16;

// Elements the split sort holds: all of a small graph's vertices, fewer when
// the state leaves less room (bytes: shared memory available for them).
__host__ __device__ inline int panel_sort_cap(int n, size_t bytes) {
    int cap = kSortCapMax;
#pragma unroll 1
    while (cap > 64 && (cap / 2 >= n || (size_t)cap * 12 > bytes)) cap /= 2;
    return cap;
}

// Shared bytes of a graph of n vertices without the sort's arrays.
__host__ __device__ inline size_t panel_state_bytes(int n, int state) {
    const size_t wn = (size_t)(n + 31) / 32;
    size_t b = wn * 4 * kPanelWordArrays;
    b = (b + 15) & ~size_t(15);
    if (state != kStateGlobal) b += wn * 32 * 4;       // keys
    if (state == kStateSmem) b += wn * 32 * 2 * 2;     // perm and its scratch copy
    return b;
}
__host__ __device__ inline size_t panel_sort_bytes(int cap) { return (size_t)cap * 12; }

// Workspace bytes per CTA.
__host__ __device__ inline size_t panel_global_bytes(int n, int state) {
    const size_t nv = (size_t)(n + 31) / 32 * 32;
    const size_t b = state == kStateSmem ? 0 : state == kStatePermGlobal ? nv * 2 * 2 : nv * 4 * 3;
    return (b + 255) & ~size_t(255);
}

template <typename Id>
struct PanelState {
    CG_ARR(Id) perm;            // vertices by position
    CG_ARR(Id) tmp;             // split classes being rewritten
    CG_ARR(uint32_t) key;       // by key_slot(vertex)
    CG_ARR(uint32_t) start;     // bit q: a class starts at position q
    CG_ARR(uint32_t) diff;      // bit q: q's key differs from q - 1's, same class
    CG_ARR(uint32_t) touch;     // bit q: q's key is not 0
    CG_ARR(uint32_t) flag;      // bit q: q's class splits
    CG_ARR(uint32_t) numbered;  // bit v: vertex v is numbered
    CG_ARR(int) dpre;           // differing keys before a word of positions
    CG_ARR(int) last;           // last class start up to the end of a word of positions
    CG_ARR(int) next;           // first class start from a word of positions on
    CG_ARR(int) nzpre;          // moved members of split classes before a word of positions
    CG_ARR(unsigned long long) comp;   // [cap] moved members: class start, inverted key, list index
    CG_ARR(uint32_t) lv;        // [cap] their vertices
    int cap;
};

// A thread writes the 32 keys of one word of vertices as eight 16-byte pieces;
// the pieces are rotated by the word's index so that neighbouring threads'
// pieces fall into different banks.
__device__ __forceinline__ unsigned key_slot(unsigned v) { return v ^ ((v >> 3) & 0x1Cu); }

template <int STATE>
__device__ inline PanelState<typename PanelId<STATE>::type> panel_carve(unsigned char *smem, unsigned char *gmem,
                                                                        int n, int cap) {
    using Id = typename PanelId<STATE>::type;
    PanelState<Id> s;
    const int wn = (n + 31) >> 5;
    const size_t nv = (size_t)wn * 32;
    unsigned char *q = smem;
    s.comp = cg_arr(reinterpret_cast<unsigned long long *>(q), cap, kChkSort);
    q += (size_t)cap * 8;
    s.lv = cg_arr(reinterpret_cast<uint32_t *>(q), cap, kChkSort);
    q += (size_t)cap * 4;
    if constexpr (STATE != kStateGlobal) {
        s.key = cg_arr(reinterpret_cast<uint32_t *>(q), nv, kChkKey);
        q += nv * 4;
    } else {
        s.key = cg_arr(reinterpret_cast<uint32_t *>(gmem), nv, kChkKey);
        gmem += nv * 4;
    }
    Id *p;
    if constexpr (STATE == kStateSmem) {
        p = reinterpret_cast<Id *>(q);
        q += nv * 2 * 2;
    } else {
        p = reinterpret_cast<Id *>(gmem);
    }
    s.perm = cg_arr(p, nv, kChkPerm);
    s.tmp = cg_arr(p + nv, nv, kChkPerm);
    uint32_t *w = reinterpret_cast<uint32_t *>(q);
    s.start = cg_arr(w, wn, kChkCls);
    s.diff = cg_arr(w + wn, wn, kChkSplit);
    s.touch = cg_arr(w + 2 * (size_t)wn, wn, kChkSplit);
    s.flag = cg_arr(w + 3 * (size_t)wn, wn, kChkSplit);
    s.numbered = cg_arr(w + 4 * (size_t)wn, wn, kChkNumbered);
    int *iw = reinterpret_cast<int *>(w + 5 * (size_t)wn);
    s.dpre = cg_arr(iw, wn, kChkSplit);
    s.last = cg_arr(iw + wn, wn, kChkSplit);
    s.next = cg_arr(iw + 2 * (size_t)wn, wn, kChkSplit);
    s.nzpre = cg_arr(iw + 3 * (size_t)wn, wn, kChkSplit);
    s.cap = cap;
    return s;
}

// One stage of the 32 x 32 bit transpose: blocks of S bits exchanged between
// r[k] and r[k + S].
template <int S, uint32_t M>
__device__ __forceinline__ void transpose_stage(uint32_t (&r)[32]) {
#pragma unroll
    for (int k = 0; k < 32; ++k)
        if (!(k & S)) {
            const uint32_t a = r[k], b = r[k + S];
            if constexpr (S == 16) {
                r[k] = __byte_perm(a, b, 0x5410);
                r[k + S] = __byte_perm(a, b, 0x7632);
            } else if constexpr (S == 8) {
                r[k] = __byte_perm(a, b, 0x6240);
                r[k + S] = __byte_perm(a, b, 0x7351);
            } else {
                r[k] = (a & M) | ((b << S) & ~M);
                r[k + S] = ((a >> S) & M) | (b & ~M);
            }
        }
}
// out[v] bit j = in[j] bit v
__device__ __forceinline__ void transpose32(uint32_t (&r)[32]) {
    transpose_stage<16, 0u>(r);
    transpose_stage<8, 0u>(r);
    transpose_stage<4, 0x0F0F0F0Fu>(r);
    transpose_stage<2, 0x33333333u>(r);
    transpose_stage<1, 0x55555555u>(r);
}

// Eight neighbouring 16- or 32-bit entries (16-byte aligned).
__device__ __forceinline__ void panel_load8(const uint16_t *p, uint16_t (&v)[8]) {
    const uint4 a = *reinterpret_cast<const uint4 *>(p);
    const uint32_t x[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = (uint16_t)(x[e >> 1] >> (16 * (e & 1)));
}
__device__ __forceinline__ void panel_load8(const uint32_t *p, uint32_t (&v)[8]) {
    const uint4 a = reinterpret_cast<const uint4 *>(p)[0], b = reinterpret_cast<const uint4 *>(p)[1];
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// The same, unpacked when they are looked at.
template <typename Id>
struct Panel8 {
    uint32_t x[2 * sizeof(Id)];
    __device__ __forceinline__ void load(const Id *p) {
#pragma unroll
        for (unsigned k = 0; k < sizeof(Id) / 2; ++k) {
            const uint4 a = reinterpret_cast<const uint4 *>(p)[k];
            x[4 * k] = a.x, x[4 * k + 1] = a.y, x[4 * k + 2] = a.z, x[4 * k + 3] = a.w;
        }
    }
    __device__ __forceinline__ uint32_t operator[](int e) const {
        return sizeof(Id) == 2 ? x[e >> 1] >> (16 * (e & 1)) & 0xFFFFu : x[e];
    }
};

// r[j] = col[v_j * stride], row4 holding 4 v_j: a byte offset is one 32 x 32 bit
// product.  The window's vertices come from shared memory, four at a time: taken
// from the lanes by shuffles, one before every load, a warp's 32 loads took
// 3,400 cycles instead of 950 (n = 1,000; 5,900 instead of 2,500 with 16 warps).
__device__ __forceinline__ void panel_load_rows(const uint32_t *__restrict__ col, int stride, const uint4 *row4,
                                                uint32_t (&r)[32]) {
    auto at = [&](uint32_t v4) {
        return *reinterpret_cast<const uint32_t *>(reinterpret_cast<const char *>(col) +
                                                   (unsigned long long)v4 * (uint32_t)stride);
    };
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const uint4 v = row4[j];
        r[4 * j] = at(v.x);
        r[4 * j + 1] = at(v.y);
        r[4 * j + 2] = at(v.z);
        r[4 * j + 3] = at(v.w);
    }
}

// The thread's warp, from a shuffle: the compiler then knows that it is the same
// in all lanes, and that loops and branches on it keep the warp together.  Without
// that every shuffle and vote in them carries a branch and code for a warp that has
// come apart.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xFFFFFFFFu, (int)(threadIdx.x >> 5), 0); }

__device__ __forceinline__ uint32_t lanes_below(int lane) { return (1u << lane) - 1u; }
__device__ __forceinline__ uint32_t low_bits(int k) { return k >= 32 ? 0xFFFFFFFFu : (1u << k) - 1u; }

// How many window vertices are visited in window order (every warp computes
// it).  Lane z's turn comes after lanes 0..z-1 if no later vertex of its class
// has a larger label with respect to them.  A lexicographic >= over lanes 0..z
// also holds over lanes 0..z-1, so as long as every lane's label is >= the next
// one's in its class, the later ones need no comparison; a lane with a larger
// label than the one before it is compared with all before it.  Lanes of a
// class that goes on beyond the window (straddle) are also compared with ub,
// the largest label out there.  *order_fails: the first lane that is not
// visited in order fails inside the window, not against ub.
__device__ __forceinline__ int panel_in_order(int lane, int w2, uint32_t starts, bool straddle, uint32_t adj,
                                              uint32_t ub, bool *order_fails) {
    const uint32_t prefix = lanes_below(lane), above = starts & (0xFFFFFFFEu << lane);
    auto loses = [&](uint32_t other) {   // label of lane < label of the other, over lanes 0..lane-1
        const uint32_t d = (adj ^ other) & prefix;
        return d != 0u && !(adj & d & (0u - d));
    };
    const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, adj, 1);
    const uint32_t f1 = __ballot_sync(0xFFFFFFFFu, straddle && lane < w2 && !above && loses(ub));
    uint32_t f0 = 0u;
#pragma unroll 1
    for (uint32_t larger = __ballot_sync(0xFFFFFFFFu, lane + 1 < w2 && !((starts >> lane) & 2u) && loses(next)); larger;
         larger &= larger - 1u) {
        const int y = __ffs(larger);   // the lane after the one that loses to it
        const uint32_t other = __shfl_sync(0xFFFFFFFFu, adj, y);
        f0 |= __ballot_sync(0xFFFFFFFFu, lane < y && !(above & low_bits(y + 1)) && loses(other));
    }
    const uint32_t f = f0 | f1 | ~low_bits(w2);
    const int r = f ? __ffs(f) - 1 : 32;
    *order_fails = r < w2 && ((f0 >> r) & 1u);
    return r;
}

// LexBFS of the window by one warp.  Lane k holds window vertex k's adjacency
// mask; starts has the first lane of every class; straddle: the last class
// continues beyond the window, and outside(j) = bit j of ub says whether
// pivot j may be adjacent to a member out there.  Returns the number of pivots;
// mypos = this lane's index among them (-1: not taken), la = the index of its
// last adjacent pivot before it (-1: none).
__device__ __forceinline__ int panel_solve(int lane, int w2, uint32_t starts, bool straddle, uint32_t adj, uint32_t ub,
                                           int *mypos_out, int *la_out) {
    uint32_t undone = low_bits(w2);
    starts &= undone;
    const uint32_t cs = straddle ? undone & (0xFFFFFFFFu << (31 - __clz(starts))) : 0u;
    uint32_t key = 0u, front = 0u, fkey = 0u, ubkey = 0u, cls = 0u;
    int r = 0, mypos = -1, la = -1;
#pragma unroll 1
    while (undone) {
        if (!front) {   // the top class's members with the largest label
            if (!(cls & undone)) {
                const int l = __ffs(undone) - 1;
                const uint32_t above = starts & (0xFFFFFFFEu << l);
                cls = undone & (above ? (above & (0u - above)) - 1u : 0xFFFFFFFFu) & (0xFFFFFFFFu << l);
            }
            const uint32_t cand = cls & undone;
            const bool in = (cand >> lane) & 1u;
            fkey = __reduce_max_sync(0xFFFFFFFFu, in ? key : 0u);
            front = __ballot_sync(0xFFFFFFFFu, in && key == fkey);
            if ((cls & cs) && fkey < ubkey) break;
        }
        const int x = __ffs(front) - 1;
        const uint32_t bit = (adj >> x) & 1u;
        const uint32_t a = __ballot_sync(0xFFFFFFFFu, bit);
        if (lane == x) mypos = r;
        undone &= ~(1u << x);
        front &= ~(1u << x);
        if (bit && ((undone >> lane) & 1u)) la = r;
        key = 2u * key + bit;
        ubkey = 2u * ubkey + ((ub >> x) & 1u);
        ++r;
        if (front) {
            const uint32_t f2 = front & a;
            fkey = 2u * fkey + (f2 ? 1u : 0u);
            if (f2) front = f2;
            if ((cls & cs) && fkey < ubkey) break;
        }
    }
    *mypos_out = mypos;
    *la_out = la;
    return r;
}

// Block-wide exclusive scans, one value each per thread: the sum of a, and with
// MINMAX the maximum of b over the threads before and the minimum of c over the
// threads after.  Returns the sum of all a.  Two barriers.
template <int T, bool MINMAX>
__device__ __forceinline__ int panel_scan(PanelScalars *sc, int &a, int &b, int &c) {
    constexpr int NW = T / 32;
    constexpr int kBig = 0x7FFFFFFF;
    const int lane = threadIdx.x & 31, warp = warp_index();
    int ia = a, ib = b, ic = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int ua = __shfl_up_sync(0xFFFFFFFFu, ia, o);
        if (lane >= o) ia += ua;
        if constexpr (MINMAX) {
            const int ub = __shfl_up_sync(0xFFFFFFFFu, ib, o);
            const int dc = __shfl_down_sync(0xFFFFFFFFu, ic, o);
            if (lane >= o) ib = max(ib, ub);
            if (lane + o < 32) ic = min(ic, dc);
        }
    }
    if (lane == 31) {
        sc->scan[0][warp] = ia;
        if constexpr (MINMAX) sc->scan[1][warp] = ib;
    }
    if constexpr (MINMAX) {
        if (lane == 0) sc->scan[2][warp] = ic;
        ib = __shfl_up_sync(0xFFFFFFFFu, ib, 1);
        ic = __shfl_down_sync(0xFFFFFFFFu, ic, 1);
        if (lane == 0) ib = -1;
        if (lane == 31) ic = kBig;
    }
    __syncthreads();
    const int wa = lane < NW ? sc->scan[0][lane] : 0;
    const int total = __reduce_add_sync(0xFFFFFFFFu, wa);
    a = ia - a + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? wa : 0);
    if constexpr (MINMAX) {
        b = max(ib, __reduce_max_sync(0xFFFFFFFFu, lane < warp ? sc->scan[1][lane] : -1));
        c = min(ic, __reduce_min_sync(0xFFFFFFFFu, lane > warp && lane < NW ? sc->scan[2][lane] : kBig));
    }
    __syncthreads();
    return total;
}

// Sorts a[0..p), p a power of two, ascending.  Pair exchanges at distances up
// to 32 stay inside a warp's 64 elements and need no CTA barrier.
template <int T>
__device__ __forceinline__ void panel_sort(unsigned long long *a, int p) {
#pragma unroll 1
    for (int k = 2; k <= p; k <<= 1)
#pragma unroll 1
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
            for (int e = threadIdx.x; e < p / 2; e += T) {
                const int lo = ((e & ~(j - 1)) << 1) | (e & (j - 1)), hi = lo | j;
                const unsigned long long x = a[lo], y = a[hi];
                if ((x > y) == ((lo & k) == 0)) {
                    a[lo] = y;
                    a[hi] = x;
                }
            }
            const int nj = j > 1 ? j >> 1 : k;
            if (j > 32 || nj > 32) __syncthreads();
            else __syncwarp();
        }
    __syncthreads();
}

// E_b from the numbered mask (padding words are zero).
template <int T, typename Arr>
__device__ __forceinline__ void panel_write_mask(uint32_t *emask, int b, int n, const Arr &numbered) {
    const int wn = (n + 31) >> 5, es = mask_stride(n);
    uint32_t *e = emask + (size_t)b * es;
#pragma unroll 1
    for (int w = threadIdx.x; w < es; w += T) e[w] = w < wn ? numbered[w] : 0u;
}

// Neighbouring positions per thread when split classes are rewritten: one for
// small CTAs (small graphs: little to do, so a short chain per position), a
// byte of the masks for large ones.  Both are rolled loops: code that runs
// once per panel is bound by instruction fetch, and the same passes unrolled
// eight times took 4,096 small graphs from 1.5 to 2.5 ms.
constexpr int panel_rewrite_width(int threads) { return threads >= 512 ? 8 : 1; }

// The classes whose members' keys differ (a lane compares eight neighbouring
// positions) are split.  cut (warp 0): the panel is cut to its first pivot, as
// more members move than the sort holds.  Returns the numbered vertices.
template <int STATE, int T, typename PivotKey, typename Cut>
__device__ __forceinline__ int panel_split(int n, int i, const PanelState<typename PanelId<STATE>::type> &st,
                                           PanelScalars *sc, int32_t *ppos_out, int &r, uint32_t &pm, bool &ident,
                                           const PivotKey &pivot_key, const Cut &cut) {
    using Id = typename PanelId<STATE>::type;
    constexpr int NW = T / 32, G = panel_rewrite_width(T);
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    const int wn = (n + 31) >> 5;
    const auto ppos = cg_arr(ppos_out, n, kChkPpos);
    int i2;
    for (;;) {
        i2 = i + r;
        if (!ident)
#pragma unroll 1
            for (int e = t; e < 128; e += T) {
                uint32_t v = 0u;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if ((e >> b) & 1) v |= sc->bit[((e >> 4) << 2) + b];
                sc->tab[e >> 4][e & 15] = v;
            }
        bool differ = false;
#pragma unroll 1
        for (int c = warp ? (i2 & ~255) + (warp - 1) * 256 : n; c < n; c += (T - 32) * 8) {   // (warp 0: commit)
            const int q0 = c + 8 * lane;
            uint32_t k[8], kp = 0u;
            if (q0 < n) {
                Id v[8];
                panel_load8(&st.perm[q0], v);
#pragma unroll
                for (int e = 0; e < 8; ++e) k[e] = st.key[key_slot(v[e])] & pm;
                if (lane == 0 && q0 > i2) kp = st.key[key_slot(st.perm[q0 - 1])] & pm;
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) k[e] = 0u;
            }
            const uint32_t up = __shfl_up_sync(kAll, k[7], 1);
            if (lane > 0) kp = up;
            if (q0 < n) {
                uint32_t dm = 0u, nm = 0u;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    dm |= (k[e] != (e ? k[e - 1] : kp) ? 1u : 0u) << e;
                    nm |= (k[e] ? 1u : 0u) << e;
                }
                uint32_t live = q0 >= i2 ? 0xFFu : q0 + 8 > i2 ? 0xFFu << (i2 - q0) : 0u;   // positions i2..n-1
                if (q0 + 8 > n) live &= low_bits(n - q0);
                nm &= live;
                if (q0 <= i2) live &= live - 1u;   // i2 itself starts a class
                dm &= live & ~(uint32_t)reinterpret_cast<const uint8_t *>(&st.start[q0 >> 5])[(q0 >> 3) & 3];
                reinterpret_cast<uint8_t *>(&st.diff[q0 >> 5])[(q0 >> 3) & 3] = (uint8_t)dm;
                reinterpret_cast<uint8_t *>(&st.touch[q0 >> 5])[(q0 >> 3) & 3] = (uint8_t)nm;
                differ |= dm != 0u;
            }
        }
        if (__any_sync(kAll, differ) && lane == 0) sc->any = 1;
        __syncthreads();
        if (!sc->any) break;
        const int pw = i2 >> 5;

        // ---- positions of the classes that split (thread t: words [wa, wb) of positions)
        const int kw = (wn + T - 1) / T, wa = min(t * kw, wn), wb = min(wa + kw, wn);
        int ds = 0, lm = -1, nm = 0x7FFFFFFF;
#pragma unroll 1
        for (int w = wa; w < wb; ++w) {
            const uint32_t b = st.start[w];
            if (w >= pw) ds += __popc(st.diff[w]);
            if (b) {
                lm = 32 * w + 31 - __clz(b);
                if (nm == 0x7FFFFFFF) nm = 32 * w + __ffs(b) - 1;
            }
        }
        const int dtotal = panel_scan<T, true>(sc, ds, lm, nm);
#pragma unroll 1
        for (int w = wa; w < wb; ++w) {
            const uint32_t b = st.start[w];
            st.dpre[w] = ds;
            if (w >= pw) ds += __popc(st.diff[w]);
            if (b) lm = 32 * w + 31 - __clz(b);
            st.last[w] = lm;
        }
        nm = min(nm, n);
#pragma unroll 1
        for (int w = wb - 1; w >= wa; --w) {
            const uint32_t b = st.start[w];
            if (b) nm = 32 * w + __ffs(b) - 1;
            st.next[w] = nm;
        }
        if (t == 0) sc->nz_max = 0;
        __syncthreads();
        auto diffs_before = [&](int q) -> int {
            if (q >= n) return dtotal;
            const int w = q >> 5;
            return w < pw ? 0 : st.dpre[w] + __popc(st.diff[w] & lanes_below(q & 31));
        };
        int nzs = 0;
#pragma unroll 1
        for (int w = wa; w < wb; ++w) {
            uint32_t f = 0u;
            if (w >= pw) {
                const uint32_t b = st.start[w], d = st.diff[w];
                const int nx = w + 1 < wn ? st.next[w + 1] : n;
                const uint32_t lead = b ? (b & (0u - b)) - 1u : kAll;   // before the word's first start
                uint32_t tail = 0u;
                if (lead && w > 0 &&
                    diffs_before(b ? 32 * w + __ffs(b) - 1 : nx) > diffs_before(st.last[w - 1]))
                    f |= lead;
                if (b) {
                    tail = kAll << (31 - __clz(b));
                    if (diffs_before(nx) > diffs_before(32 * w + 31 - __clz(b))) f |= tail;
                }
                uint32_t inner = d & ~lead & ~tail;   // classes inside the word
#pragma unroll 1
                while (inner) {
                    const int q = __ffs(inner) - 1;
                    const uint32_t lo = 31 - __clz(b & lanes_below(q + 1)), up = b & (0xFFFFFFFEu << q);
                    const uint32_t m = ((up & (0u - up)) - 1u) & (kAll << lo);
                    f |= m;
                    inner &= ~m;
                }
                nzs += __popc(st.touch[w] & f);
            }
            st.flag[w] = f;
        }
        int unused0 = 0, unused1 = 0;
        const int m = panel_scan<T, false>(sc, nzs, unused0, unused1);
        if (m > st.cap && r > 1) {   // more to sort than fits: the panel ends after its first pivot
            r = 1;
            pm = 1u;
            if (warp == 0) {
                if (lane == 0) {
                    if (sc->set_start >= 0) st.start[sc->set_start >> 5] &= ~(1u << (sc->set_start & 31));
                    sc->any = 0;
                }
                __syncwarp();
                cut();
            }
            ident = true;
            __syncthreads();
            continue;
        }
#pragma unroll 1
        for (int w = wa; w < wb; ++w) {
            st.nzpre[w] = nzs;
            if (w >= pw) nzs += __popc(st.touch[w] & st.flag[w]);
        }
        __syncthreads();
        // moved members of split classes before position q (w >= pw); a class's start and end
        auto moved_before = [&](int q) -> int {
            return q >= n ? m : st.nzpre[q >> 5] + __popc(st.touch[q >> 5] & st.flag[q >> 5] & lanes_below(q & 31));
        };
        auto class_start = [&](int q) -> int {
            const uint32_t b = st.start[q >> 5] & low_bits((q & 31) + 1);
            return b ? (q & ~31) + 31 - __clz(b) : st.last[(q >> 5) - 1];
        };
        auto class_end = [&](int q) -> int {
            const uint32_t b = st.start[q >> 5] & (0xFFFFFFFEu << (q & 31));
            return b ? (q & ~31) + __ffs(b) - 1 : (q >> 5) + 1 < wn ? st.next[(q >> 5) + 1] : n;
        };
        // ---- moved members listed, the others shifted to the end of their class
#pragma unroll 1
        for (int q0 = (i2 & ~(G - 1)) + G * t; q0 < n; q0 += G * T) {
            const int w = q0 >> 5, sh = q0 & 31;
            uint32_t f = (st.flag[w] >> sh) & low_bits(min(G, n - q0));
            if (!f) continue;
            const uint32_t nz = st.touch[w] & st.flag[w], nzw = nz >> sh, b = st.start[w] >> sh;
            int before = st.nzpre[w] + __popc(nz & lanes_below(sh));
            int s = -1, ms = 0, me = 0;   // the class at hand: its start, moved members before and up to its end
#pragma unroll 1
            for (; f; f &= f - 1u) {
                const int e = __ffs(f) - 1, q = q0 + e;
                if (s < 0 || ((b >> e) & 1u)) {
                    s = class_start(q);
                    ms = moved_before(s);
                    me = moved_before(class_end(q));
                }
                const Id v = st.perm[q];
                if (!((nzw >> e) & 1u)) {
                    st.tmp[q + me - before] = v;
                    continue;
                }
                if (r == 1) {
                    st.tmp[s + before - ms] = v;
                } else {
                    const uint32_t pk = pivot_key(st.key[key_slot(v)] & pm);
                    st.comp[before] = (unsigned long long)s << 44 | (unsigned long long)~pk << 12 | (unsigned)before;
                    st.lv[before] = v;
                    if (before == ms) atomicMax(&sc->nz_max, me - ms);
                }
                ++before;
            }
        }
        __syncthreads();
        // ---- the moved members in their new order
        if (r > 1) {
            if (sc->nz_max <= kPanelCount) {   // four lanes count the members of e's class before e
#pragma unroll 1
                for (int e0 = warp * 8; e0 < m; e0 += NW * 8) {
                    const int e = min(e0 + (lane >> 2), m - 1);
                    const unsigned long long c = st.comp[e];
                    const int s = (int)(c >> 44), lo = moved_before(s), hi = moved_before(class_end(s));
                    int rank = 0;
#pragma unroll 4
                    for (int k = lo + (lane & 3); k < hi; k += 4) rank += st.comp[k] < c ? 1 : 0;
                    rank += __shfl_xor_sync(kAll, rank, 1);
                    rank += __shfl_xor_sync(kAll, rank, 2);
                    if ((lane & 3) == 0) st.tmp[s + rank] = (Id)st.lv[e];
                }
            } else {
                int p = 64;
#pragma unroll 1
                while (p < m) p <<= 1;
#pragma unroll 1
                for (int e = m + t; e < p; e += T) st.comp[e] = ~0ull;
                __syncthreads();
                panel_sort<T>(st.comp, p);
#pragma unroll 1
                for (int e = t; e < m; e += T) {
                    const unsigned long long c = st.comp[e];
                    const int s = (int)(c >> 44);
                    st.tmp[s + e - moved_before(s)] = (Id)st.lv[c & 0xFFFu];
                }
            }
            __syncthreads();
        }
        // ---- back into perm, with the new boundaries (a warp's lanes share words: old ones are read first)
#pragma unroll 1
        for (int c = (i2 & ~(32 * G - 1)) + warp * 32 * G; c < n; c += T * G) {
            const int q0 = c + G * lane, w = q0 >> 5, sh = q0 & 31;
            uint32_t f = q0 < n ? (st.flag[w] >> sh) & low_bits(min(G, n - q0)) : 0u;
            const uint32_t bw = q0 < n ? st.start[w] : 0u;
            uint32_t fresh = 0u, kp = 0u;
            if (f & ~(bw >> sh) & 1u) kp = st.key[key_slot(st.tmp[q0 - 1])] & pm;
#pragma unroll 1
            for (; f; f &= f - 1u) {
                const int e = __ffs(f) - 1, q = q0 + e;
                const Id v = st.tmp[q];
                st.perm[q] = v;
                const uint32_t k = st.key[key_slot(v)] & pm;
                if (k != kp && !((bw >> (sh + e)) & 1u)) {
                    fresh |= 1u << e;
                    // the members that did not move keep the class's last adjacent pivot
                    if (ppos_out && k == 0u) {
                        const uint32_t le = bw & low_bits(sh + e + 1);
                        ppos[q] = __ldcg(&ppos[le ? (w << 5) + 31 - __clz(le) : st.last[w - 1]]);
                    }
                }
                kp = k;
            }
            if constexpr (G == 1) {
                const uint32_t nb = __ballot_sync(kAll, fresh != 0u);
                if (lane == 0 && nb) st.start[w] = bw | nb;
            } else {
                __syncwarp();
                if (fresh) reinterpret_cast<uint8_t *>(&st.start[w])[sh >> 3] = (uint8_t)((bw >> sh) | fresh);
            }
        }
        __syncthreads();
        break;
    }
    return i2;
}

// The panel's results; every class's last adjacent pivot (starts: not when a
// settled panel of steps has set them).  Returns the mask E_b to be written next.
template <int STATE, int T, typename PivotKey>
__device__ __forceinline__ int panel_results(int n, int i, int i2, int r, uint32_t pm, bool ident, bool starts,
                                             const PanelState<typename PanelId<STATE>::type> &st, PanelScalars *sc,
                                             int32_t *__restrict__ order, int32_t *__restrict__ pos, int32_t *ppos_out,
                                             const uint32_t *emask, const PivotKey &pivot_key) {
    using Id = typename PanelId<STATE>::type;
    constexpr int NW = T / 32;
    const int lane = threadIdx.x & 31, warp = warp_index();
    const int wn = (n + 31) >> 5;
    const auto ppos = cg_arr(ppos_out, n, kChkPpos);
    const int b2 = i2 >> 5;
    const int eb = emask && 32 * b2 > i && 32 * b2 < n ? b2 : 0;
    if (warp == 0 && lane < r) {
        const int v = sc->piv[lane];
        order[i + lane] = v;
        if (pos) pos[v] = i + lane;
        if (ppos_out) ppos[i + lane] = sc->par[lane];
        if (eb == 0 || i + lane < 32 * eb) atomicOr(&st.numbered[v >> 5], 1u << (v & 31));
    }
    if (ppos_out && starts) {   // (a split class's members have moved: its starts' keys are looked up)
        constexpr int U = 4;   // words at once, so that their gathers overlap
        const bool split = sc->any != 0;
#pragma unroll 1
        for (int w0 = (i2 >> 5) + warp; w0 < wn; w0 += U * NW) {
            Id v[U];
            uint32_t k[U], b[U];
            bool on[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int w = w0 + u * NW;
                b[u] = w < wn ? st.start[w] & (st.touch[w] | (split ? st.flag[w] : 0u)) : 0u;
            }
            if (!(b[0] | b[1] | b[2] | b[3])) continue;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = (min(w0 + u * NW, wn - 1) << 5) + lane;
                on[u] = q >= i2 && ((b[u] >> lane) & 1u);
                v[u] = st.perm[q];
            }
#pragma unroll
            for (int u = 0; u < U; ++u) k[u] = on[u] ? st.key[key_slot(v[u])] & pm : 0u;
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k[u])
                    ppos[((w0 + u * NW) << 5) + lane] = sc->piv[ident ? 31 - __clz(k[u]) : 32 - __ffs(pivot_key(k[u]))];
        }
    }
    return eb;
}

// The last panel's pivots after E_eb, after that has been written (warp 0).
template <typename Arr>
__device__ __forceinline__ void panel_complete_mask(const PanelScalars *sc, int i, int eb, const Arr &numbered) {
    const int lane = threadIdx.x & 31;
    if (lane < sc->r && i - sc->r + lane >= 32 * eb) atomicOr(&numbered[sc->piv[lane] >> 5], 1u << (sc->piv[lane] & 31));
}

// A row's words of thread t: the neighbours without a seen bit are listed (the
// first 32 of them; *count: how many there are).
template <int T, int B, typename Arr>
__device__ __forceinline__ void panel_scan_row(const uint32_t *__restrict__ row, int wn, int t, const Arr &seen,
                                               uint32_t *list, int *count) {
#pragma unroll 1
    for (int w0 = t; w0 < wn; w0 += B * T) {
        uint32_t rw[B];
#pragma unroll
        for (int u = 0; u < B; ++u) rw[u] = w0 + u * T < wn ? row[w0 + u * T] : 0u;
#pragma unroll
        for (int u = 0; u < B; ++u) {
            if (w0 + u * T >= wn) break;
#pragma unroll 1
            for (uint32_t nb = rw[u] & ~(uint32_t)seen[w0 + u * T]; nb; nb &= nb - 1u) {
                const int k = atomicAdd(count, 1);
                if (k < 32) list[k] = (uint32_t)(32 * (w0 + u * T) + __ffs(nb) - 1);
            }
        }
    }
}

// Up to 32 pivots one by one, from position i on.  Warp 0 keeps a lane per vertex
// that has met a pivot and is not numbered yet (its label in this panel; at most
// 32 of them at any time, else the panel ends before the pivot that meets more).
// A step reads the pivot's row (warp 0 alone, or, rows of more than 4 words per
// lane, all threads between two barriers), adds its bit to the adjacent lanes'
// labels and gives the vertices met first to free lanes; the next pivot is the
// lane of the class at hand with the largest label, or the class's first member
// that has not been met; a class that is used up gives way to the next one.
// What is left of the last class makes room in front for its pivots and, when no
// other class has any, for its members that were met, in their new classes.  Then
// the panel is settled: there is nothing left to split.  Otherwise the keys are
// completed and the caller splits the classes as after a window.
// The masks of vertices lie in arrays that the split passes use too; the mask of
// the last class's members is kept from panel to panel (ls: where that class
// starts, -1: the mask is to be built).
// Returns the number of pivots (| kPanelSettled), 0: the first one meets too many.
// A step is about 1,000 cycles of latency in one warp, 600 of them the row's load.
// Steps by all threads, keys in shared memory and a CTA-wide maximum took 1,500 at
// n = 1,000; requesting the likely next row a step ahead made a path a third slower
// and disjoint K4 no faster; a walking warp that differs from CTA to CTA, 5% slower.
template <int STATE, int T>
__device__ __forceinline__ int panel_steps(const uint32_t *__restrict__ rows, int stride, int n, int i,
                                           const PanelState<typename PanelId<STATE>::type> &st, PanelScalars *sc,
                                           int32_t *ppos_out, int &ls) {
    const auto ppos = cg_arr(ppos_out, n, kChkPpos);
    using Id = typename PanelId<STATE>::type;
    constexpr int NW = T / 32;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    constexpr int B = 4;   // words of a row in flight per thread
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    const int wn = (n + 31) >> 5;
    const auto &done = st.dpre, &seen = st.last, &last = st.next;   // numbered; or met; members of the last class
    const bool build = ls < 0;
    if (build) {
        for (int w0 = (wn - 1) & ~31; ls < 0; w0 -= 32) {   // (position 0 or i starts a class)
            const uint32_t b = w0 + lane < wn ? st.start[w0 + lane] : 0u, any = __ballot_sync(kAll, b != 0u);
            if (any) ls = 32 * (w0 + 31 - __clz(any)) + 31 - __clz(__shfl_sync(kAll, b, 31 - __clz(any)));
        }
        ls = max(ls, i);
    }
#pragma unroll 1
    for (int w = t; w < wn; w += T) {
        const int d = (int)(st.numbered[w] | (w == wn - 1 && (n & 31) ? ~low_bits(n & 31) : 0u));
        last[w] = build ? 0 : last[w] & ~seen[w];
        seen[w] = d;
        done[w] = d;
    }
    __syncthreads();
    if (build) {
#pragma unroll 1
        for (int q0 = (ls & ~7) + 8 * t; q0 < n; q0 += 8 * T) {   // members are in id order: few words per thread
            Panel8<Id> v;
            v.load(&st.perm[q0]);
            int word = -1;
            uint32_t bits = 0u;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (q0 + e < ls || q0 + e >= n) continue;
                const int w = (int)(v[e] >> 5);
                if (w != word && bits) atomicOr(&last[word], (int)bits);
                if (w != word) word = w, bits = 0u;
                bits |= 1u << (v[e] & 31);
            }
            if (bits) atomicOr(&last[word], (int)bits);
        }
        __syncthreads();
    }

    const bool all = wn > 32 * B;   // all threads read the rows
    uint32_t *list = reinterpret_cast<uint32_t *>((unsigned long long *)st.comp);   // [32] the vertices met first
    if (warp == 0) {
        int y = -1;             // the lane's vertex, its label in pivot order (the first pivot highest),
        uint32_t ky = 0u;       // and whether it is of the class at hand
        bool in = false;
        int cs = i, ce = n, q = i, own = -1;   // the class at hand; its members from position q on; its last adjacent pivot
        int mem = -1;
        auto in_class = [&](int v) -> bool {
            if (ce == n) return v >= 0 && ((last[v >> 5] >> (v & 31)) & 1);
            bool hit = false;
            if (ce - cs <= 32) {
#pragma unroll 1
                for (int k = 0; k < ce - cs; ++k) hit |= __shfl_sync(kAll, mem, k) == v;
                return hit;
            }
            int lo = cs, hi = ce - 1;
#pragma unroll 1
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if ((int)st.perm[mid] < v) lo = mid + 1; else hi = mid;
            }
            return (int)st.perm[lo] == v;
        };
        auto members = [&]() { mem = q + lane < ce ? (int)st.perm[q + lane] : -1; };
        auto enter = [&](int s) {
            cs = q = s;
            ce = n;
            if (ppos_out) own = __ldcg(&ppos[s]);
#pragma unroll 1
            for (int w0 = s >> 5; w0 < wn; w0 += 32) {
                const int w = w0 + lane;
                uint32_t b = w < wn ? st.start[w] : 0u;
                if (w == (s >> 5)) b &= 0xFFFFFFFEu << (s & 31);
                const uint32_t any = __ballot_sync(kAll, b != 0u);
                if (any) {
                    const int l = __ffs(any) - 1;
                    ce = 32 * (w0 + l) + __ffs(__shfl_sync(kAll, b, l)) - 1;
                    break;
                }
            }
            members();
            in = in_class(y);
        };
        enter(i);
        int r = 0, x = __shfl_sync(kAll, mem, 0);   // no label yet: the lowest id
        uint32_t label = 0u;
#pragma unroll 1
        for (;;) {
            const uint32_t *row = rows + (size_t)x * stride;
            const bool mine = y == x;   // (no lane when the pivot has not been met)
            if (mine) y = -1;
            const uint32_t aw = y >= 0 ? row[y >> 5] : 0u;
            uint32_t rw[B];
            if (!all) {   // (the bookkeeping below hides part of the loads)
#pragma unroll
                for (int u = 0; u < B; ++u) rw[u] = lane + 32 * u < wn ? row[lane + 32 * u] : 0u;
            }
            if (lane == 0) {
                sc->piv[r] = x;
                done[x >> 5] |= 1 << (x & 31);
                seen[x >> 5] |= 1 << (x & 31);
                sc->nz_max = 0;
                sc->cend = x;
                sc->par[r] = label ? sc->piv[32 - __ffs((int)label)] : own;
            }
            int met = 0;
            if (all) {
                named_barrier(1, T);   // the others read the row with this warp
                panel_scan_row<T, B>(row, wn, t, seen, list, &sc->nz_max);
                named_barrier(1, T);
                met = sc->nz_max;
            } else {
                __syncwarp();
                uint32_t sw[B];
#pragma unroll
                for (int u = 0; u < B; ++u) sw[u] = lane + 32 * u < wn ? (uint32_t)seen[lane + 32 * u] : ~0u;
#pragma unroll
                for (int u = 0; u < B; ++u) {
                    if (32 * u >= wn) break;
                    uint32_t nb = rw[u] & ~sw[u];
#pragma unroll 1
                    for (;;) {
                        const uint32_t b = __ballot_sync(kAll, nb != 0u);
                        if (!b) break;
                        const int k = met + __popc(b & lanes_below(lane));
                        if (nb && k < 32) list[k] = (uint32_t)(32 * (lane + 32 * u) + __ffs(nb) - 1);
                        nb &= nb - 1u;
                        met += __popc(b);
                    }
                }
                __syncwarp();
            }
            const uint32_t room = __ballot_sync(kAll, y < 0);
            if (met > __popc(room)) {   // the panel ends before x
                if (lane == 0) {
                    done[x >> 5] &= ~(1 << (x & 31));
                    if (!label) seen[x >> 5] &= ~(1 << (x & 31));
                }
                if (mine) y = x;
                break;
            }
            const uint32_t bit = 0x80000000u >> r;
            if (y >= 0 && ((aw >> (y & 31)) & 1u)) ky |= bit;
            if (met) {
                const int k = __popc(room & lanes_below(lane));
                const bool fresh = y < 0 && k < met;
                if (fresh) {
                    y = (int)list[k];
                    ky = bit;
                    atomicOr(&seen[y >> 5], 1 << (y & 31));
                }
                const bool c = in_class(y);
                if (fresh) in = c;
                __syncwarp();
            }
            ++r;
            if (r == 32 || i + r == n) break;
            // ---- the next pivot
#pragma unroll 1
            for (;;) {
                label = __reduce_max_sync(kAll, y >= 0 && in ? ky : 0u);
                if (label) {
                    x = (int)__reduce_min_sync(kAll, y >= 0 && in && ky == label ? (unsigned)y : kNoVertex);
                    break;
                }
                uint32_t ok;
                __syncwarp();
#pragma unroll 1
                for (;;) {   // the first member not met
                    ok = __ballot_sync(kAll, mem >= 0 && !((seen[max(mem, 0) >> 5] >> (mem & 31)) & 1));
                    if (ok || q + 32 >= ce) break;
                    q += 32;
                    members();
                }
                if (ok) {
                    x = __shfl_sync(kAll, mem, __ffs(ok) - 1);
                    break;
                }
                enter(i + r);
            }
        }
        const uint32_t cand = __ballot_sync(kAll, y >= 0), away = __ballot_sync(kAll, y >= 0 && !in);
        const bool rest = i + r < ce;   // something is left of the class at hand
        __syncwarp();
        if (y >= 0)
            st.comp[__popc(cand & lanes_below(lane))] = (unsigned long long)ky << 32 | (uint32_t)~y;
        if (lane == 0) {
            sc->r = r;
            sc->cend = all ? -1 : 0;   // (the others leave their loop)
            sc->ident = own;
            sc->nz_max = __popc(cand);
            sc->ub = away || (cand && !rest) ? 1u : 0u;
            sc->scan[0][0] = cs;   // (these stay as they are until all have read them)
            sc->scan[0][1] = ce;
        }
        if (all) named_barrier(1, T);
    } else if (all) {
#pragma unroll 1
        for (;;) {
            named_barrier(1, T);
            const int x = sc->cend;
            if (x < 0) break;
            panel_scan_row<T, B>(rows + (size_t)x * stride, wn, t, seen, list, &sc->nz_max);
            named_barrier(1, T);
        }
    }
    __syncthreads();
    const int r = sc->r, cs = sc->scan[0][0], ce = sc->scan[0][1], own = sc->ident, met = sc->nz_max;
    const bool settled = sc->ub == 0u;
    if (r == 0) return 0;
    const int i2 = i + r, p = i2 - cs, s = settled ? met : 0;   // pivots of the last class; members that leave it with them
    // ---- the class's other members move up to i2 + s..ce-1
    auto leaving = [&](int q0, const Panel8<Id> &v) -> uint32_t {   // which of eight positions' members leave
        uint32_t out = 0u;
#pragma unroll
        for (int e = 0; e < 8; ++e)
            if (q0 + e >= cs && q0 + e < ce) {
                const int w = (int)(v[e] >> 5);
                out |= (((uint32_t)(s ? seen[w] : done[w]) >> (v[e] & 31)) & 1u) << e;
            }
        return out;
    };
    auto lanes_after = [&](uint32_t out) -> int {   // how many leave at the higher lanes' positions
        int a = __popc(out);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_down_sync(kAll, a, o);
            if (lane + o < 32) a += u;
        }
        return a - __popc(out);
    };
    if (i2 < ce && p + s > 0) {
        // NW chunks of 256 positions at a time, from the end: all of them are read before any is written, and a
        // member moves to where all has been read
        int gone = 0, slot = 0;   // members that leave from higher positions
        int *counts = sc->scan[1];   // [2][32]
        static_assert(sizeof(sc->scan) >= 96 * sizeof(int), "two slots of warp counts");
#pragma unroll 1
        for (int top = ((ce - 1) & ~255) + 256; top > cs; top -= 256 * NW, slot ^= 1) {
            const int q0 = top - 256 * (warp + 1) + 8 * lane;   // (warp 0: the highest)
            Panel8<Id> v{};
            uint32_t out = 0u;
            if (q0 < ce && q0 + 8 > cs) {
                v.load(&st.perm[q0]);
                out = leaving(q0, v);
            }
            const int chunk = __reduce_add_sync(kAll, __popc(out));
            if (lane == 0) counts[32 * slot + warp] = chunk;
            __syncthreads();
            const int c = lane < NW ? counts[32 * slot + lane] : 0;
            int k = gone + __reduce_add_sync(kAll, lane < warp ? c : 0);
            gone += __reduce_add_sync(kAll, c);
            if (k + chunk == 0) continue;
            k += lanes_after(out);
#pragma unroll
            for (int e = 7; e >= 0; --e) {
                if ((out >> e) & 1u) ++k;
                else if (k && q0 + e >= cs && q0 + e < ce) st.perm[q0 + e + k] = (Id)v[e];
            }
        }
        __syncthreads();
    }
    if (warp == 0) {
        if (lane < s) {
            const unsigned long long mine = st.comp[lane];
            int rank = 0;
            bool first = true;   // of its new class
#pragma unroll 1
            for (int k = 0; k < s; ++k) {
                const unsigned long long o = st.comp[k];
                rank += o > mine ? 1 : 0;
                if (o > mine && (o >> 32) == (mine >> 32)) first = false;
            }
            const int q = i2 + rank;
            st.perm[q] = (Id)~(uint32_t)mine;
            if (first) {
                atomicOr(&st.start[q >> 5], 1u << (q & 31));
                if (ppos_out) ppos[q] = sc->piv[32 - __ffs((int)(mine >> 32))];
            }
        }
        if (lane < r) st.perm[i + lane] = (Id)sc->piv[lane];
        __syncwarp();
        const int q = i2 + s;   // the first member without a label of this panel
        if (lane == 0 && q < ce && !((st.start[q >> 5] >> (q & 31)) & 1u)) {
            atomicOr(&st.start[q >> 5], 1u << (q & 31));
            if (ppos_out) ppos[q] = own;
        }
    }
    if (settled) {
        if (ce == n) ls = i2 + s < n ? i2 + s : -1;   // (the mask loses the members seen)
    } else {
        ls = -1;
#pragma unroll 1
        for (int w = t; w < wn; w += T)
#pragma unroll
            for (int c = 0; c < 8; ++c) *reinterpret_cast<uint4 *>(&st.key[32 * w + 4 * c]) = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        if (t < met) {
            const unsigned long long c = st.comp[t];
            st.key[key_slot((uint32_t)~(uint32_t)c)] = __brev((uint32_t)(c >> 32));
        }
    }
    __syncthreads();
    return settled ? r | kPanelSettled : r;
}

// Panels of steps: at most `panels`, fewer when one numbers few vertices.  Returns
// the numbered vertices.
template <int STATE, int T>
__device__ __forceinline__ int panel_narrow(const uint32_t *__restrict__ rows, int stride, int n, int i, int cap,
                                         unsigned char *gstate, int32_t *__restrict__ order,
                                         int32_t *__restrict__ pos, int32_t *ppos_out, uint32_t *emask, int panels) {
    extern __shared__ __align__(16) unsigned char smem[];
    PanelScalars *sc = reinterpret_cast<PanelScalars *>(smem);
    const auto st = panel_carve<STATE>(smem + kPanelScalarBytes, gstate, n, cap);
    const int t = threadIdx.x, warp = warp_index();
    const auto pivot_key = [](uint32_t k) { return __brev(k); };   // the pivots are the key's bits in order
    int eb = 0, ls = -1;
#pragma unroll 1
    for (int r = 32; panels > 0 && i < n && r >= kStepsBelow; --panels) {
        if (eb > 0) panel_write_mask<T>(emask, eb, n, st.numbered);
        if (t == 0) sc->any = 0;
        __syncthreads();
        if (eb > 0) {
            if (warp == 0) panel_complete_mask(sc, i, eb, st.numbered);
            __syncthreads();
        }
        r = panel_steps<STATE, T>(rows, stride, n, i, st, sc, ppos_out, ls);
        if (r == 0) {
            eb = 0;
            break;
        }
        const bool settled = (r & kPanelSettled) != 0;
        r &= ~kPanelSettled;
        int i2 = i + r;
        uint32_t pm = low_bits(r);
        bool ident = true;
        if (!settled) i2 = panel_split<STATE, T>(n, i, st, sc, ppos_out, r, pm, ident, pivot_key, [] {});
        eb = panel_results<STATE, T>(n, i, i2, r, pm, true, !settled, st, sc, order, pos, ppos_out, emask, pivot_key);
        i = i2;
        __syncthreads();
    }
    if (eb > 0) {
        panel_write_mask<T>(emask, eb, n, st.numbered);
        __syncthreads();
        if (warp == 0) panel_complete_mask(sc, i, eb, st.numbered);
        __syncthreads();
    }
    return i;
}

// Panels of a window each, from position i on, until all vertices are numbered or
// the windows have fallen short (lost) of too many pivots.  Returns the numbered
// vertices.
template <int STATE, int T>
__device__ __forceinline__ int panel_windows(const uint32_t *__restrict__ rows, int stride, int n, int i, int cap,
                                             unsigned char *gstate, int32_t *__restrict__ order,
                                             int32_t *__restrict__ pos, int32_t *ppos_out, uint32_t *emask, int &lost,
                                             int &span) {
    extern __shared__ __align__(16) unsigned char smem[];
    PanelScalars *sc = reinterpret_cast<PanelScalars *>(smem);
    const auto st = panel_carve<STATE>(smem + kPanelScalarBytes, gstate, n, cap);
    using Id = typename PanelId<STATE>::type;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    const int wn = (n + 31) >> 5;
    const auto ppos = cg_arr(ppos_out, n, kChkPpos);
    int eb = 0;   // E_eb is to be written at the start of the next panel (0: none)
    while (i < n) {
        const int w2 = min(32, n - i);
        const int vk = lane < w2 ? (int)st.perm[i + lane] : 0;
        // the window's classes (read before warp 0 may set a start for the next panel)
        const uint32_t starts =
            __funnelshift_r(st.start[i >> 5], (i >> 5) + 1 < wn ? st.start[(i >> 5) + 1] : 0u, i & 31) & low_bits(w2);
        const bool straddle = i + w2 < n && !((st.start[(i + w2) >> 5] >> ((i + w2) & 31)) & 1u);
        int cp = -1;   // warp 0: the classes' last adjacent pivots, requested early
        if (warp == 0 && ppos_out && lane < w2) cp = __ldcg(&ppos[i + lane]);
        if (eb > 0) panel_write_mask<T>(emask, eb, n, st.numbered);
        reinterpret_cast<uint32_t *>(sc->row4)[lane] = 4u * (uint32_t)vk;
        __syncwarp();
        // ---- keys: a word of vertices per thread and pass
#pragma unroll 1
        for (int wb = warp * 32; wb < wn; wb += T) {
            const int w = wb + lane;
            const bool on = w < wn && st.numbered[w] != kAll;   // some vertex still to come
            if (!__any_sync(kAll, on)) continue;
            // (rows past w2 are row 0: no one reads the key bits beyond the window's vertices)
            uint32_t r[32];
            panel_load_rows(rows + (on ? w : 0), stride, sc->row4, r);
            transpose32(r);
            if (on) {
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4 *>(&st.key[32 * w + ((c ^ (w & 7)) << 2)]) =
                        make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
            }
        }
        if (t == 0) sc->any = 0;
        __syncthreads();
        if (warp == 0 && eb > 0) panel_complete_mask(sc, i, eb, st.numbered);

        // ---- the pivots: window vertices 0..r-1 in order, or what warp 0 finds
        const uint32_t adj = lane < w2 ? st.key[key_slot(vk)] : 0u;   // window vertex `lane` in the window
        int mypos = -1, la = -1;   // warp 0
        auto commit = [&](int r) {
            const bool ident = __ballot_sync(kAll, mypos >= 0 && mypos != lane) == 0u;
            const uint32_t taken = __ballot_sync(kAll, mypos >= 0), left = low_bits(w2) & ~taken;
            const int own = __shfl_sync(kAll, cp, 31 - __clz((starts | 1u) & low_bits(lane + 1)));   // its class's value
            const int cl = left ? __ffs(left) - 1 : w2 - 1;   // a member of the class that goes on at position i + r
            const int cpl = __shfl_sync(kAll, own, cl);
            if (mypos >= 0) sc->piv[mypos] = vk;
            if (!ident) {
                const int dest = mypos >= 0 ? mypos : r + __popc(left & lanes_below(lane));
                if (lane < w2) st.perm[i + dest] = (Id)vk;
                sc->bit[lane] = mypos >= 0 ? 0x80000000u >> mypos : 0u;
            }
            __syncwarp();
            if (mypos >= 0) sc->par[mypos] = la >= 0 ? sc->piv[la] : own;
            if (lane == 0) {
                const int i2 = i + r;
                int set = -1;
                if (i2 < n && !((st.start[i2 >> 5] >> (i2 & 31)) & 1u)) {
                    st.start[i2 >> 5] |= 1u << (i2 & 31);
                    set = i2;
                    if (ppos_out) ppos[i2] = cpl;
                }
                sc->set_start = set;
                sc->r = r;
                sc->pivmask = taken;
                sc->ident = ident ? 1 : 0;
            }
        };
        auto commit_in_order = [&](int r) {
            mypos = lane < r ? lane : -1;
            const uint32_t before = adj & lanes_below(lane);
            la = before ? 31 - __clz(before) : -1;
            commit(r);
        };
        uint32_t ub = kAll;
        bool order_fails;
        int r = panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
        bool ident = true;
        if (r < w2 && r < kPanelFew) {   // too few (the same in every warp)
            if (!order_fails) {          // stopped by the class that goes on beyond the window: look at it
                if (t == 0) {
                    sc->cend = n;
                    sc->ub = 0u;
                }
                __syncthreads();
                const int q0 = i + w2;
#pragma unroll 1
                for (int w = (q0 >> 5) + t; w < wn; w += T) {
                    const uint32_t b = st.start[w] & (w == (q0 >> 5) ? kAll << (q0 & 31) : kAll);
                    if (b) {
                        atomicMin(&sc->cend, 32 * w + __ffs(b) - 1);
                        break;
                    }
                }
                __syncthreads();
                const int ce = sc->cend;
                uint32_t any = 0u;
#pragma unroll 1
                for (int q = q0 + t; q < ce; q += T) any |= st.key[key_slot(st.perm[q])];
                any = __reduce_or_sync(kAll, any);
                if (lane == 0 && any) atomicOr(&sc->ub, any);
                __syncthreads();
                ub = sc->ub;
                r = panel_in_order(lane, w2, starts, straddle, adj, ub, &order_fails);
            }
            ident = !(order_fails && r < kPanelFew);
        }
        uint32_t pm = low_bits(r);
        if (ident) {
            if (warp == 0) commit_in_order(r);
        } else {
            __syncthreads();   // every warp has read ub
            if (warp == 0) commit(panel_solve(lane, w2, starts, straddle, adj, ub, &mypos, &la));
            __syncthreads();
            r = sc->r;
            pm = sc->pivmask;
            ident = sc->ident != 0;
        }
        if (r >= kStepsBelow) {
            lost = max(lost + kStepsBelow - r, 0);
            span = 1;
        } else if (__reduce_max_sync(kAll, __popc(adj)) <= kStepsDegree) {
            lost += kStepsBelow - r;
        }

        // a key's bits in pivot order, the first pivot's highest
        auto pivot_key = [&](uint32_t k) -> uint32_t {
            if (ident) return __brev(k);
            uint32_t v = 0u;
    #pragma unroll
            for (int b = 0; b < 8; ++b) v |= sc->tab[b][(k >> (4 * b)) & 15u];
            return v;
        };
        const int i2 = panel_split<STATE, T>(n, i, st, sc, ppos_out, r, pm, ident, pivot_key, [&] {
            if (!ident && lane < w2) st.perm[i + lane] = (Id)vk;
            __syncwarp();
            commit_in_order(1);
        });
        eb = panel_results<STATE, T>(n, i, i2, r, pm, ident, true, st, sc, order, pos, ppos_out, emask, pivot_key);
        i = i2;
        __syncthreads();
        if (lost > panel_lost_limit(n)) break;
    }
    if (eb > 0) {
        panel_write_mask<T>(emask, eb, n, st.numbered);
        if (i < n) {
            __syncthreads();
            if (warp == 0) panel_complete_mask(sc, i, eb, st.numbered);
            __syncthreads();
        }
    }
    return i;
}

// One CTA computes the LexBFS order of one graph (rows: n rows of `stride`
// words in global memory; gstate: this CTA's workspace).  order gets the vertices
// by position; pos (nullable) its inverse; ppos (nullable) p(order[i]) by position
// (-1: none), exact; emask (nullable) the masks E_b, b >= 1, rows of
// mask_stride(n) words.
template <int STATE, int T>
__device__ __forceinline__ void lexbfs_panels(const uint32_t *__restrict__ rows, int stride, int n, int cap,
                                              unsigned char *gstate, int32_t *__restrict__ order,
                                              int32_t *__restrict__ pos, int32_t *ppos_out, uint32_t *emask) {
    if (n <= 0) return;   // (ppos has no entry then: a batch packs the next graph's there)
    extern __shared__ __align__(16) unsigned char smem[];
    {
        const auto st = panel_carve<STATE>(smem + kPanelScalarBytes, gstate, n, cap);
        using Id = typename PanelId<STATE>::type;
        const int t = threadIdx.x, wn = (n + 31) >> 5;
#pragma unroll 1
        for (int q = t; q < 32 * wn; q += T) st.perm[q] = (Id)q;   // positions past n too: they are read in eights
#pragma unroll 1
        for (int w = t; w < wn; w += T) {
            st.start[w] = w == 0 ? 1u : 0u;
            st.diff[w] = 0u;
            st.touch[w] = 0u;
            st.flag[w] = 0u;
            st.numbered[w] = 0u;
        }
        if (t == 0 && ppos_out) cg_arr(ppos_out, n, kChkPpos)[0] = -1;
        __syncthreads();
    }
    // windows as long as they pay, then a panel of steps, windows again, four panels of steps, and so on
    int lost = 0, span = 1;
#pragma unroll 1
    for (int i = 0;;) {
        i = panel_windows<STATE, T>(rows, stride, n, i, cap, gstate, order, pos, ppos_out, emask, lost, span);
        if (i >= n) return;
        const int i0 = i;
        i = panel_narrow<STATE, T>(rows, stride, n, i, cap, gstate, order, pos, ppos_out, emask, span);
        span = min(4 * span, kStepsMost);
        // the next window that does not pay is the last one, unless the steps did not pay either
        lost = i - i0 < kStepsBelow ? 0 : panel_lost_limit(n);
    }
}

}  // namespace cg
