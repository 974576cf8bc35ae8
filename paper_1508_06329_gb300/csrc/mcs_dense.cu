// mcs_dense.cu — Maximum Cardinality Search on dense graphs, one CTA.
//
// Method (Section 5.1; Tarjan and Yannakakis): every unnumbered vertex carries
// the number of its numbered neighbours; each step numbers a vertex with the
// largest count (lowest id among equals, as for LexBFS) and counts it at its
// unnumbered neighbours.  By Theorem 5.2 the graph is chordal iff the MCS
// order is a perfect elimination order, so the same check follows.
//
// One step at a time (mcs_step_kernel) is a latency chain of a row load, a
// CTA-wide maximum and a barrier per vertex.  Large graphs begin in panels of up
// to 32 pivots (mcs_panel_kernel).  A panel takes the 32 vertices with the
// largest (count, id) as a window and runs MCS on them alone:
//   1. sixteen warps read the window's rows and transpose them in registers:
//      vertex y's key, bit j = adjacent to window vertex j; meanwhile the last
//      warp, one lane per window vertex, visits the window;
//   2. a vertex outside the window comes into it before step j when its count
//      plus its neighbours among the first j pivots beats pivot j: the first
//      such step ends the panel.  Only vertices whose count is within 32 of the
//      least pivot's are looked at, then eight steps at a time;
//   3. the counts of all vertices grow by their neighbours among the r pivots,
//      and the next window is found: the 32nd largest of the maxima over 128
//      groups of vertices (strided, so that neighbouring ids fall into different
//      ones) is a bound that at least 32 vertices reach, usually about 130,
//      which are ranked by counting; when more than kMcsCand reach it, the
//      bound is bisected.
// A panel numbers about 31 vertices on dense chordal graphs, 10 on G(n, 1/2) (5 to
// 7 of the first ones) and fewer on sparse ones, and costs as much as kMcsWorth
// steps (13 us against 0.92 us a step at n = 16,384; below about 8,000 vertices
// steps are too cheap to beat).  So the panels keep count of what they gained; when
// they have lost kMcsPatience steps, they leave the rest to mcs_step_kernel.
// n = 16,384 at density 0.1: 15.1 -> 6.7 ms, 9,000 at density 0.05 6.0 -> 3.0, a clique of 9,000 16.0 -> 8.4;
// G(n, p), which soon goes on in steps: G(15,000, 1/2) 17.4 -> 17.5, G(10,000, 1/2) 9.9 -> 10.1.
#include <algorithm>

#include "kernels.h"
#include "lexbfs_dense.cuh"

namespace cg {

namespace {

constexpr int kMcsMaxN = 65520;
constexpr int kMcsWorkers = 512;                // threads that hold vertices
constexpr int kMcsThreads = kMcsWorkers + 32;   // and the warp that visits the window
constexpr int kMcsGroups = 128;
constexpr int kMcsCand = 512;
constexpr size_t kMcsSmemRows = 200 * 1024;     // dynamic shared memory limit for the row copy
constexpr int kMcsPanelMin = 8192, kMcsPanelMax = 36608;   // keys and counts in shared memory
constexpr int kMcsWorth = 20;                   // steps that cost as much as a panel (13 to 18 us)
// The panels stop when they have lost this many steps (the first panel, which has no counts to go by, aside), or,
// after many that paid, this many and kMcsCredit more.  The second panel of G(n, p) numbers 5 vertices, that of the
// subtree-intersection graphs 10 to 32: one look is enough, and a panel of G(10,000, 1/2) costs 35 us.
constexpr int kMcsPatience = 12, kMcsCredit = 63;

// What the panels leave to the steps.
struct alignas(16) McsLeft {
    int i, x;          // numbered vertices; the next pivot
    int pad[2];
    alignas(16) uint16_t cnt[8];   // [32 * ceil(n / 32)] counts as the panels keep them
};

struct McsShared {
    uint4 row4[8];                // four times the window's vertices
    int v[32];                    // the window, largest (count, id) first
    int cnt[32];
    uint32_t mask[33];            // window vertices among the first j pivots
    unsigned beat[32];            // (count, id) of pivot j when it is visited
    uint32_t mask8[4];            // first 8, 16, 24, 32 pivots; the least beat of these steps
    unsigned beat8[4];
    int piv[32];
    int r;                        // pivots of the panel
    alignas(16) unsigned group[kMcsGroups];   // maxima of (count, id)
    unsigned bound;
    int ncand;
    unsigned cand[kMcsCand];
    uint16_t near_v[kMcsWorkers / 32][256];   // a warp's vertices to look at (of a chunk)
};

// (count, id) as one number: larger counts first, lower ids among equals.
__device__ __forceinline__ unsigned mcs_comp(unsigned c, unsigned v) { return c << 16 | (65535u - v); }

__global__ void __launch_bounds__(kMcsThreads, 1) mcs_panel_kernel(DenseDesc d, int32_t *__restrict__ order,
                                                                  int32_t *__restrict__ pos, McsLeft *left) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ McsShared sh;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int t = threadIdx.x, lane = t & 31, warp = warp_index();
    const bool worker = warp < kMcsWorkers / 32;
    const int n = d.n, wn = (n + 31) >> 5;
    const uint32_t *__restrict__ rows = d.rows;
    uint32_t *key = reinterpret_cast<uint32_t *>(smem);                        // [32 * wn]
    uint16_t *cnt = reinterpret_cast<uint16_t *>(smem + (size_t)wn * 128);   // [32 * wn]
    prefetch_range_l2<kMcsThreads>(rows, (size_t)n * d.words * sizeof(uint32_t));
#pragma unroll 1
    for (int v = t; v < 32 * wn; v += kMcsThreads) cnt[v] = v < n ? 1 : 0;
    if (t < 32) {
        sh.v[t] = t;
        sh.cnt[t] = 1;
        reinterpret_cast<unsigned *>(sh.row4)[t] = 4u * min(t, n - 1);
    }
    __syncthreads();

    int credit = 0, panels = 0;
    for (int i = 0; i < n;) {
        const int w2 = min(32, n - i);
        int mycnt = 0, myv = 0, mypos = -1;   // last warp: its lane's window vertex
        uint32_t adj = 0u;
        // eight neighbouring vertices' counts and keys
        auto load8 = [&](int q, uint16_t (&c)[8], uint32_t (&k)[8]) {
            panel_load8(cnt + 8 * q, c);
            const int w = q >> 2, p = (q & 3) << 1;
            const uint4 a = *reinterpret_cast<const uint4 *>(&key[32 * w + ((p ^ (w & 7)) << 2)]);
            const uint4 b = *reinterpret_cast<const uint4 *>(&key[32 * w + (((p + 1) ^ (w & 7)) << 2)]);
            k[0] = a.x, k[1] = a.y, k[2] = a.z, k[3] = a.w, k[4] = b.x, k[5] = b.y, k[6] = b.z, k[7] = b.w;
        };

        // ---- keys, and the window visited by the last warp
        if (worker) {
#pragma unroll 1
            for (int wb = warp * 32; wb < wn; wb += kMcsWorkers) {
                const int w = wb + lane;
                uint32_t r[32];
                panel_load_rows(rows + min(w, wn - 1), d.words, sh.row4, r);   // (key bits from w2 on: not read)
                transpose32(r);
                if (w < wn) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<uint4 *>(&key[32 * w + ((c ^ (w & 7)) << 2)]) =
                            make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
                }
            }
            if (t < kMcsGroups) sh.group[t] = 0u;
        } else {
            myv = lane < w2 ? sh.v[lane] : 0;
            mycnt = sh.cnt[lane];
            uint32_t a[32];
            panel_load_rows(rows + (myv >> 5), d.words, sh.row4, a);
#pragma unroll
            for (int j = 0; j < 32; ++j) adj |= ((a[j] >> (myv & 31)) & 1u) << j;
            adj &= ~(1u << lane);
            if (lane < w2) cnt[myv] = 0;
            unsigned comp = lane < w2 ? mcs_comp(mycnt, myv) : 0u;
            uint32_t done = 0u, before = 0u;   // lane j keeps step j
            unsigned beat = kAll;
#pragma unroll 1
            for (int j = 0; j < w2; ++j) {
                const unsigned best = __reduce_max_sync(kAll, comp);
                const uint32_t at = __ballot_sync(kAll, comp == best);
                if (lane == j) {
                    before = done;
                    beat = best;
                }
                comp = comp == best ? 0u : comp ? comp + ((adj & at) ? 0x10000u : 0u) : 0u;
                if (at == (1u << lane)) mypos = j;
                done |= at;
            }
            sh.mask[lane] = lane < w2 ? before : done;
            sh.beat[lane] = beat;
            // eight steps at a time: the pivots before the next eight, the least beat
            const uint32_t m8 = __shfl_down_sync(kAll, before, 1);
            unsigned b8 = min(beat, __shfl_xor_sync(kAll, beat, 1));
            b8 = min(b8, __shfl_xor_sync(kAll, b8, 2));
            b8 = min(b8, __shfl_xor_sync(kAll, b8, 4));
            if ((lane & 7) == 7) {
                sh.mask8[lane >> 3] = lane + 1 < w2 ? m8 : done;
                sh.beat8[lane >> 3] = b8;
            }
            if (lane == 0) {
                sh.mask[32] = done;
                sh.r = w2;
                sh.ncand = 0;
                sh.bound = 0u;
            }
            if (mypos >= 0) sh.piv[mypos] = myv;
        }
        __syncthreads();
        // ---- the first step at which a vertex outside the window would be visited
        uint32_t m8[4];
        unsigned b8[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) m8[k] = sh.mask8[k], b8[k] = sh.beat8[k];
        const int least = (int)(min(min(b8[0], b8[1]), min(b8[2], b8[3])) >> 16);
        const unsigned near = max(least - 32, 1);
        int r = w2;
        if (worker) {
            {
                uint16_t *near_v = sh.near_v[warp];
#pragma unroll 1
                for (int q0 = 32 * warp; q0 < 4 * wn; q0 += kMcsWorkers) {
                    const int q = q0 + lane;
                    uint16_t c[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                    if (q < 4 * wn) panel_load8(cnt + 8 * q, c);
                    int found = 0;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const bool in = c[e] >= near;
                        const uint32_t b = __ballot_sync(kAll, in);
                        if (in) near_v[found + __popc(b & lanes_below(lane))] = (uint16_t)(8 * q + e);
                        found += __popc(b);
                    }
                    __syncwarp();
#pragma unroll 1
                    for (int k = lane; k < found; k += 32) {
                        const unsigned id = near_v[k], ce = cnt[id];
                        const uint32_t ke = key[key_slot(id)];
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            if (mcs_comp(ce + __popc(ke & m8[b]), id) <= b8[b]) continue;
#pragma unroll 1
                            for (int j = 8 * b; j < min(8 * b + 8, r); ++j)
                                if (mcs_comp(ce + __popc(ke & sh.mask[j]), id) > sh.beat[j]) r = j;
                        }
                    }
                    __syncwarp();
                }
            }
        }
        if (worker) {
            r = __reduce_min_sync(kAll, r);
            if (lane == 0 && r < w2) atomicMin(&sh.r, r);
        }
        __syncthreads();
        // ---- counts, group maxima, results.  (Step 0 visits the largest of all: r > 0.)
        r = max(sh.r, 1);
        const uint32_t taken = sh.mask[r];
        if (!worker) {
            if (lane < r) {
                const int x = sh.piv[lane];
                order[d.obase + i + lane] = x;
                if (pos) pos[d.vbase + x] = i + lane;
            }
            mycnt += __popc(adj & taken);
            if (lane < w2 && mypos >= r)
                atomicMax(&sh.group[(myv & 31) << 2 | ((myv >> 8) & 3)], mcs_comp(mycnt, myv));
        }
        if (worker) {
            unsigned best[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll 1
            for (int q = t; q < 4 * wn; q += kMcsWorkers) {
                uint16_t c[8];
                uint32_t k[8];
                load8(q, c, k);
                const unsigned v0 = 8 * q;
                uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    unsigned ce = c[e];
                    if (ce) {
                        ce += __popc(k[e] & taken);
                        best[e] = max(best[e], mcs_comp(ce, v0 + e));
                    }
                    o[e >> 1] |= ce << (16 * (e & 1));
                }
                *reinterpret_cast<uint4 *>(cnt + v0) = make_uint4(o[0], o[1], o[2], o[3]);
            }
            // a lane's vertices are 8 (lane & 3) + e modulo 32: groups of the same residue
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                unsigned b = best[e];
                b = max(b, __shfl_xor_sync(kAll, b, 4));
                b = max(b, __shfl_xor_sync(kAll, b, 8));
                b = max(b, __shfl_xor_sync(kAll, b, 16));
                if (lane < 4 && b) atomicMax(&sh.group[(8 * lane + e) << 2 | (warp & 3)], b);
            }
        }
        i += r;
        if (++panels > 1) credit = min(credit + r - kMcsWorth, kMcsCredit);
        if (i >= n) break;
        __syncthreads();
        // ---- the next window: at least `need` vertices reach the bound
        const int need = min(32, n - i);
        if (!worker && lane < w2 && mypos >= r) cnt[myv] = (uint16_t)mycnt;
        if (t < kMcsGroups) {   // the need-th largest group maximum, if there are as many
            const unsigned mine = sh.group[t];
            int above = 0;
#pragma unroll 1
            for (int k = 0; k < kMcsGroups; k += 4) {
                const uint4 g = *reinterpret_cast<const uint4 *>(&sh.group[k]);
                above += (g.x > mine) + (g.y > mine) + (g.z > mine) + (g.w > mine);
            }
            if (mine && above == need - 1) sh.bound = mine;
        }
        __syncthreads();
        unsigned bound = max(sh.bound, 1u), lo = 1u, hi = 0xFFFFFFFFu;
#pragma unroll 1
        for (int it = 0; it < 34; ++it) {
            if (worker) {
#pragma unroll 1
                for (int q = t; q < 4 * wn; q += kMcsWorkers) {
                    uint16_t c[8];
                    panel_load8(cnt + 8 * q, c);
                    uint32_t in = 0u;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        in |= (c[e] && mcs_comp(c[e], 8 * q + e) >= bound ? 1u : 0u) << e;
                    if (in) {
                        int at = atomicAdd(&sh.ncand, __popc(in));
#pragma unroll 1
                        for (; in; in &= in - 1u) {
                            const int e = __ffs(in) - 1;
                            if (at < kMcsCand) sh.cand[at] = mcs_comp(cnt[8 * q + e], 8 * q + e);
                            ++at;
                        }
                    }
                }
            }
            __syncthreads();
            const int got = sh.ncand;
            if (got >= need && got <= kMcsCand) break;
            if (got < need) hi = bound; else lo = bound;   // too few below hi, too many from lo on
            bound = lo + (hi - lo) / 2;
            __syncthreads();
            if (t == 0) sh.ncand = 0;
            __syncthreads();
        }
        const int got = min(sh.ncand, kMcsCand);
        const int lg = got <= 32 ? 4 : got <= 64 ? 3 : got <= 128 ? 2 : got <= 256 ? 1 : 0, step = 1 << lg;
        if (worker && (warp * 32) >> lg < got) {
            const int e = t >> lg;
            const unsigned mine = e < got ? sh.cand[e] : 0u;
            int rank = 0;
#pragma unroll 4
            for (int k = t & (step - 1); k < got; k += step) rank += sh.cand[k] > mine ? 1 : 0;
#pragma unroll 1
            for (int o = 1; o < step; o <<= 1) rank += __shfl_xor_sync(kAll, rank, o);
            if (e < got && (t & (step - 1)) == 0 && rank < 32) {
                const int v = 65535 - (int)(mine & 0xFFFFu);
                sh.v[rank] = v;
                sh.cnt[rank] = (int)(mine >> 16);
                reinterpret_cast<unsigned *>(sh.row4)[rank] = 4u * v;
            }
        }
        __syncthreads();
        if (credit < -kMcsPatience) {   // the rest goes step by step
            for (int q = t; q < 4 * wn; q += kMcsThreads)
                reinterpret_cast<uint4 *>(left->cnt)[q] = *reinterpret_cast<const uint4 *>(cnt + 8 * q);
            if (t == 0) {
                left->i = i;
                left->x = sh.v[0];
            }
            return;
        }
    }
    if (t == 0) left->i = n;
}

// One step per vertex, from the beginning (left null) or from where the panels
// stopped.  Counts as 16-bit values in shared memory with a numbered bitmask.
// Thread t owns a bit slice of row words and keeps in a register the largest key
// (count << 16 | 65535 - v) of the unnumbered vertices of its slice.  A step: the
// owners of the pivot's unnumbered neighbours raise their counts and keys; the
// owner of the pivot's own slice (or, for slices longer than 4 bits, that
// thread's warp) rescans it; a block-wide max of the keys (warp max, one barrier,
// then every warp reduces the warp maxima) names the next pivot.  The pivot's row
// is the one load on the step's critical path: a graph whose rows fit beside the
// counts is first copied into shared memory (n <= ~1,340); a larger one is
// bulk-prefetched into L2.
template <int T, int WPT, bool WARP_RESCAN>
__global__ void __launch_bounds__(T) mcs_step_kernel(DenseDesc d, int32_t *__restrict__ order,
                                                     int32_t *__restrict__ pos, uint32_t smem_bytes,
                                                     const McsLeft *left) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned red[2][T / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int n = d.n, i0 = left ? left->i : 0;   // vertices numbered already
    if (i0 >= n) return;
    {
        int32_t *ord = order + d.obase;
        int32_t *ps = pos ? pos + d.vbase : nullptr;
        const int wn = (n + 31) >> 5;
        const uint32_t lastmask = (n & 31) ? ((1u << (n & 31)) - 1u) : 0xFFFFFFFFu;
        const size_t label_bytes = ((size_t)n * 2 + 15) & ~size_t(15);
        const size_t state_bytes = label_bytes + (size_t)wn * 4;
        uint16_t *label = reinterpret_cast<uint16_t *>(smem);
        uint32_t *numbered = reinterpret_cast<uint32_t *>(smem + label_bytes);
        const uint32_t *rows = d.rows;
        int stride = d.words;
        // (kept from the compiler: with the parameter's own registers in the step's addresses G(8,000, 1/2) took 7.28
        // ms instead of 7.11, G(15,000, 1/2) 18.0 instead of 17.6)
        asm volatile("" : "+l"(rows), "+r"(stride));
        const size_t rows_off = (state_bytes + 15) & ~size_t(15);
        if (rows_off + (size_t)n * wn * 4 <= smem_bytes) {   // compact copy (stride wn) beside the counts
            uint32_t *rs = reinterpret_cast<uint32_t *>(smem + rows_off);
            for (int v = warp; v < n; v += T / 32)
                for (int w = lane; w < wn; w += 32) rs[(size_t)v * wn + w] = __ldg(d.rows + (size_t)v * d.words + w);
            rows = rs;
            stride = wn;
        } else {
            prefetch_range_l2<T>(d.rows, (size_t)n * d.words * sizeof(uint32_t));
        }
        int lpw = 1;
        while (lpw < 32 && T / (lpw * 2) >= wn) lpw *= 2;
        const int kGroups = T / lpw, kSlice = 32 / lpw;
        const int lpwShift = __ffs(lpw) - 1, sliceShift = __ffs(kSlice) - 1, groupShift = __ffs(kGroups) - 1;
        const int wt = t / lpw, sl = t % lpw;
        const uint32_t part = lpw == 1 ? 0xFFFFFFFFu : (((1u << kSlice) - 1u) << (sl * kSlice));
        if (left) {
            for (int v = t; v < n; v += T) label[v] = (uint16_t)max((int)left->cnt[v] - 1, 0);
            for (int w = t; w < wn; w += T) {
                uint32_t m = 0u;   // (count 0: numbered, or past the end)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    uint16_t c[8];
                    panel_load8(&left->cnt[32 * w + 8 * q], c);
#pragma unroll
                    for (int e = 0; e < 8; ++e) m |= (c[e] ? 0u : 1u) << (8 * q + e);
                }
                numbered[w] = m;
            }
            __syncthreads();
        } else {
            for (int v = t; v < n; v += T) label[v] = 0;
            for (int w = t; w < wn; w += T) numbered[w] = 0u;
        }
        // initial keys: count 0, so the lowest id of each slice
        unsigned kmax[WPT];
        uint32_t row[WPT];
#pragma unroll
        for (int k = 0; k < WPT; ++k) {
            const int w = k * kGroups + wt;
            uint32_t valid = w < wn ? (w == wn - 1 ? lastmask : 0xFFFFFFFFu) & part : 0u;
            kmax[k] = valid ? (65535u - (unsigned)((w << 5) + __ffs(valid) - 1)) : 0u;
            if (left && w < wn) {
                kmax[k] = 0u;
                for (valid &= ~numbered[w]; valid; valid &= valid - 1u) {
                    const unsigned y = (w << 5) + __ffs(valid) - 1;
                    kmax[k] = max(kmax[k], ((unsigned)label[y] << 16) | (65535u - y));
                }
            }
        }
        int x = left ? left->x : 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < WPT; ++k) {   // row of the first pivot
            const int w = k * kGroups + wt;
            row[k] = w < wn ? rows[(size_t)x * stride + w] & part : 0u;
        }
        for (int i = i0; i < n; ++i) {
            const int slot = i & 1;
            if (t == 0) {
                ord[i] = x;
                if (ps) ps[x] = i;
            }
            unsigned best = 0u;
            if constexpr (!WARP_RESCAN) {
                // short slices: the owner of x's slice recomputes its maximum without x
#pragma unroll
                for (int k = 0; k < WPT; ++k) {
                    const int w = k * kGroups + wt;
                    if (w < wn) {
                        uint32_t nb = numbered[w];
                        const bool mine = w == (x >> 5) && ((part >> (x & 31)) & 1u);
                        if (mine) {
                            nb |= 1u << (x & 31);
                            numbered[w] = nb;
                        }
                        uint32_t bits = row[k] & ~nb;   // unnumbered neighbours of x in this slice
                        if (w == wn - 1) bits &= lastmask;
                        while (bits) {
                            const int y = (w << 5) + __ffs(bits) - 1;
                            bits &= bits - 1;
                            const unsigned c = (unsigned)label[y] + 1u;
                            label[y] = (uint16_t)c;
                            const unsigned key = (c << 16) | (65535u - (unsigned)y);
                            kmax[k] = key > kmax[k] ? key : kmax[k];
                        }
                        if (mine) {
                            uint32_t live = ~nb & part;
                            if (w == wn - 1) live &= lastmask;
                            unsigned m = 0u;
                            while (live) {
                                const int y = (w << 5) + __ffs(live) - 1;
                                live &= live - 1;
                                const unsigned key = ((unsigned)label[y] << 16) | (65535u - (unsigned)y);
                                m = key > m ? key : m;
                            }
                            kmax[k] = m;
                        }
                    }
                    best = kmax[k] > best ? kmax[k] : best;
                }
            } else {
                // long slices: the warp of x's owner recomputes that slice's
                // maximum without x, one lane per vertex.  x's slice: word xw,
                // slice xs, held by thread xt as its item xk (lpw, kSlice and
                // kGroups are powers of two).
                const int xw = x >> 5, xs = (x & 31) >> sliceShift;
                const int xk = xw >> groupShift, xt = ((xw & (kGroups - 1)) << lpwShift) + xs;
#pragma unroll
                for (int k = 0; k < WPT; ++k) {
                    const int w = k * kGroups + wt;
                    if (w < wn) {
                        uint32_t nb = numbered[w];
                        if (t == xt && k == xk) {
                            nb |= 1u << (x & 31);
                            numbered[w] = nb;
                        }
                        uint32_t bits = row[k] & ~nb;
                        if (w == wn - 1) bits &= lastmask;
                        unsigned km = kmax[k];
                        while (bits) {
                            const int y = (w << 5) + __ffs(bits) - 1;
                            bits &= bits - 1;
                            const unsigned c = (unsigned)label[y] + 1u;
                            label[y] = (uint16_t)c;
                            km = max(km, (c << 16) | (65535u - (unsigned)y));
                        }
                        kmax[k] = km;
                    }
                }
                if ((xt >> 5) == warp) {
                    __syncwarp();
                    const int y = (xw << 5) + xs * kSlice + lane;
                    unsigned key = 0u;
                    if (lane < kSlice && y < n && !((numbered[xw] >> (y & 31)) & 1u))
                        key = ((unsigned)label[y] << 16) | (65535u - (unsigned)y);
                    key = __reduce_max_sync(0xFFFFFFFFu, key);
#pragma unroll
                    for (int k = 0; k < WPT; ++k)
                        if (t == xt && k == xk) kmax[k] = key;
                }
#pragma unroll
                for (int k = 0; k < WPT; ++k) best = kmax[k] > best ? kmax[k] : best;
            }
            best = __reduce_max_sync(0xFFFFFFFFu, best);
            if (lane == 0) red[slot][warp] = best;
            __syncthreads();
            const unsigned r = lane < T / 32 ? red[slot][lane] : 0u;
            const unsigned top = __reduce_max_sync(0xFFFFFFFFu, r);
            if (i + 1 == n) break;
            x = (int)(65535u - (top & 0xFFFFu));
            if (x >= n) x = n - 1;   // unreachable while an unnumbered vertex remains; keeps loads in bounds
#pragma unroll
            for (int k = 0; k < WPT; ++k) {
                const int w = k * kGroups + wt;
                row[k] = w < wn ? rows[(size_t)x * stride + w] & part : 0u;
            }
        }
    }
}

// Lanes per row word as the kernel chooses them for n (the smallest power of
// two whose word groups still cover the row).
int mcs_lpw(int T, int n) {
    const int wn = (n + 31) / 32;
    int lpw = 1;
    while (lpw < 32 && T / (lpw * 2) >= wn) lpw *= 2;
    return lpw;
}

template <int T, int WPT>
int launch_steps(size_t smem, DenseDesc d, int32_t *order, int32_t *pos, const McsLeft *left, cudaStream_t stream) {
    // slices of more than 4 bits are rescanned by a warp, shorter ones by their owner
    auto kern = 32 / mcs_lpw(T, d.n) > 4 ? mcs_step_kernel<T, WPT, true> : mcs_step_kernel<T, WPT, false>;
    CG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<1, T, smem, stream>>>(d, order, pos, (uint32_t)smem, left);
    CG_LAUNCH_CHECK("mcs_step_kernel");
    return CG_OK;
}

}  // namespace

size_t mcs_workspace_bytes(int n) {
    return n >= kMcsPanelMin && n <= kMcsPanelMax ? sizeof(McsLeft) + (size_t)((n + 31) / 32) * 64 : 0;
}

int mcs_dense_launch(DenseDesc d, int32_t *order, int32_t *pos, void *ws, cudaStream_t stream) {
    const int n = d.n;
    if (n <= 0) return CG_OK;
    if (n > kMcsMaxN) return set_error(CG_EINVAL, "dense MCS supports n <= %d (got %d)", kMcsMaxN, n);
    const size_t wn = (size_t)(n + 31) / 32;
    McsLeft *left = nullptr;
    if (mcs_workspace_bytes(n)) {
        left = static_cast<McsLeft *>(ws);
        const size_t smem = wn * 192;
        CG_CUDA_TRY(cudaFuncSetAttribute(mcs_panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        mcs_panel_kernel<<<1, kMcsThreads, smem, stream>>>(d, order, pos, left);
        CG_LAUNCH_CHECK("mcs_panel_kernel");
    }
    // counts + numbered bits; with the rows too when they fit (n <= ~1,340)
    const size_t state = ((((size_t)n * 2 + 15) & ~size_t(15)) + wn * 4 + 15) & ~size_t(15);
    const size_t with_rows = state + (size_t)n * wn * 4;
    const size_t smem = with_rows <= kMcsSmemRows ? with_rows : state;
    if (n <= 2048) return launch_steps<512, 1>(smem, d, order, pos, left, stream);
    if (n <= 32768) return launch_steps<1024, 1>(smem, d, order, pos, left, stream);
    return launch_steps<1024, 2>(smem, d, order, pos, left, stream);
}

}  // namespace cg
