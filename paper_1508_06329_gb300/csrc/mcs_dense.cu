// mcs_dense.cu — Maximum Cardinality Search on dense graphs in panels of up to
// 32 pivots, one CTA.
//
// Method (Section 5.1; Tarjan and Yannakakis): every unnumbered vertex carries
// the number of its numbered neighbours; each step numbers a vertex with the
// largest count (lowest id among equals, as for LexBFS) and counts it at its
// unnumbered neighbours.  By Theorem 5.2 the graph is chordal iff the MCS
// order is a perfect elimination order, so the same check follows.
//
// One step at a time is a latency chain of a row load, a CTA-wide maximum and a
// barrier per vertex.  A panel takes the 32 vertices with the largest
// (count, id) as a window and runs MCS on them alone:
//   1. sixteen warps read the window's rows and transpose them in registers:
//      vertex y's key, bit j = adjacent to window vertex j; meanwhile the last
//      warp, one lane per window vertex, visits the window;
//   2. a vertex outside the window comes into it before step j when its count
//      plus its neighbours among the first j pivots beats pivot j: the first
//      such step (a few comparisons of bounds over eight steps each, all steps
//      for the vertices that pass) ends the panel;
//   3. the counts of all vertices grow by their neighbours among the r pivots,
//      and the next window is found: the 32nd largest of the maxima over 128
//      groups of vertices (strided, so that neighbouring ids fall into different
//      ones) is a bound that at least 32 vertices reach, usually about 130,
//      which are ranked by counting; when more than kMcsCand reach it, the
//      bound is bisected.
// A panel numbers about 31 vertices on dense chordal graphs and 10 on
// G(n, 1/2).
//
// The counts (16 bits, plus one; 0: numbered, or in the window) and the keys of
// kMcsKeyWords words of vertices are in shared memory; a larger graph passes
// over its rows twice per panel, in chunks.
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
constexpr size_t kMcsSmem = 220 * 1024;

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
};

// (count, id) as one number: larger counts first, lower ids among equals.
__device__ __forceinline__ unsigned mcs_comp(unsigned c, unsigned v) { return c << 16 | (65535u - v); }

__global__ void __launch_bounds__(kMcsThreads, 1) mcs_dense_kernel(DenseDesc d, int key_words,
                                                                int32_t *__restrict__ order,
                                                                int32_t *__restrict__ pos) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ McsShared sh;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const bool worker = t < kMcsWorkers;
    const int n = d.n, wn = (n + 31) >> 5;
    const uint32_t *__restrict__ rows = d.rows;
    uint32_t *key = reinterpret_cast<uint32_t *>(smem);                     // [32 * key_words]
    uint16_t *cnt = reinterpret_cast<uint16_t *>(smem + (size_t)key_words * 128);   // [32 * wn]
    prefetch_range_l2<kMcsThreads>(rows, (size_t)n * d.words * sizeof(uint32_t));
    for (int v = t; v < 32 * wn; v += kMcsThreads) cnt[v] = v < n ? 1 : 0;
    if (t < 32) {
        sh.v[t] = t;
        sh.cnt[t] = 1;
        reinterpret_cast<unsigned *>(sh.row4)[t] = 4u * min(t, n - 1);
    }
    __syncthreads();

    const int chunks = (wn + key_words - 1) / key_words;
    for (int i = 0; i < n;) {
        const int w2 = min(32, n - i);
        int mycnt = 0, myv = 0, mypos = -1;   // last warp: its lane's window vertex
        uint32_t adj = 0u;
        // keys of words [w0, w0 + key_words)
        auto keys = [&](int w0) {
            const int we = min(key_words, wn - w0);
            for (int wb = warp * 32; wb < we; wb += kMcsWorkers) {
                const int w = wb + lane;
                uint32_t r[32];
                panel_load_rows(rows + min(w0 + w, wn - 1), d.words, sh.row4, r);   // (key bits from w2 on: not read)
                transpose32(r);
                if (w < we) {
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        *reinterpret_cast<uint4 *>(&key[32 * w + ((c ^ (w & 7)) << 2)]) =
                            make_uint4(r[4 * c], r[4 * c + 1], r[4 * c + 2], r[4 * c + 3]);
                }
            }
        };
        // eight neighbouring vertices of a chunk: their counts and keys
        auto load8 = [&](int w0, int q, uint16_t (&c)[8], uint32_t (&k)[8]) {
            panel_load8(cnt + 32 * w0 + 8 * q, c);
            const int w = q >> 2, p = (q & 3) << 1;
            const uint4 a = *reinterpret_cast<const uint4 *>(&key[32 * w + ((p ^ (w & 7)) << 2)]);
            const uint4 b = *reinterpret_cast<const uint4 *>(&key[32 * w + (((p + 1) ^ (w & 7)) << 2)]);
            k[0] = a.x, k[1] = a.y, k[2] = a.z, k[3] = a.w, k[4] = b.x, k[5] = b.y, k[6] = b.z, k[7] = b.w;
        };

        // ---- keys, and the window visited by the last warp
        if (worker) {
            keys(0);
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
            uint32_t done = 0u, m8 = 0u;
            unsigned b8 = kAll;
            for (int j = 0; j < w2; ++j) {
                const unsigned best = __reduce_max_sync(kAll, comp);
                const int x = __ffs(__ballot_sync(kAll, comp == best)) - 1;
                if (lane == x) {
                    mypos = j;
                    comp = 0u;
                } else if (comp) {
                    comp += ((adj >> x) & 1u) << 16;
                }
                b8 = min(b8, best);
                if (lane == 0) {
                    sh.mask[j] = done;
                    sh.beat[j] = best;
                }
                done |= 1u << x;
                if ((j & 7) == 7 || j + 1 == w2) {
                    m8 = done;
                    if (lane == 0) {
                        sh.mask8[j >> 3] = m8;
                        sh.beat8[j >> 3] = b8;
                    }
                    b8 = kAll;
                }
            }
            if (lane == 0) {
                sh.mask[w2] = done;
                sh.r = w2;
                for (int k = (w2 + 7) >> 3; k < 4; ++k) {
                    sh.mask8[k] = 0u;
                    sh.beat8[k] = kAll;
                }
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
        for (int ch = 0; ch < chunks; ++ch) {
            const int w0 = ch * key_words;
            if (ch > 0) {
                __syncthreads();
                if (worker) keys(w0);
                __syncthreads();
            }
            if (worker) {
                const int qe = 4 * min(key_words, wn - w0);
                for (int q = t; q < qe; q += kMcsWorkers) {
                    uint16_t c[8];
                    panel_load8(cnt + 32 * w0 + 8 * q, c);
                    const unsigned v0 = 32 * w0 + 8 * q;
                    uint32_t in = 0u;   // within 32 of the least beat
#pragma unroll
                    for (int e = 0; e < 8; ++e) in |= (c[e] >= near ? 1u : 0u) << e;
#pragma unroll 1
                    for (; in; in &= in - 1u) {
                        const int e = __ffs(in) - 1;
                        const unsigned ce = cnt[v0 + e];
                        const int w = q >> 2, p = ((q & 3) << 1) + (e >> 2);
                        const uint32_t ke = key[32 * w + ((p ^ (w & 7)) << 2) + (e & 3)];
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            if (mcs_comp(ce + __popc(ke & m8[b]), v0 + e) <= b8[b]) continue;
                            for (int j = 8 * b; j < min(8 * b + 8, r); ++j)
                                if (mcs_comp(ce + __popc(ke & sh.mask[j]), v0 + e) > sh.beat[j]) r = j;
                        }
                    }
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
        for (int ch = 0; ch < chunks; ++ch) {
            const int w0 = ch * key_words;
            if (chunks > 1) {
                __syncthreads();
                if (worker) keys(w0);
                __syncthreads();
            }
            if (!worker) continue;
            const int qe = 4 * min(key_words, wn - w0);
            unsigned best[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
            for (int q = t; q < qe; q += kMcsWorkers) {
                uint16_t c[8];
                uint32_t k[8];
                load8(w0, q, c, k);
                const unsigned v0 = 32 * w0 + 8 * q;
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
        if (i >= n) break;
        __syncthreads();
        // ---- the next window: at least `need` vertices reach the bound
        const int need = min(32, n - i);
        if (!worker && lane < w2 && mypos >= r) cnt[myv] = (uint16_t)mycnt;
        if (t < kMcsGroups) {   // the need-th largest group maximum, if there are as many
            const unsigned mine = sh.group[t];
            int above = 0;
            for (int k = 0; k < kMcsGroups; k += 4) {
                const uint4 g = *reinterpret_cast<const uint4 *>(&sh.group[k]);
                above += (g.x > mine) + (g.y > mine) + (g.z > mine) + (g.w > mine);
            }
            if (mine && above == need - 1) sh.bound = mine;
        }
        __syncthreads();
        unsigned bound = max(sh.bound, 1u), lo = 1u, hi = 0xFFFFFFFFu;
        for (int it = 0; it < 34; ++it) {
            if (worker) {
                for (int q = t; q < 4 * wn; q += kMcsWorkers) {
                    uint16_t c[8];
                    panel_load8(cnt + 8 * q, c);
                    uint32_t in = 0u;
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        in |= (c[e] && mcs_comp(c[e], 8 * q + e) >= bound ? 1u : 0u) << e;
                    if (in) {
                        int at = atomicAdd(&sh.ncand, __popc(in));
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
            for (int o = 1; o < step; o <<= 1) rank += __shfl_xor_sync(kAll, rank, o);
            if (e < got && (t & (step - 1)) == 0 && rank < 32) {
                const int v = 65535 - (int)(mine & 0xFFFFu);
                sh.v[rank] = v;
                sh.cnt[rank] = (int)(mine >> 16);
                reinterpret_cast<unsigned *>(sh.row4)[rank] = 4u * v;
            }
        }
        __syncthreads();
    }
}

}  // namespace

int mcs_dense_launch(DenseDesc d, int32_t *order, int32_t *pos, cudaStream_t stream) {
    if (d.n <= 0) return CG_OK;
    if (d.n > kMcsMaxN) return set_error(CG_EINVAL, "dense MCS supports n <= %d (got %d)", kMcsMaxN, d.n);
    const int wn = (d.n + 31) / 32;
    const size_t counts = (size_t)wn * 64;
    const int key_words = (int)std::min<size_t>((size_t)wn, (kMcsSmem - counts) / 128);
    const size_t smem = (size_t)key_words * 128 + counts;
    CG_CUDA_TRY(cudaFuncSetAttribute(mcs_dense_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    mcs_dense_kernel<<<1, kMcsThreads, smem, stream>>>(d, key_words, order, pos);
    CG_LAUNCH_CHECK("mcs_dense_kernel");
    return CG_OK;
}

}  // namespace cg
