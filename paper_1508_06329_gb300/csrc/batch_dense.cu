// batch_dense.cu — the whole chordality test of one small dense graph in one
// CTA, many graphs per launch (the batched path).
//
// Each CTA takes graphs from an atomic counter (graphs pre-sorted largest
// first by the host), runs the panel LexBFS of lexbfs_dense.cuh, then the
// perfect-elimination check of Sections 5.2 / 6.2 on the same graph, and
// writes (chordal, v, p, u).  The search reads each row about once, so the rows
// stay in global memory (L2) and an SM holds as many CTAs as the state allows.
#include <algorithm>

#include "kernels.h"
#include "lexbfs_dense.cuh"

namespace cg {

namespace {

// The perfect-elimination check of the order that lexbfs_panels left in perm,
// by groups of 32 positions: E (the numbered mask, rebuilt) holds the vertices
// before the group; a warp per position reads row v & ~row p(v) & E, then the
// group's own earlier positions one per lane.  Groups run in order, so the
// first group with a violation ends the check.  Two positions and two words per
// lane at a time, so that eight loads are in flight: one by one, 4,096 graphs of
// 16..2,048 vertices took 1.53 ms instead of 1.25 (search included).
template <int T, typename St>
__device__ void check_cta(const uint32_t *__restrict__ rows, int stride, int n, const St &st,
                          const int32_t *__restrict__ ppos, unsigned long long *skey) {
    constexpr int NW = T / 32;
    constexpr unsigned kAll = 0xFFFFFFFFu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int wn = (n + 31) >> 5;
    for (int w = threadIdx.x; w < wn; w += T) st.numbered[w] = 0u;
    __syncthreads();
    for (int g0 = 0; g0 < n; g0 += 32) {
        const bool on = g0 + lane < n;
        const int vg = on ? (int)st.perm[g0 + lane] : -1;
        const int pg = on ? __ldcg(ppos + g0 + lane) : -1;
#pragma unroll 1
        for (int j0 = warp; j0 < 32; j0 += 2 * NW) {
            int p[2];
            const uint32_t *rv[2], *rp[2];
            unsigned m[2] = {kNoVertex, kNoVertex};
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int v = __shfl_sync(kAll, vg, j0 + k * NW);
                p[k] = __shfl_sync(kAll, pg, j0 + k * NW);   // -1: no earlier neighbour (or past the end)
                rv[k] = rows + (size_t)max(v, 0) * stride;
                rp[k] = rows + (size_t)max(p[k], 0) * stride;
            }
#pragma unroll 1
            for (int w0 = 0; w0 < wn; w0 += 64) {
                uint32_t bits[2][2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int w = w0 + 32 * u + lane;
#pragma unroll
                    for (int k = 0; k < 2; ++k) bits[k][u] = w < wn && p[k] >= 0 ? rv[k][w] & ~rp[k][w] : 0u;
                }
#pragma unroll
                for (int u = 1; u >= 0; --u) {
                    const int w = w0 + 32 * u + lane;
                    const uint32_t e = w < wn ? st.numbered[w] : 0u;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        bits[k][u] &= e;
                        if (w == (p[k] >> 5)) bits[k][u] &= ~(1u << (p[k] & 31));
                        if (bits[k][u]) m[k] = min(m[k], (unsigned)((w << 5) + __ffs(bits[k][u]) - 1));
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int j = j0 + k * NW;
                if (p[k] < 0) continue;
                if (lane < j && vg != p[k]) {
                    const uint32_t bit = 1u << (vg & 31);
                    if ((rv[k][vg >> 5] & bit) && !(rp[k][vg >> 5] & bit)) m[k] = min(m[k], (unsigned)vg);
                }
                m[k] = __reduce_min_sync(kAll, m[k]);
                if (lane == 0 && m[k] != kNoVertex)
                    atomicMin(skey, ((unsigned long long)(unsigned)(g0 + j) << 32) | m[k]);
            }
        }
        __syncthreads();
        if (*skey != ~0ull) break;
        if (warp == 0 && on) atomicOr(&st.numbered[vg >> 5], 1u << (vg & 31));
        __syncthreads();
    }
}

// CTAs per SM that the registers allow at least (the shared memory of small graphs has room for more): without it
// CTAs of 64 threads take 96 registers instead of 64, those of 256 118 instead of 80.
constexpr int fused_min_ctas(int threads) { return threads <= 64 ? 16 : threads <= 128 ? 7 : threads <= 256 ? 3 : 1; }

template <int T>
__global__ void __launch_bounds__(T, fused_min_ctas(T))
chordal_dense_fused_kernel(const DenseDesc *__restrict__ descs, int count, int32_t *__restrict__ order, int32_t *ppos,
                           cg_result *__restrict__ res, int *work_counter, int cap) {
    extern __shared__ __align__(16) unsigned char smem[];
    PanelScalars *sc = reinterpret_cast<PanelScalars *>(smem);
    __shared__ unsigned long long skey;
    for (;;) {
        if (threadIdx.x == 0) {
            sc->next_graph = atomicAdd(work_counter, 1);
            skey = ~0ull;
        }
        __syncthreads();
        const int gi = sc->next_graph;
        __syncthreads();
        if (gi >= count) break;
        const DenseDesc d = descs[gi];
        const int n = d.n;
        prefetch_range_l2<T>(d.rows, (size_t)n * d.words * sizeof(uint32_t));
        const auto st = panel_carve<kStateSmem>(smem + kPanelScalarBytes, nullptr, n, cap);
        int32_t *ord = order + d.obase;
        int32_t *pp = ppos + d.vbase;
        lexbfs_panels<kStateSmem, T>(d.rows, d.words, n, cap, nullptr, ord, nullptr, pp, nullptr);
        __syncthreads();
        check_cta<T>(d.rows, d.words, n, st, pp, &skey);
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned long long k = skey;
            cg_result r;
            if (k == ~0ull) {
                r.chordal = 1;
                r.v = r.p = r.u = -1;
            } else {
                const int i = (int)(k >> 32);
                r.chordal = 0;
                r.v = (int)st.perm[i];
                r.p = __ldcg(pp + i);
                r.u = (int)(k & 0xFFFFFFFFu);
            }
            res[d.rindex] = r;
        }
        __syncthreads();
    }
}

template <int T>
int launch_fused(const FusedPlan &plan, const DenseDesc *descs, int count, int ctas, int32_t *order, int32_t *ppos,
                 cg_result *res, int *work_counter, cudaStream_t stream) {
    auto kern = chordal_dense_fused_kernel<T>;
    CG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes));
    CG_CUDA_TRY(cudaMemsetAsync(work_counter, 0, sizeof(int), stream));
    kern<<<ctas, T, plan.smem_bytes, stream>>>(descs, count, order, ppos, res, work_counter, plan.sort_cap);
    CG_LAUNCH_CHECK("chordal_dense_fused_kernel");
    CG_DEBUG_CHECK(stream, "chordal_dense_fused_kernel");
    return CG_OK;
}

}  // namespace

int fused_dense_plan(int n_max, int threads, FusedPlan *plan) {
    if (n_max < 0 || n_max > kFusedMaxN)
        return set_error(CG_EINVAL, "fused batch path supports n <= %d (got %d)", kFusedMaxN, n_max);
    const int n = std::max(n_max, 1);
    FusedPlan p{};
    // for batches that fill the GPU: with 64 / 128 / 256 / 512 threads 1,200 graphs of 250 vertices take 140 / 170 /
    // 217 / 546 us, of 1,000 723 / 791 / 841 / 1,971, of 2,000 2,883 / 2,011 / 2,043 / 4,045.  (Two graphs of 250 take
    // 106 / 83 / 70 / 87, of 1,000 471 / 307 / 236 / 244: cg_batch_autotune finds that.)
    if (threads == 0) threads = n <= 256 ? 64 : n <= 2048 ? 128 : 256;
    if (threads != 64 && threads != 128 && threads != 256 && threads != 512)
        return set_error(CG_EINVAL, "fused batch path: unsupported CTA size %d", threads);
    p.threads = threads;
    p.sort_cap = panel_sort_cap(n, panel_sort_bytes(kSortCapMax));
    p.smem_bytes = kPanelScalarBytes + panel_state_bytes(n, kStateSmem) + panel_sort_bytes(p.sort_cap);
    *plan = p;
    return CG_OK;
}

int fused_dense_launch(const FusedPlan &plan, const DenseDesc *descs, int count, int ctas, int32_t *order,
                       int32_t *ppos, cg_result *res, int *work_counter, cudaStream_t stream) {
    if (count <= 0) return CG_OK;
    ctas = std::max(1, std::min(ctas, count));
    auto go = [&](auto launch) { return launch(plan, descs, count, ctas, order, ppos, res, work_counter, stream); };
    switch (plan.threads) {
        case 64: return go(launch_fused<64>);
        case 128: return go(launch_fused<128>);
        case 256: return go(launch_fused<256>);
        case 512: return go(launch_fused<512>);
        default:
            return set_error(CG_EINVAL, "fused batch path: unsupported CTA size %d", plan.threads);
    }
}

int fused_ctas_per_sm(const FusedPlan &plan) {
    const int by_smem = (int)std::max<size_t>(1, (228 * 1024) / (plan.smem_bytes + 1024 + 16));
    const int by_threads = std::max(1, 2048 / plan.threads);
    return std::max(1, std::min(std::min(by_smem, by_threads), 32));
}

}  // namespace cg
