// lexbfs_dense.cu — kernels and launcher of the one-CTA-per-graph dense LexBFS.
#include <algorithm>

#include "kernels.h"
#include "lexbfs_dense.cuh"

namespace cg {

#ifdef CG_BOUNDS_CHECK
// A code set by cg_debug_inject: the next dense LexBFS launch records it as a
// bounds-check error without touching memory out of range (a test of the
// status path).
static __device__ unsigned cg_dbg_inject_code;
#endif

namespace {

constexpr size_t kSmemLimit = 227 * 1024;    // opt-in dynamic shared memory per CTA (sm_100 family)
constexpr int kDenseMaxN = 131072;

template <int STATE, int T>
__global__ void __launch_bounds__(T) lexbfs_dense_kernel(const DenseDesc *__restrict__ descs, DenseDesc single,
                                                         int count, int32_t *__restrict__ order,
                                                         int32_t *__restrict__ pos, int32_t *ppos,
                                                         unsigned char *gstate, size_t gstate_stride,
                                                         int *work_counter, uint32_t *emask, int cap,
                                                         unsigned long long *keys) {
    extern __shared__ __align__(16) unsigned char smem[];
    PanelScalars *sc = reinterpret_cast<PanelScalars *>(smem);
#ifdef CG_BOUNDS_CHECK
    if (blockIdx.x == 0 && threadIdx.x == 0 && cg_dbg_inject_code) {
        cg_dbg_record(cg_dbg_inject_code, 0ull);
        cg_dbg_inject_code = 0u;
    }
#endif
    if (keys && blockIdx.x == 0)   // the check's initial keys: "no violation", then its CTA counter and error word
        for (int k = threadIdx.x; k < count + 2; k += T) keys[k] = k < count ? ~0ull : 0ull;
    for (;;) {
        if (threadIdx.x == 0) sc->next_graph = count == 1 ? (int)blockIdx.x : atomicAdd(work_counter, 1);
        __syncthreads();
        const int gi = sc->next_graph;
        __syncthreads();
        if (gi >= count) break;
        const DenseDesc d = descs ? descs[gi] : single;
        const int n = d.n;
        prefetch_range_l2<T>(d.rows, (size_t)n * d.words * sizeof(uint32_t));
        lexbfs_panels<STATE, T>(d.rows, d.words, n, cap,
                                STATE == kStateSmem ? nullptr : gstate + (size_t)blockIdx.x * gstate_stride,
                                order + d.obase, pos ? pos + d.vbase : nullptr, ppos ? ppos + d.vbase : nullptr,
                                emask ? emask + d.ebase : nullptr);
        __syncthreads();
        if (count == 1) break;
    }
}

template <int STATE, int T>
int launch_variant(const LexPlan &plan, const DenseDesc *descs, DenseDesc single, int count, int ctas,
                   int32_t *order, int32_t *pos, int32_t *ppos, void *gstate, int *work_counter,
                   cudaStream_t stream, unsigned long long *keys, uint32_t *emask) {
    auto kern = lexbfs_dense_kernel<STATE, T>;
    CG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)plan.smem_bytes));
    if (count > 1) CG_CUDA_TRY(cudaMemsetAsync(work_counter, 0, sizeof(int), stream));
    kern<<<ctas, T, plan.smem_bytes, stream>>>(descs, single, count, order, pos, ppos,
                                               static_cast<unsigned char *>(gstate), plan.gstate_bytes, work_counter,
                                               emask, plan.sort_cap, keys);
    CG_LAUNCH_CHECK("lexbfs_dense_kernel");
    CG_DEBUG_CHECK(stream, "lexbfs_dense_kernel");
    return CG_OK;
}

}  // namespace

int lexbfs_dense_plan(int n_max, int threads_override, LexPlan *plan) {
    if (n_max < 0 || n_max > kDenseMaxN)
        return set_error(CG_EINVAL, "dense LexBFS supports n <= %d (got %d); use the CSR entry points", kDenseMaxN,
                         n_max);
    LexPlan p{};
    const int n = std::max(n_max, 1);
    auto room = [&](int state) {   // shared memory left for the sort's arrays
        const size_t used = kPanelScalarBytes + panel_state_bytes(n, state);
        return used < kSmemLimit ? kSmemLimit - used : 0;
    };
    // the keys are gathered at random, so they leave shared memory last
    if (room(kStateSmem) >= panel_sort_bytes(kSortCapMax)) p.state = kStateSmem;
    else if (room(kStatePermGlobal) >= panel_sort_bytes(1024) && n <= 65535) p.state = kStatePermGlobal;
    else p.state = kStateGlobal;
    p.sort_cap = panel_sort_cap(n, room(p.state));
    p.smem_bytes = kPanelScalarBytes + panel_state_bytes(n, p.state) + panel_sort_bytes(p.sort_cap);
    p.gstate_bytes = panel_global_bytes(n, p.state);
    // measured on GB300 (us) with 128 / 256 / 512 threads: n = 1,000 226 / 187 / 210, 2,048 512 / 393 / 390,
    // 4,096 1,147 / 813 / 686; the pair of n = 16,384 with 512 4,350, with 1,024 4,570
    int th = n <= 2048 ? 256 : 512;
    if (threads_override) th = threads_override;
    if (p.state != kStateSmem) th = 1024;
    if (th != 128 && th != 256 && th != 512 && th != 1024)
        return set_error(CG_EINVAL, "unsupported CTA size %d", th);
    p.threads = th;
    p.n_max = n;
    *plan = p;
    return CG_OK;
}

int lexbfs_dense_launch(const LexPlan &plan, const DenseDesc *descs, DenseDesc single, int count, int ctas,
                        int32_t *order, int32_t *pos, int32_t *ppos, void *gstate, int *work_counter,
                        cudaStream_t stream, unsigned long long *keys, uint32_t *emask) {
    if (count <= 0) return CG_OK;
    if (emask && (reinterpret_cast<uintptr_t>(emask) & 15) != 0)
        return set_error(CG_EINVAL, "earlier-than mask buffer not 16-byte aligned");
    ctas = std::max(1, std::min(ctas, count));
    auto go = [&](auto launch) {
        return launch(plan, descs, single, count, ctas, order, pos, ppos, gstate, work_counter, stream, keys, emask);
    };
    if (plan.state == kStateGlobal) return go(launch_variant<kStateGlobal, 1024>);
    if (plan.state == kStatePermGlobal) return go(launch_variant<kStatePermGlobal, 1024>);
    switch (plan.threads) {
        case 128: return go(launch_variant<kStateSmem, 128>);
        case 256: return go(launch_variant<kStateSmem, 256>);
        case 512: return go(launch_variant<kStateSmem, 512>);
        default: return go(launch_variant<kStateSmem, 1024>);
    }
}

int debug_inject(unsigned code) {
#ifdef CG_BOUNDS_CHECK
    CG_CUDA_TRY(cudaMemcpyToSymbol(cg_dbg_inject_code, &code, sizeof(code)));
    return CG_OK;
#else
    (void)code;
    return set_error(CG_EINVAL, "not a bounds-checking build (CG_BOUNDS_CHECK)");
#endif
}

}  // namespace cg
