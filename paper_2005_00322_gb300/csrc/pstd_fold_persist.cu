// pstd_fold_persist.cu -- a whole run of folded passes as one cooperative
// kernel (grid and barrier as in pstd_persist.cuh), for one plan or a batch.
#include "pstd_fkernels.cuh"

namespace pstd {
namespace {
__global__ void __launch_bounds__(fold::kAnyThreads, 2) k_fold_persist(const __grid_constant__ FoldPersistArgs a) {
#ifdef __CUDA_ARCH__
    extern __shared__ float4 wsm4[];
    for (int64_t s = 0; s < a.nsteps; ++s) {
        for (int k = 0; k < a.ndim; ++k) {
            const int ax = a.ndim - 1 - k;
            const int64_t* pre = a.members ? a.prefix + (size_t)k * (a.members + 1) : nullptr;
            const int64_t items = a.members ? pre[a.members] : (int64_t)a.items[ax];
            for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
                const int m = a.members ? member_of(pre, a.members, it) : 0;
                const FoldArgs& w = a.members ? a.mem[(size_t)m * 3 + k] : a.ax[ax];
                const unsigned item = (unsigned)(a.members ? it - pre[m] : it);
                if (w.ax.inner > 1) fold::fold_pass<fold::AnyCfg, true, FOLD_STEP>(w, item, wsm4, threadIdx.x, blockDim.x);
                else fold::fold_pass<fold::AnyCfg, false, FOLD_STEP>(w, item, wsm4, threadIdx.x, blockDim.x);
                __syncthreads();     // shared memory is reused by the next item
            }
            if (!grid_sync(a.sync)) return;
        }
    }
#endif
}
}  // namespace
const void* fold_any_persist() { return (const void*)k_fold_persist; }
}  // namespace pstd
