// pstd_fold_any_step.cu -- leapfrog pass of the run-time schedules.
#include "pstd_fkernels.cuh"

namespace pstd {
const void* fold_any_step(bool strided) {
    return strided ? (const void*)fold::k_fold_any<true, FOLD_STEP> : (const void*)fold::k_fold_any<false, FOLD_STEP>;
}
}  // namespace pstd
