// pstd_fold_any_misc_c.cu -- derivatives, velocity conversions and the
// second-order pass of the folded passes, contiguous lines.
#include "pstd_fkernels.cuh"

namespace pstd {
const void* fold_any_misc_c() { return (const void*)fold::k_fold_any<false, -1>; }
}  // namespace pstd
