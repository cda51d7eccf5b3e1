// pstd_fold_any_misc_s.cu -- derivatives, velocity conversions and the
// second-order pass of the folded passes, strided lines.
#include "pstd_fkernels.cuh"

namespace pstd {
const void* fold_any_misc_s() { return (const void*)fold::k_fold_any<true, -1>; }
}  // namespace pstd
