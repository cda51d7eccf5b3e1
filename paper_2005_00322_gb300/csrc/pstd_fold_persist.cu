// pstd_fold_persist.cu -- cooperative run of the run-time schedules.
#include "pstd_fkernels.cuh"

namespace pstd {
const void* fold_any_persist() { return (const void*)fold::k_fold_persist<fold::AnyCfg, fold::AnyCfg>; }
}  // namespace pstd
