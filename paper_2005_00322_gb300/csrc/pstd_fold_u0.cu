// pstd_fold_u0.cu -- fixed schedules of the folded passes, group 0 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(0)
}  // namespace pstd
