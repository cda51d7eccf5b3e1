// pstd_fold_u6.cu -- fixed schedules of the folded passes, group 6 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(6)
}  // namespace pstd
