// pstd_fold_u7.cu -- fixed schedules of the folded passes, group 7 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(7)
}  // namespace pstd
