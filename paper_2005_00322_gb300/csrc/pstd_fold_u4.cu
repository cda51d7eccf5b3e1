// pstd_fold_u4.cu -- fixed schedules of the folded passes, group 4 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(4)
}  // namespace pstd
