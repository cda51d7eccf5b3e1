// pstd_fold_u9.cu -- fixed schedules of the folded passes, group 9 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(9)
}  // namespace pstd
