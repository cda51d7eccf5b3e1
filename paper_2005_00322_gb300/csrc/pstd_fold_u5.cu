// pstd_fold_u5.cu -- fixed schedules of the folded passes, group 5 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(5)
}  // namespace pstd
