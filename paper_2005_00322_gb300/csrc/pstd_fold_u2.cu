// pstd_fold_u2.cu -- fixed schedules of the folded passes, group 2 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(2)
}  // namespace pstd
