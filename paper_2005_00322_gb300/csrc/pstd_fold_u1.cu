// pstd_fold_u1.cu -- fixed schedules of the folded passes, group 1 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(1)
}  // namespace pstd
