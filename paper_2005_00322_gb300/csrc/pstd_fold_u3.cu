// pstd_fold_u3.cu -- fixed schedules of the folded passes, group 3 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(3)
}  // namespace pstd
