// pstd_fold_u8.cu -- fixed schedules of the folded passes, group 8 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_FOLD_UNIT(8)
}  // namespace pstd
