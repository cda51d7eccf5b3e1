// pstd_fold_c3.cu -- convolution passes on folded transforms, group 3 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_CONV_UNIT(3)
}  // namespace pstd
