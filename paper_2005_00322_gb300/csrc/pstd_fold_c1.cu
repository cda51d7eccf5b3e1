// pstd_fold_c1.cu -- convolution passes on folded transforms, group 1 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_CONV_UNIT(1)
}  // namespace pstd
