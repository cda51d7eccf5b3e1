// pstd_fold_c2.cu -- convolution passes on folded transforms, group 2 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_CONV_UNIT(2)
}  // namespace pstd
