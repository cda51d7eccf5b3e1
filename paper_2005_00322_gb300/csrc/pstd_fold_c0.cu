// pstd_fold_c0.cu -- convolution passes on folded transforms, group 0 of pstd_fold_list.h.
#include "pstd_fkernels.cuh"

namespace pstd {
PSTD_CONV_UNIT(0)
}  // namespace pstd
