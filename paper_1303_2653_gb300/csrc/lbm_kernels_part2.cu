// D3Q19 in FP64 and FP32: a part of the instantiations of lbm_kernels.cu.
#define LBDPS_LBM_PART 2
#include "lbm_kernels.cu"
