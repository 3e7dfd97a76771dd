// D2Q9 in the 16-bit storages: a part of the instantiations of lbm_kernels.cu.
#define LBDPS_LBM_PART 1
#include "lbm_kernels.cu"
