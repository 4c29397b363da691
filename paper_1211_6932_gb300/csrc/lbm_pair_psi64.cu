// FP32 pair-kernel instantiations: single lattices with the psi_fp64 option.
#include "lbm_pair_impl.cuh"

LBM_INSTANTIATE_PAIR(lbm::PAIR_PSI64)
