// FP32 pair-kernel instantiations: constant viscosity.
#include "lbm_pair_impl.cuh"

LBM_INSTANTIATE_PAIR(lbm::VISC_CONST)
