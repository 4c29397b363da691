// FP32 pair-kernel instantiations: viscosity linear in density.
#include "lbm_pair_impl.cuh"

LBM_INSTANTIATE_PAIR(lbm::VISC_LINEAR)
