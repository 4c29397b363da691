// FP32 pair-kernel instantiations: a viscosity step.
#include "lbm_pair_impl.cuh"

LBM_INSTANTIATE_PAIR(lbm::VISC_STEP)
