// FP32 pair-kernel instantiations: batches whose instances differ in viscosity rule, b, G or rates.
#include "lbm_pair_impl.cuh"

LBM_INSTANTIATE_PAIR(lbm::PAIR_ANY)
