// FP32 (deviation storage): the one-column step kernel, the moments passes and the helpers.
#include "lbm_pair_impl.cuh"

namespace lbm {

template <>
cudaError_t launch_sweep<float>(int nt, int mode, int full, const float* fin, float* fout,
                                const InstParams* d_inst, const WorkItem* d_items, int n_items,
                                const MomArgs<float>& mo, int* d_status, cudaStream_t st) {
  if (nt == 64) return launch_sweep_mode<float, 64>(mode, full, fin, fout, d_inst, d_items, n_items, mo, d_status, st);
  if (nt == 128) return launch_sweep_mode<float, 128>(mode, full, fin, fout, d_inst, d_items, n_items, mo, d_status, st);
  if (nt == 256) return launch_sweep_mode<float, 256>(mode, full, fin, fout, d_inst, d_items, n_items, mo, d_status, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_pair_moments(int nt, int full, const RowMaps& maps, int slab,
                                const InstParams* d_inst, const WorkItem* d_items, int n_items,
                                const MomArgs<float>& mo, int* d_status, cudaStream_t st) {
  const PairConsts none{};  // every constant comes from the instance (PAIR_ANY)
#define LBM_PAIR_MOM(T)                                                                     \
  if (nt == T)                                                                              \
    return full ? launch_sweep2_cfg<T, MODE_MOMENTS, true, PAIR_ANY>(                       \
                      maps, slab, nullptr, d_inst, d_items, n_items, mo, d_status, none, false, st) \
                : launch_sweep2_cfg<T, MODE_MOMENTS, false, PAIR_ANY>(                      \
                      maps, slab, nullptr, d_inst, d_items, n_items, mo, d_status, none, false, st);
  LBM_PAIR_MOM(32)
  LBM_PAIR_MOM(64)
  LBM_PAIR_MOM(96)
  LBM_PAIR_MOM(128)
#undef LBM_PAIR_MOM
  return cudaErrorInvalidValue;
}

template <>
int sweep_occupancy<float>(int nt) {
  if (nt == 64) return occupancy_cfg<float, 64>();
  if (nt == 128) return occupancy_cfg<float, 128>();
  if (nt == 256) return occupancy_cfg<float, 256>();
  return 1;
}

}  // namespace lbm

LBM_INSTANTIATE_HELPERS(float)
