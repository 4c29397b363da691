// FP32 (deviation storage): the one-column step kernel, the moments passes and the helpers.
#include "lbm_pair_impl.cuh"

namespace lbm {

template <>
cudaError_t launch_sweep<float>(bool psi64, int nt, int mode, int full, const float* fin,
                                float* fout, const InstParams* d_inst, const WorkItem* d_items,
                                int n_items, const MomArgs<float>& mo, int* d_status,
                                cudaStream_t st) {
#define LBM_SWEEP_NT(T)                                                                         \
  if (nt == T)                                                                                  \
    return psi64 ? launch_sweep_mode<float, T, true>(mode, full, fin, fout, d_inst, d_items,    \
                                                     n_items, mo, d_status, st)                 \
                 : launch_sweep_mode<float, T, false>(mode, full, fin, fout, d_inst, d_items,   \
                                                      n_items, mo, d_status, st);
  LBM_SWEEP_NT(64)
  LBM_SWEEP_NT(128)
  LBM_SWEEP_NT(256)
#undef LBM_SWEEP_NT
  return cudaErrorInvalidValue;
}

template <int VISC>
static cudaError_t launch_moments_cfg(int nt, int full, const RowMaps& maps, int slab,
                                      const InstParams* d_inst, const WorkItem* d_items,
                                      int n_items, const MomArgs<float>& mo, int* d_status,
                                      const PairConsts& shared, cudaStream_t st) {
#define LBM_PAIR_MOM(T)                                                                     \
  if (nt == T)                                                                              \
    return full ? launch_sweep2_cfg<T, MODE_MOMENTS, true, VISC>(                           \
                      maps, slab, nullptr, d_inst, d_items, n_items, mo, d_status, shared,  \
                      false, st)                                                            \
                : launch_sweep2_cfg<T, MODE_MOMENTS, false, VISC>(                          \
                      maps, slab, nullptr, d_inst, d_items, n_items, mo, d_status, shared,  \
                      false, st);
  LBM_PAIR_MOM(32)
  LBM_PAIR_MOM(64)
  LBM_PAIR_MOM(96)
  LBM_PAIR_MOM(128)
#undef LBM_PAIR_MOM
  return cudaErrorInvalidValue;
}

cudaError_t launch_pair_moments(int rule, int nt, int full, const RowMaps& maps, int slab,
                                const InstParams* d_inst, const WorkItem* d_items, int n_items,
                                const MomArgs<float>& mo, int* d_status,
                                const PairConsts& shared, cudaStream_t st) {
  // PAIR_ANY takes every constant from the instance
  return rule == PAIR_PSI64
             ? launch_moments_cfg<PAIR_PSI64>(nt, full, maps, slab, d_inst, d_items, n_items, mo,
                                              d_status, shared, st)
             : launch_moments_cfg<PAIR_ANY>(nt, full, maps, slab, d_inst, d_items, n_items, mo,
                                            d_status, shared, st);
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
