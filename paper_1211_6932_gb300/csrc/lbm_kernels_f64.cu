// FP64 instantiations of the step kernel and helpers.
#include "lbm_kernels_impl.cuh"

namespace lbm {

template <>
cudaError_t launch_sweep<double>(bool, int nt, int mode, int full, const double* fin, double* fout,
                                 const InstParams* d_inst, const WorkItem* d_items, int n_items,
                                 const MomArgs<double>& mo, int* d_status, cudaStream_t st) {
  if (nt == 64) return launch_sweep_mode<double, 64, false>(mode, full, fin, fout, d_inst, d_items, n_items, mo, d_status, st);
  if (nt == 128) return launch_sweep_mode<double, 128, false>(mode, full, fin, fout, d_inst, d_items, n_items, mo, d_status, st);
  return cudaErrorInvalidValue;
}

template <int NT, bool FULL>
static cudaError_t launch_short64_cfg(const RowMaps& maps, int slab, double* fout,
                                      const InstParams* d_inst, const WorkItem* d_items,
                                      int n_items, int* d_status, cudaStream_t st) {
  constexpr size_t smem = Short64Cfg<NT>::BYTES;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = ensure_smem_attr(short64_kernel<NT, FULL>, smem, done);
  if (e != cudaSuccess) return e;
  if (n_items <= 0) return cudaSuccess;
  return launch_kernel(short64_kernel<NT, FULL>, n_items, NT, smem, false, st, maps, slab, fout,
                       d_inst, d_items, n_items, d_status);
}

cudaError_t launch_short64(int nt, int full, const RowMaps& maps, int slab, double* fout,
                           const InstParams* d_inst, const WorkItem* d_items, int n_items,
                           int* d_status, cudaStream_t st) {
  if (nt == 64)
    return full ? launch_short64_cfg<64, true>(maps, slab, fout, d_inst, d_items, n_items, d_status, st)
                : launch_short64_cfg<64, false>(maps, slab, fout, d_inst, d_items, n_items, d_status, st);
  if (nt == 128)
    return full ? launch_short64_cfg<128, true>(maps, slab, fout, d_inst, d_items, n_items, d_status, st)
                : launch_short64_cfg<128, false>(maps, slab, fout, d_inst, d_items, n_items, d_status, st);
  return cudaErrorInvalidValue;
}

template <>
int sweep_occupancy<double>(int nt) {
  if (nt == 64) return occupancy_cfg<double, 64>();
  if (nt == 128) return occupancy_cfg<double, 128>();
  return 1;
}

}  // namespace lbm

LBM_INSTANTIATE_HELPERS(double)
