// Launchers of the step and helper kernels for one storage type (included once per type).
#pragma once
#include <atomic>

#include "lbm_aux.cuh"
#include "lbm_internal.h"

namespace lbm {

// Set a kernel's dynamic shared-memory limit once per device: the attribute belongs to the
// current device's context, so `done` keeps one bit per device ordinal (below 64; others
// are set on every launch).
template <typename F>
static cudaError_t ensure_smem_attr(F* fn, size_t smem, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess && bit) done.fetch_or(bit);
  return e;
}

// Launch a kernel, as a programmatic dependent of the stream's previous kernel if asked
// (step_begin waits for that one's completion).
template <typename... P, typename... A>
static cudaError_t launch_kernel(void (*kernel)(P...), int blocks, int threads, size_t smem,
                                 bool dependent, cudaStream_t st, const A&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <typename S, int NT, int MODE, int FULL, bool PSI64>
static cudaError_t launch_sweep_cfg(const S* fin, S* fout, const InstParams* d_inst,
                                    const WorkItem* d_items, int n_items, const MomArgs<S>& mo,
                                    int* d_status, cudaStream_t st) {
  constexpr size_t smem = SweepCfg<S, NT>::BYTES;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = ensure_smem_attr(sweep_kernel<S, NT, MODE, FULL, PSI64>, smem, done);
  if (e != cudaSuccess) return e;
  if (n_items <= 0) return cudaSuccess;
  sweep_kernel<S, NT, MODE, FULL, PSI64><<<n_items, NT, smem, st>>>(fin, fout, d_inst, d_items,
                                                                   n_items, mo, d_status);
  return cudaGetLastError();
}

template <typename S, int NT, bool PSI64>
static cudaError_t launch_sweep_mode(int mode, int full, const S* fin, S* fout, const InstParams* d_inst,
                                     const WorkItem* d_items, int n_items,
                                     const MomArgs<S>& mo, int* d_status, cudaStream_t st) {
#define LBM_SWEEP(M, F)                                                                         \
  launch_sweep_cfg<S, NT, M, F, PSI64>(fin, fout, d_inst, d_items, n_items, mo, d_status, st)
  if (mode == MODE_STEP) return full ? LBM_SWEEP(MODE_STEP, 1) : LBM_SWEEP(MODE_STEP, 0);
  return full == 2 ? LBM_SWEEP(MODE_MOMENTS, 2)
         : full    ? LBM_SWEEP(MODE_MOMENTS, 1)
                   : LBM_SWEEP(MODE_MOMENTS, 0);
#undef LBM_SWEEP
}

template <typename S, int NT>
static int occupancy_cfg() {
  constexpr size_t smem = SweepCfg<S, NT>::BYTES;
  cudaFuncSetAttribute(sweep_kernel<S, NT, MODE_STEP, 0, false>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &occ, sweep_kernel<S, NT, MODE_STEP, 0, false>, NT, smem);
  return (e == cudaSuccess && occ > 0) ? occ : 1;
}

static inline int grid_for(long long n) {
  long long g = (n + 255) / 256;
  if (g < 1) g = 1;
  if (g > 152 * 16) g = 152 * 16;
  return (int)g;
}

template <typename S>
cudaError_t launch_set_pops(const double* d_fc, S* buf, const InstParams& P, cudaStream_t st) {
  set_pops_kernel<S><<<grid_for((long long)P.nx * P.ny), 256, 0, st>>>(d_fc, buf, P);
  return cudaGetLastError();
}
template <typename S>
cudaError_t launch_get_pops(const S* buf, double* d_fc, const InstParams& P, cudaStream_t st) {
  get_pops_kernel<S><<<grid_for((long long)P.nx * P.ny), 256, 0, st>>>(buf, d_fc, P);
  return cudaGetLastError();
}
template <typename S>
cudaError_t launch_init_eq(const double* rho, const double* ux, const double* uy, S* buf,
                           const InstParams& P, int* d_bad, cudaStream_t st) {
  init_eq_kernel<S><<<grid_for((long long)P.nx * P.ny), 256, 0, st>>>(rho, ux, uy, buf, P,
                                                                      d_bad);
  return cudaGetLastError();
}
template <typename S>
cudaError_t launch_fill_ghosts(S* buf, const InstParams& P, cudaStream_t st) {
  fill_ghosts_kernel<S><<<grid_for((long long)Q * P.ny * 4), 256, 0, st>>>(buf, P);
  return cudaGetLastError();
}
template <typename S>
cudaError_t launch_psi(const double* d_rho, double* d_out, long long n,
                       const InstParams* d_inst, cudaStream_t st) {
  psi_kernel<S><<<grid_for(n), 256, 0, st>>>(d_rho, d_out, n, d_inst);
  return cudaGetLastError();
}

}  // namespace lbm

#define LBM_INSTANTIATE_HELPERS(S)                                                          \
  template cudaError_t lbm::launch_set_pops<S>(const double*, S*, const lbm::InstParams&,   \
                                               cudaStream_t);                               \
  template cudaError_t lbm::launch_get_pops<S>(const S*, double*, const lbm::InstParams&,   \
                                               cudaStream_t);                               \
  template cudaError_t lbm::launch_init_eq<S>(const double*, const double*, const double*,  \
                                              S*, const lbm::InstParams&, int*,             \
                                              cudaStream_t);                                \
  template cudaError_t lbm::launch_psi<S>(const double*, double*, long long,                \
                                          const lbm::InstParams*, cudaStream_t);            \
  template cudaError_t lbm::launch_fill_ghosts<S>(S*, const lbm::InstParams&, cudaStream_t);
