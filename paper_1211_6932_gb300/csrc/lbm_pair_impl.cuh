// Launchers of the FP32 pair kernel (two columns per thread, packed float2 arithmetic) for
// one viscosity rule (VISC_*, PAIR_ANY or PAIR_PSI64), one translation unit per rule.
#pragma once
#include "lbm_kernels_impl.cuh"

namespace lbm {

template <int NT, int MODE, bool FULL, int VISC>
static cudaError_t launch_sweep2_cfg(const RowMaps& maps, int slab, float* fout, const InstParams* d_inst,
                                     const WorkItem* d_items, int n_items,
                                     const MomArgs<float>& mo, int* d_status,
                                     const PairConsts& shared, bool dependent, cudaStream_t st) {
  constexpr size_t smem = Sweep2Cfg<NT>::BYTES;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = ensure_smem_attr(sweep2_kernel<NT, MODE, FULL, VISC>, smem, done);
  if (e != cudaSuccess) return e;
  if (n_items <= 0) return cudaSuccess;
  return launch_kernel(sweep2_kernel<NT, MODE, FULL, VISC>, n_items, NT, smem, dependent, st, maps,
                       slab, fout, d_inst, d_items, n_items, mo, d_status, shared);
}

// Chunks of at most ROWS rows (sweep2_short_kernel).
template <int NT, int ROWS, bool FULL, int VISC>
static cudaError_t launch_short_cfg(const RowMaps& maps, int slab, float* fout,
                                    const InstParams* d_inst, const WorkItem* d_items,
                                    int n_items, int* d_status, const PairConsts& shared,
                                    bool dependent, cudaStream_t st) {
  constexpr size_t smem = ShortCfg<NT, ROWS>::BYTES;
  static std::atomic<unsigned long long> done{0};
  cudaError_t e = ensure_smem_attr(sweep2_short_kernel<NT, ROWS, FULL, VISC>, smem, done);
  if (e != cudaSuccess) return e;
  if (n_items <= 0) return cudaSuccess;
  return launch_kernel(sweep2_short_kernel<NT, ROWS, FULL, VISC>, n_items, NT, smem, dependent, st,
                       maps, slab, fout, d_inst, d_items, n_items, d_status, shared);
}

// Persistent pair kernel (sweep2_persist_kernel) with `grid` CTAs.
template <int NT, int KIND, int VISC>
static cudaError_t launch_persist2_cfg(const RowMaps& maps, int slab, float* slab0, float* slab1, const InstParams* d_inst,
                                       const WorkItem* items2, const ItemLink* links2,
                                       int n_items, int steps, int* queue, int* done,
                                       int* d_status, int grid, int dep_limit,
                                       const PairConsts& shared, cudaStream_t st) {
  constexpr size_t smem = Sweep2Cfg<NT>::BYTES;
  static std::atomic<unsigned long long> flag{0};
  cudaError_t e = ensure_smem_attr(sweep2_persist_kernel<NT, KIND, VISC>, smem, flag);
  if (e != cudaSuccess) return e;
  if (n_items <= 0 || steps <= 0 || grid <= 0) return cudaSuccess;
  sweep2_persist_kernel<NT, KIND, VISC><<<grid, NT, smem, st>>>(
      maps, slab, slab0, slab1, d_inst, items2, links2, n_items, steps, queue, done, d_status, dep_limit,
      shared);
  return cudaGetLastError();
}

template <typename F>
static int pair_occupancy(F* fn, int nt, size_t smem) {
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int occ = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, nt, smem);
  return (e == cudaSuccess && occ > 0) ? occ : 1;
}

template <int VISC>
cudaError_t launch_pair_step(int nt, int rows, int full, const RowMaps& maps, int slab,
                             float* fout, const InstParams* d_inst, const WorkItem* d_items,
                             int n_items, int* d_status, const PairConsts& shared,
                             bool dependent, cudaStream_t st) {
  const MomArgs<float> mo{};
#define LBM_PAIR_KIND(T, F)                                                                    \
  if (nt == T && (full != 0) == F)                                                             \
    return rows == 1   ? launch_short_cfg<T, 1, F, VISC>(maps, slab, fout, d_inst, d_items,    \
                                                         n_items, d_status, shared, dependent, \
                                                         st)                                   \
           : rows == 2 ? launch_short_cfg<T, 2, F, VISC>(maps, slab, fout, d_inst, d_items,    \
                                                         n_items, d_status, shared, dependent, \
                                                         st)                                   \
                       : launch_sweep2_cfg<T, MODE_STEP, F, VISC>(maps, slab, fout, d_inst,    \
                                                                  d_items, n_items, mo,        \
                                                                  d_status, shared, dependent, \
                                                                  st);
#define LBM_PAIR(T) LBM_PAIR_KIND(T, true) LBM_PAIR_KIND(T, false)
  LBM_PAIR(32)
  LBM_PAIR(64)
  LBM_PAIR(96)
  LBM_PAIR(128)
#undef LBM_PAIR
#undef LBM_PAIR_KIND
  return cudaErrorInvalidValue;
}

template <int VISC>
cudaError_t launch_pair_persist(int nt, int kind, const RowMaps& maps, int slab,
                                float* slab0, float* slab1,
                                const InstParams* d_inst, const WorkItem* items2,
                                const ItemLink* links2, int n_items, int steps, int* queue,
                                int* done, int* d_status, int grid, int dep_limit,
                                const PairConsts& shared, cudaStream_t st) {
#define LBM_PERSIST_KIND(T, K)                                                               \
  if (nt == T && kind == K)                                                                  \
    return launch_persist2_cfg<T, K, VISC>(maps, slab, slab0, slab1, d_inst, items2, links2, n_items,    \
                                           steps, queue, done, d_status, grid, dep_limit,    \
                                           shared, st);
#define LBM_PERSIST(T)                  \
  LBM_PERSIST_KIND(T, PERSIST_STRIP)    \
  LBM_PERSIST_KIND(T, PERSIST_FULL)     \
  LBM_PERSIST_KIND(T, PERSIST_MIXED)
  LBM_PERSIST(32)
  LBM_PERSIST(64)
  LBM_PERSIST(96)
  LBM_PERSIST(128)
#undef LBM_PERSIST
#undef LBM_PERSIST_KIND
  return cudaErrorInvalidValue;
}

template <int VISC>
int pair_persist_occupancy(int nt, int kind) {
#define LBM_PERSIST_OCC(T)                                                                     \
  if (nt == T)                                                                                 \
    return kind == PERSIST_MIXED                                                               \
               ? pair_occupancy(sweep2_persist_kernel<T, PERSIST_MIXED, VISC>, T,              \
                                Sweep2Cfg<T>::BYTES)                                           \
           : kind == PERSIST_FULL ? pair_occupancy(sweep2_persist_kernel<T, PERSIST_FULL, VISC>, \
                                                   T, Sweep2Cfg<T>::BYTES)                     \
                                  : pair_occupancy(sweep2_persist_kernel<T, PERSIST_STRIP, VISC>, \
                                                   T, Sweep2Cfg<T>::BYTES);
  LBM_PERSIST_OCC(32)
  LBM_PERSIST_OCC(64)
  LBM_PERSIST_OCC(96)
  LBM_PERSIST_OCC(128)
#undef LBM_PERSIST_OCC
  return 1;
}

template <int VISC>
int pair_step_occupancy(int nt, int rows) {
#define LBM_PAIR_OCC(T)                                                                       \
  if (nt == T)                                                                                \
    return rows == 1   ? pair_occupancy(sweep2_short_kernel<T, 1, false, VISC>, T,            \
                                        ShortCfg<T, 1>::BYTES)                                \
           : rows == 2 ? pair_occupancy(sweep2_short_kernel<T, 2, false, VISC>, T,            \
                                        ShortCfg<T, 2>::BYTES)                                \
                       : pair_occupancy(sweep2_kernel<T, MODE_STEP, false, VISC>, T,          \
                                        Sweep2Cfg<T>::BYTES);
  LBM_PAIR_OCC(32)
  LBM_PAIR_OCC(64)
  LBM_PAIR_OCC(96)
  LBM_PAIR_OCC(128)
#undef LBM_PAIR_OCC
  return 1;
}

}  // namespace lbm

#define LBM_INSTANTIATE_PAIR(V)                                                               \
  template cudaError_t lbm::launch_pair_step<V>(int, int, int, const lbm::RowMaps&, int, float*,               \
                                                const lbm::InstParams*, const lbm::WorkItem*, \
                                                int, int*, const lbm::PairConsts&, bool,      \
                                                cudaStream_t);                                \
  template cudaError_t lbm::launch_pair_persist<V>(                                           \
      int, int, const lbm::RowMaps&, int, float*, float*, const lbm::InstParams*,          \
      const lbm::WorkItem*,                 \
      const lbm::ItemLink*, int, int, int*, int*, int*, int, int, const lbm::PairConsts&,     \
      cudaStream_t);                                                                          \
  template int lbm::pair_persist_occupancy<V>(int, int);                                      \
  template int lbm::pair_step_occupancy<V>(int, int);
