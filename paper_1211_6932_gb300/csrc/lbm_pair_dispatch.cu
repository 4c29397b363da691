// Dispatch of the FP32 pair kernel to its instantiations, one translation unit per viscosity
// rule (lbm_pair_*.cu).
#include "lbm_internal.h"

namespace lbm {

#define LBM_BY_RULE(FN, ...)                                                       \
  switch (rule) {                                                                  \
    case VISC_CONST: return FN<VISC_CONST>(__VA_ARGS__);                           \
    case VISC_STEP: return FN<VISC_STEP>(__VA_ARGS__);                             \
    case VISC_LINEAR: return FN<VISC_LINEAR>(__VA_ARGS__);                         \
    case PAIR_PSI64: return FN<PAIR_PSI64>(__VA_ARGS__);                           \
    default: return FN<PAIR_ANY>(__VA_ARGS__);                                     \
  }

cudaError_t launch_pair(int rule, int nt, int rows, int full, const RowMaps& maps, int slab,
                        float* fout,
                        const InstParams* d_inst, const WorkItem* d_items, int n_items,
                        int* d_status, const PairConsts& shared, bool dependent,
                        cudaStream_t st) {
  LBM_BY_RULE(launch_pair_step, nt, rows, full, maps, slab, fout, d_inst, d_items, n_items, d_status, shared,
              dependent, st)
}

cudaError_t launch_persist(int rule, int nt, int kind, const RowMaps& maps, int slab,
                           float* slab0, float* slab1,
                           const InstParams* d_inst, const WorkItem* items2,
                           const ItemLink* links2, int n_items, int steps, int* queue,
                           int* done, int* d_status, int grid, int dep_limit,
                           const PairConsts& shared, cudaStream_t st) {
  LBM_BY_RULE(launch_pair_persist, nt, kind, maps, slab, slab0, slab1, d_inst, items2, links2, n_items,
              steps, queue, done, d_status, grid, dep_limit, shared, st)
}

int persist_occupancy(int rule, int nt, int kind) {
  LBM_BY_RULE(pair_persist_occupancy, nt, kind)
}

int pair_occupancy(int rule, int nt, int rows) { LBM_BY_RULE(pair_step_occupancy, nt, rows) }

}  // namespace lbm
