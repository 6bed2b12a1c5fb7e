// Folded skew-packed streaming kernel, GROM_F64 storage.
#include "k1t.cuh"

namespace grom {

cudaError_t k1t_dispatch_f64(int qm, int nb, const K1TArgs& a, const StepArgs& st, int grid, size_t smem,
                             cudaStream_t s) {
  switch (qm) {  // grom_max_n: n <= 4096
    case 1: return k1t_pick_nb<GROM_F64, 1>(nb, a, st, grid, smem, s);
    case 2: return k1t_pick_nb<GROM_F64, 2>(nb, a, st, grid, smem, s);
    case 4: return k1t_pick_nb<GROM_F64, 4>(nb, a, st, grid, smem, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace grom
