// FP64 storage and arithmetic (parity path).
#include "pflb_launch.cuh"
namespace pflb {
cudaError_t fold_diag(Lattice &L, int d, int64_t step, pflb_diag_raw_t *out) {
  return launch_dependent(k_diag_fold, 1, 256, 0, L.stream, (const double *)diag_acc(L, d),
                          (const int *)L.err, step, out);
}
PFLB_INSTANTIATE(double, double)
}
