// FP64 force kernel: instances for a run-time species count.
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_f64_any(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s,
                           bool virial) {
  return fwd::launch_species<double, 0>(c, f, acc, eatom, s, virial);
}
}  // namespace tgb
