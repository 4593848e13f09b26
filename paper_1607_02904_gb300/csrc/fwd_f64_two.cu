// FP64 force kernel: two-species instances.
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_f64_two(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s,
                           bool virial) {
  return fwd::launch_species<double, 2>(c, f, acc, eatom, s, virial);
}
}  // namespace tgb
