// FP64 force kernel: instances for batches of systems.
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_batch_f64(Ctx* c, double* f, cudaStream_t s) {
  return fwd::launch_batch<double>(c, f, s);
}
}  // namespace tgb
