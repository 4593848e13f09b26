// FP64 force kernel: instances for boxes with a long edge.
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_f64_long(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s, bool virial) {
  fwd::launch_buckets<double, 0, false, 1>(c, fwd::make_args<double>(c, f, acc, eatom, virial), s);
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}
int launch_forward_batch_f64_long(Ctx* c, double* f, cudaStream_t s) {
  if (c->n > 0) fwd::launch_buckets<double, 0, true, 1>(c, fwd::make_args<double>(c, f, nullptr, c->d_eatom), s);
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}
}  // namespace tgb
