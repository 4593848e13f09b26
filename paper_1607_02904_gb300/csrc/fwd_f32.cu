// Mixed-precision instances of the force kernel (float terms, double sums).
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_f32(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s,
                       bool virial) {
  switch (c->ns) {
    case 1: return fwd::launch_species<float, 1>(c, f, acc, eatom, s, virial);
    case 2: return fwd::launch_species<float, 2>(c, f, acc, eatom, s, virial);
    default: return fwd::launch_species<float, 0>(c, f, acc, eatom, s, virial);
  }
}
fwd::FwdArgs<float> resident_args(Ctx* c) { return fwd::make_args<float>(c, c->d_extra, nullptr, nullptr, false); }

int launch_forward_batch_f32(Ctx* c, double* f, cudaStream_t s) {
  return fwd::launch_batch<float>(c, f, s);
}
}  // namespace tgb
