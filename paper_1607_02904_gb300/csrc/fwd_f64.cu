// FP64 force kernel: one-species instances, and the choice of the path and the
// species count.
#include "fwd_launch.cuh"

namespace tgb {
int launch_forward_batch(Ctx* c, double* f, cudaStream_t s) {
  if (c->n == 0) return TERSOFF_OK;
  if (c->precision == TERSOFF_MIXED) return launch_forward_batch_f32(c, f, s);
  if (c->grid.long64 && fwd::use_lanes64(c)) return launch_forward_batch_f64_long(c, f, s);
  return launch_forward_batch_f64(c, f, s);
}

int launch_forward(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s, bool virial) {
  if (c->n == 0) return TERSOFF_OK;
  if (c->precision == TERSOFF_MIXED) return launch_forward_f32(c, f, acc, eatom, s, virial);
  if (c->grid.long64 && fwd::use_lanes64(c) && !(c->ablate & TERSOFF_ABLATE_FASTFWD))
    return launch_forward_f64_long(c, f, acc, eatom, s, virial);
  switch (c->ns) {
    case 1: return fwd::launch_species<double, 1>(c, f, acc, eatom, s, virial);
    case 2: return launch_forward_f64_two(c, f, acc, eatom, s, virial);
    default: return launch_forward_f64_any(c, f, acc, eatom, s, virial);
  }
}
}  // namespace tgb
