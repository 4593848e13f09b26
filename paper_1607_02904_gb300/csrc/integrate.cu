// Per-step atom kernels: position packing for the force kernels and the
// velocity-Verlet kick/drift on the FP64 state (x, v, f).
#include "step.cuh"

namespace tgb {
namespace {

template <bool P64>
__global__ void k_pack(const __grid_constant__ PackArgs a, const double* __restrict__ x) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  float d2 = 0.0f;
  if (i < a.n) {
    const double* xi = x + 3 * (size_t)i;
    d2 = pack_one<P64>(a, i, a.types[i], xi[0], xi[1], xi[2]);
  }
  track_max(a, d2);
}

// The FP64 path's positions in a box with a long edge (Grid::long64), in place of
// those that the packing kernels wrote: a pass of its own, so that no other box
// pays for its arithmetic (inside k_step it cost 2.5 us of 512,000 atoms).
__global__ void k_pos_long(const __grid_constant__ PackArgs a, const double* __restrict__ x) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  const Box64& b = a.sys ? a.sys[a.atom_sys[i]].box : a.box;
  const double* xi = x + 3 * (size_t)i;
  ipos4 p;
  p.w = word64(xi[0], xi[1], xi[2], a.types[i]);
  p.x = wrap_long(xi[0], a.fix64, b, 0, p.w);
  p.y = wrap_long(xi[1], a.fix64, b, 1, p.w);
  p.z = wrap_long(xi[2], a.fix64, b, 2, p.w);
  a.pos64[i] = p;
}

// One step of all atoms (step_atom); optional kinetic energy of the previous
// step; clears the accumulator for the coming force evaluation.
template <bool MG, bool KE>
__global__ void k_step(const __grid_constant__ PackArgs pk, const __grid_constant__ GatherArgs ga, int gather_, double* __restrict__ x,
                       double* __restrict__ v, const double* __restrict__ f, const __grid_constant__ Coef cf,
                       double dt, int kick, int do_pack, double* ke_row_, double* acc_zero,
                       double* __restrict__ snap) {
  pdl_wait();  // the previous kernel's writes (a launch with launch_pdl)
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int gather = MG ? 1 : gather_;
  double* const ke_row = MG ? (KE ? ke_row_ : nullptr) : ke_row_;
  if (acc_zero && i < 8) acc_zero[i * ACC_STRIDE] = 0.0;
  float d2 = 0.0f;
  double ke = 0.0;   // FP64 path
  float kef = 0.0f;  // mixed path: in float (m v^2 / 2 in amu A^2/ps^2, ~1e1 per atom)
  if (i < pk.n)
    step_atom<MG>(pk, ga, gather, x, v, f, cf, dt, kick, do_pack, ke_row != nullptr, snap, i, d2, ke, kef);
  if (do_pack) track_max(pk, d2);
  if (ke_row) {
    if (MG || (gather && !ga.fp64 && !ga.atomic_mode))
      block_sum_add_f(kef, ke_row);
    else
      block_sum_add(ke, ke_row);
  }
}

// closing half kick with gathered forces, which are also written to f.
// MG: the mixed path's gathered forces (float slots, compensated sums): the
// force is the float pair carried into double (one rounding), the velocity
// increment is formed in float as in k_step, and the kinetic energy in float
// with a compensated block sum; otherwise all in double.
template <bool MG>
__global__ void k_final_kick(GatherArgs ga, const int* __restrict__ types,
                             double* __restrict__ v, double* __restrict__ f, const __grid_constant__ Coef cf,
                             double* ke_row) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (MG) {
    float kef = 0.0f;
    if (i < ga.n) {
      const int t = types[i];
      const size_t b = 3 * (size_t)i;
      const double v0 = v[b], v1 = v[b + 1], v2 = v[b + 2];
      double E0, E1, E2;  // fallback-buffer forces (zero unless flagged)
      float sc[6];
      gather_force(ga, i, E0, E1, E2, sc);
      const bool extra = ga.flags[FLAG_EXTRA] | ga.flags[FLAG_EXTRA_STICKY];
      const float kf = cf.cf[t];
      float d0 = kf * sc[0] + kf * sc[3];
      float d1 = kf * sc[1] + kf * sc[4];
      float d2 = kf * sc[2] + kf * sc[5];
      double F0 = gather_f2d(sc[0]) + gather_f2d(sc[3]);
      double F1 = gather_f2d(sc[1]) + gather_f2d(sc[4]);
      double F2 = gather_f2d(sc[2]) + gather_f2d(sc[5]);
      if (extra) {
        d0 = fmaf(kf, d2f_bits(E0), d0);
        d1 = fmaf(kf, d2f_bits(E1), d1);
        d2 = fmaf(kf, d2f_bits(E2), d2);
        F0 += E0;
        F1 += E1;
        F2 += E2;
      }
      const double w0 = v0 + gather_f2d(d0), w1 = v1 + gather_f2d(d1), w2 = v2 + gather_f2d(d2);
      f[b] = F0;
      f[b + 1] = F1;
      f[b + 2] = F2;
      v[b] = w0;
      v[b + 1] = w1;
      v[b + 2] = w2;
      if (ke_row) {
        const float u0 = d2f_bits(w0), u1 = d2f_bits(w1), u2 = d2f_bits(w2);
        kef = cf.hmf[t] * fmaf(u0, u0, fmaf(u1, u1, u2 * u2));
      }
    }
    if (ke_row) block_sum_add_f(kef, ke_row);
    return;
  }
  double ke = 0.0;
  if (i < ga.n) {
    const int t = types[i];
    const size_t b = 3 * (size_t)i;
    const double v0 = v[b], v1 = v[b + 1], v2 = v[b + 2];
    double F0, F1, F2;
    gather_force(ga, i, F0, F1, F2);
    const double cu = cf.c[t];
    const double w0 = fma(cu, F0, v0), w1 = fma(cu, F1, v1), w2 = fma(cu, F2, v2);
    f[b] = F0;
    f[b + 1] = F1;
    f[b + 2] = F2;
    v[b] = w0;
    v[b + 1] = w1;
    v[b + 2] = w2;
    ke = 0.5 * cf.m[t] * fma(w0, w0, fma(w1, w1, w2 * w2));
  }
  if (ke_row) block_sum_add(ke, ke_row);
}

__global__ void k_gather(GatherArgs ga, double* __restrict__ f) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ga.n) return;
  double F[3];
  gather_force(ga, i, F[0], F[1], F[2]);
  f[3 * (size_t)i] = F[0];
  f[3 * (size_t)i + 1] = F[1];
  f[3 * (size_t)i + 2] = F[2];
}

// one block per system: sums of the per-atom energy and virial over the
// system's atom range (fixed order: deterministic)
__global__ void k_system_sums(const int* __restrict__ off, const double* __restrict__ eatom,
                              const double* __restrict__ vatom, double* __restrict__ energy,
                              double* __restrict__ virial) {
  const int sys = blockIdx.x;
  const int a0 = off[sys], a1 = off[sys + 1];
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int i = a0 + threadIdx.x; i < a1; i += blockDim.x) {
    v[0] += eatom[i];
    for (int q = 0; q < 6; ++q) v[1 + q] += vatom[6 * (size_t)i + q];
  }
  __shared__ double part[7][8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int q = 0; q < 7; ++q) {
    double t = v[q];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) part[q][wid] = t;
  }
  __syncthreads();
  if (threadIdx.x < 7) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[threadIdx.x][w];
    if (threadIdx.x == 0) {
      if (energy) energy[sys] = t;
    } else if (virial) {
      virial[6 * (size_t)sys + threadIdx.x - 1] = t;
    }
  }
}

// one thread: rebuild when the running max squared displacement (float bits,
// non-negative) exceeds lim2
__global__ void k_decide_rebuild(int* flags, float lim2, cudaGraphConditionalHandle h) {
  const bool go = __int_as_float(flags[FLAG_DMAX]) > lim2;
  if (go) flags[FLAG_NREBUILD] += 1;
  cudaGraphSetConditional(h, go ? 1u : 0u);
}

// rows: ACC_LEN doubles per step (energy, virial[6], kinetic in mass units)
__global__ void k_thermo_rows(const double* rows, int nsteps, double mvv2e, double* out) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= nsteps) return;
  const double pe = rows[ACC_LEN * (size_t)s];
  const double ke = rows[ACC_LEN * (size_t)s + 7 * ACC_STRIDE] * mvv2e;
  out[3 * (size_t)s + 0] = pe;
  out[3 * (size_t)s + 1] = ke;
  out[3 * (size_t)s + 2] = pe + ke;
}

}  // namespace

int launch_pos_long(Ctx* c, const double* x, cudaStream_t s) {
  if (c->n == 0 || c->precision != TERSOFF_FP64 || !c->grid.long64) return TERSOFF_OK;
  const int B = c->opt_block;
  TGB_CUDA(c, launch_pdl(k_pos_long, (c->n + B - 1) / B, B, 0, s, make_pack(c, false), x));
  c->launches++;
  return TERSOFF_OK;
}

int launch_pack_positions(Ctx* c, const double* x, bool build, cudaStream_t s) {
  if (c->n == 0) return TERSOFF_OK;
  const int B = c->opt_block;
  TGB_CUDA(c, launch_pdl(c->precision == TERSOFF_FP64 ? k_pack<true> : k_pack<false>, (c->n + B - 1) / B, B, 0, s,
                         make_pack(c, !build, build), x));
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return launch_pos_long(c, x, s);
}

int launch_md_step(Ctx* c, double* x, double* v, double* f, double dt, int kick, bool pack,
                   double* ke_row, double* acc_zero, cudaStream_t s, double* snap) {
  const int B = c->opt_block;
  const GatherArgs ga = make_gather(c);
  const int grid = (c->n + B - 1) / B;
  if (kick == 2 && !ga.fp64 && !ga.atomic_mode) {
    if (ke_row)
      TGB_CUDA(c, launch_pdl(k_step<true, true>, grid, B, 0, s, make_pack(c, true), ga, 1, x, v,
                             f, c->coef, dt, kick, pack ? 1 : 0, ke_row, acc_zero,
                             (double*)nullptr));
    else
      TGB_CUDA(c, launch_pdl(k_step<true, false>, grid, B, 0, s, make_pack(c, true), ga, 1, x, v,
                             f, c->coef, dt, kick, pack ? 1 : 0, (double*)nullptr, acc_zero,
                             (double*)nullptr));
  } else {
    TGB_CUDA(c, launch_pdl(k_step<false, false>, grid, B, 0, s, make_pack(c, true), ga,
                           kick == 2 ? 1 : 0, x, v, f, c->coef, dt, kick, pack ? 1 : 0, ke_row,
                           acc_zero, snap));
  }
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return pack ? launch_pos_long(c, x, s) : TERSOFF_OK;
}

int launch_final_kick(Ctx* c, double* v, double* f, double* ke_row, cudaStream_t s) {
  const int B = c->opt_block;
  const GatherArgs ga = make_gather(c);
  if (!ga.fp64 && !ga.atomic_mode)
    TGB_CUDA(c, launch_pdl(k_final_kick<true>, (c->n + B - 1) / B, B, 0, s, ga, c->d_types, v, f, c->coef, ke_row));
  else
    TGB_CUDA(c, launch_pdl(k_final_kick<false>, (c->n + B - 1) / B, B, 0, s, ga, c->d_types, v, f, c->coef, ke_row));
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

int launch_gather(Ctx* c, double* f, cudaStream_t s) {
  if (c->n == 0) return TERSOFF_OK;
  const int B = c->opt_block;
  k_gather<<<(c->n + B - 1) / B, B, 0, s>>>(make_gather(c), f);
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

int launch_system_sums(Ctx* c, double* energy, double* virial, cudaStream_t s) {
  if (c->n_sys <= 0) return TERSOFF_OK;
  k_system_sums<<<c->n_sys, 256, 0, s>>>(c->d_sys_off, c->d_eatom, c->d_vatom, energy, virial);
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

int launch_decide_rebuild(Ctx* c, float lim2, cudaGraphConditionalHandle h, cudaStream_t s) {
  k_decide_rebuild<<<1, 1, 0, s>>>(c->d_flags, lim2, h);
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

int launch_thermo_rows(Ctx* c, const double* rows, int nsteps, double mvv2e, double* thermo,
                       cudaStream_t s) {
  if (nsteps <= 0) return TERSOFF_OK;
  k_thermo_rows<<<(nsteps + 127) / 128, 128, 0, s>>>(rows, nsteps, mvv2e, thermo);
  c->launches++;
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

}  // namespace tgb
