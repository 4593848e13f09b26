// Per-step atom arithmetic shared by the step kernels: position packing, the
// velocity-Verlet kick and drift, and the block sums of the kinetic energy.
#pragma once
#include "gather.cuh"
#include "internal.cuh"
#include "pos64.cuh"

namespace tgb {

// 1.5 * 2^52: adding it to a double of magnitude < 2^51 rounds it to an
// integer held in the low mantissa bits (IEEE-754 binary64 layout).
constexpr double ROUND_MAGIC = 6755399441055744.0;

struct PackArgs {
  int n;
  const double* qorg;    // 1.5*2^52 - o_i 2^S
  int4* qref;            // offsets at the build (displacement tracking)
  const int* types;
  int fp64;              // also write the FP64 path's positions
  int track;             // update the running max displacement
  int build;             // at a build: float offsets and displacement references
  double scale;          // 2^S
  float inv_scale;       // 2^-S
  float4* pos32;
  int4* posq;
  ipos4* pos64;
  int fix64;
  Box64 box;             // of a single system ...
  const SysShift* sys;   // ... or the systems' (batches) and each atom's system
  const int* atom_sys;
  int* flags;
};

// Packs atom i (species t) at position (x0, x1, x2); qo: its fixed-point
// origin words; returns its squared displacement since the build (A^2) when
// tracking. Loads are issued before any store.
// P64: the FP64 path's positions may be wanted (instances of the mixed path
// leave their arithmetic out, which costs registers).
template <bool P64>
__device__ __forceinline__ float pack_one(const PackArgs& a, int i, int t, double x0, double x1,
                                          double x2) {
  const double* qo = a.qorg + 3 * (size_t)i;
  const double qo0 = qo[0], qo1 = qo[1], qo2 = qo[2];
  int4 r = make_int4(0, 0, 0, 0);
  if (a.track) r = a.qref[i];
  // q = round((x - o) 2^S) with one rounding: fma(x, 2^S, magic - o 2^S)
  const long long mb = __double_as_longlong(ROUND_MAGIC);
  const int q0 = (int)(__double_as_longlong(fma(x0, a.scale, qo0)) - mb);
  const int q1 = (int)(__double_as_longlong(fma(x1, a.scale, qo1)) - mb);
  const int q2 = (int)(__double_as_longlong(fma(x2, a.scale, qo2)) - mb);
  a.posq[i] = make_int4(q0, q1, q2, t);
  if (a.build) {
    a.pos32[i] = make_float4((float)q0 * a.inv_scale, (float)q1 * a.inv_scale,
                             (float)q2 * a.inv_scale, __int_as_float(t));
    a.qref[i] = make_int4(q0, q1, q2, t);
  }
  if (P64 && a.fp64) {
    if (a.sys)
      a.pos64[i] = make_pos64(x0, x1, x2, t, a.fix64, a.sys[a.atom_sys[i]].box);
    else
      a.pos64[i] = make_pos64(x0, x1, x2, t, a.fix64, a.box);
  }
  float d2 = 0.0f;
  if (a.track) {
    const float d0 = (float)(q0 - r.x) * a.inv_scale;
    const float d1 = (float)(q1 - r.y) * a.inv_scale;
    const float dd = (float)(q2 - r.z) * a.inv_scale;
    d2 = d0 * d0 + d1 * d1 + dd * dd;
  }
  return d2;
}

// block max, one atomic per block (non-negative floats order like their bits)
__device__ __forceinline__ void track_max(const PackArgs& a, float d2) {
  if (!a.track) return;
  __shared__ float wmax[32];
  for (int o = 16; o > 0; o >>= 1) d2 = fmaxf(d2, __shfl_xor_sync(0xffffffffu, d2, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = d2;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.0f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, wmax[w]);
    atomicMax(&a.flags[FLAG_DMAX], __float_as_int(m));
  }
}

// double -> float rounded to nearest (ties away from zero) through the IEEE-754
// bit layouts, for values in float's normal range (velocities, forces); below
// it gives signed zero. Integer operations only: conversions involving double
// run on GB300's FP64 pipe at 1/62 of the FP32 rate.
__device__ __forceinline__ float d2f_bits(double d) {
  const unsigned long long u = __double_as_longlong(d);
  const unsigned long long mag = (u & 0x7fffffffffffffffull) + 0x10000000ull;  // + half ulp
  const int e = (int)(mag >> 52) - 1023 + 127;
  uint32_t f = ((uint32_t)e << 23) | (uint32_t)((mag >> 29) & 0x7fffffu);
  f = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : f);
  return __uint_as_float(f | (uint32_t)(u >> 32 & 0x80000000ull));
}

// Block sum of one float per thread, added to dst: compensated float pairs
// over the warp (TwoSum), warp totals carried into double.
__device__ __forceinline__ void block_sum_add_f(float x, double* dst) {
  float s = x, e = 0.0f;
  for (int o = 16; o > 0; o >>= 1) {
    const float os = __shfl_xor_sync(0xffffffffu, s, o);
    const float oe = __shfl_xor_sync(0xffffffffu, e, o);
    const float t = s + os;
    const float bp = t - s;
    e = (e + oe) + ((s - (t - bp)) + (os - bp));
    s = t;
  }
  __shared__ double ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) ws[wid] = gather_f2d(s) + gather_f2d(e);
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
    atomicAdd(dst, t);
  }
}

__device__ __forceinline__ void block_sum_add(double v, double* dst) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __shared__ double ws[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) ws[wid] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += ws[w];
    atomicAdd(dst, s);
  }
}

// One step of atom i: v += kick coef F ; x += dt v ; pack. F: from f on the
// first step of a call, gathered from the last force evaluation afterwards.
// All loads of an atom are issued before its stores.
// MG: the instance for the mixed path's gathered steps (gather set, float
// slots with compensated sums), KE its kinetic-energy row; with MG false both
// are decided at run time. The specialised instances carry fewer registers.
// snap (first step of a call, MG false; may be null): receives x, v and f as
// read (three n x 3 blocks), the state a rerun of the call starts from.
// Returned: the squared displacement since the build (d2) and the previous
// step's kinetic energy (kef on the mixed path, else ke).
template <bool MG>
__device__ __forceinline__ void step_atom(const PackArgs& pk, const GatherArgs& ga, int gather,
                                          double* __restrict__ x, double* __restrict__ v,
                                          const double* __restrict__ f, const Coef& cf, double dt,
                                          int kick, int do_pack, bool ke_row, double* __restrict__ snap,
                                          int i, float& d2, double& ke, float& kef) {
  const int t = pk.types[i];
  const size_t b = 3 * (size_t)i;
  const double x0 = x[b], x1 = x[b + 1], x2 = x[b + 2];
  const double v0 = v[b], v1 = v[b + 1], v2 = v[b + 2];
  double F0, F1, F2;
  float sc[6] = {0, 0, 0, 0, 0, 0};
  const bool mixed = MG || (gather && !ga.fp64 && !ga.atomic_mode);
  if (gather) {
    gather_force(ga, i, F0, F1, F2, mixed ? sc : nullptr);
  } else {
    F0 = f[b];
    F1 = f[b + 1];
    F2 = f[b + 2];
  }
  if (!MG && snap) {
    const size_t m = 3 * (size_t)pk.n;
    snap[b] = x0;
    snap[b + 1] = x1;
    snap[b + 2] = x2;
    snap[m + b] = v0;
    snap[m + b + 1] = v1;
    snap[m + b + 2] = v2;
    snap[2 * m + b] = F0;
    snap[2 * m + b + 1] = F1;
    snap[2 * m + b + 2] = F2;
  }
  const double cu = cf.c[t];
  const double kcu = kick == 2 ? cf.c2[t] : cu;
  double vn0, vn1, vn2;
  if (mixed) {
    // the velocity increment from the float force pair in float (the forces
    // are float-accurate), accumulated into the double velocity; F0..2 hold
    // the (rare) fallback-buffer forces, whose share of the increment is
    // also formed in float (no FP64 operation on the common path)
    const float kf = kick == 2 ? cf.c2f[t] : cf.cf[t];
    float d0 = kf * sc[0] + kf * sc[3];
    float d1 = kf * sc[1] + kf * sc[4];
    float d2v = kf * sc[2] + kf * sc[5];
    const bool extra = ga.flags[FLAG_EXTRA] | ga.flags[FLAG_EXTRA_STICKY];
    if (ke_row) {
      // the previous step's full velocity in float (the kinetic energy is a
      // thermo output; it does not feed the dynamics)
      const float hf = cf.cf[t];
      float w0 = d2f_bits(v0) + (hf * sc[0] + hf * sc[3]);
      float w1 = d2f_bits(v1) + (hf * sc[1] + hf * sc[4]);
      float w2 = d2f_bits(v2) + (hf * sc[2] + hf * sc[5]);
      if (extra) {  // forces scattered through the fallback buffer
        w0 = fmaf(hf, d2f_bits(F0), w0);
        w1 = fmaf(hf, d2f_bits(F1), w1);
        w2 = fmaf(hf, d2f_bits(F2), w2);
      }
      kef = cf.hmf[t] * fmaf(w0, w0, fmaf(w1, w1, w2 * w2));
    }
    if (extra) {
      d0 = fmaf(kf, d2f_bits(F0), d0);
      d1 = fmaf(kf, d2f_bits(F1), d1);
      d2v = fmaf(kf, d2f_bits(F2), d2v);
    }
    vn0 = v0 + gather_f2d(d0);
    vn1 = v1 + gather_f2d(d1);
    vn2 = v2 + gather_f2d(d2v);
  } else {
    if (ke_row) {
      // full-step velocity of the previous step
      const double w0 = fma(cu, F0, v0), w1 = fma(cu, F1, v1), w2 = fma(cu, F2, v2);
      ke = 0.5 * cf.m[t] * fma(w0, w0, fma(w1, w1, w2 * w2));
    }
    vn0 = fma(kcu, F0, v0);
    vn1 = fma(kcu, F1, v1);
    vn2 = fma(kcu, F2, v2);
  }
  const double xn0 = fma(dt, vn0, x0), xn1 = fma(dt, vn1, x1), xn2 = fma(dt, vn2, x2);
  v[b] = vn0;
  v[b + 1] = vn1;
  v[b + 2] = vn2;
  x[b] = xn0;
  x[b + 1] = xn1;
  x[b + 2] = xn2;
  if (do_pack) d2 = pack_one<!MG>(pk, i, t, xn0, xn1, xn2);
}

inline PackArgs make_pack(Ctx* c, bool track, bool build = false) {
  PackArgs a;
  a.n = c->n;
  a.qorg = c->d_qorg;
  a.qref = c->d_qref;
  a.types = c->d_types;
  a.fp64 = c->precision == TERSOFF_FP64;
  a.track = track ? 1 : 0;
  a.build = build ? 1 : 0;
  a.scale = ldexp(1.0, c->grid.fix_shift);
  a.inv_scale = ldexpf(1.0f, -c->grid.fix_shift);
  a.pos32 = c->d_pos32;
  a.posq = c->d_posq;
  a.pos64 = c->d_pos64;
  a.fix64 = c->grid.fix64;
  a.box = c->box64;
  a.sys = c->n_sys > 0 ? c->d_sys : nullptr;
  a.atom_sys = c->d_atom_sys;
  a.flags = c->d_flags;
  return a;
}

}  // namespace tgb
