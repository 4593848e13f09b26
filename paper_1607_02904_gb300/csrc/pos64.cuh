// Fixed-point positions of the FP64 path (ipos4).
#pragma once
#include "fxmath.cuh"
#include "internal.cuh"

namespace tgb {

// x 2^q as an integer, rounded, modulo 2^64 (integer operations: conversions
// run on the FP64 pipe)
__device__ __forceinline__ long long to_fixed(double x, int q) {
  const fx::Mant a = fx::unpack(x);
  const int s = a.e + q - 63;
  const unsigned long long v =
      s >= 0 ? (s < 64 ? a.m << s : 0ull) : (s > -64 ? ((a.m >> (-s - 1)) + 1) >> 1 : 0ull);
  return (long long)(__double_as_longlong(x) < 0 ? 0ull - v : v);
}

// x in float, cut off, by its bits
__device__ __forceinline__ float cut_to_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  const uint32_t m = e <= 0 ? 0u : (e >= 255 ? 0x7f800000u : (((uint32_t)e << 23) | (uint32_t)((b >> 29) & 0x7fffffu)));
  return __uint_as_float(m | (uint32_t)(b >> 32 & 0x80000000ull));
}

// coordinate x in fixed point, moved by whole box edges L (1 / L = invL) into
// [0, L) up to a few units of rounding
__device__ __forceinline__ long long wrap64(double x, int q, long long L, double invL, float invLf) {
  const float u = cut_to_float(x) * invLf;
  // beyond 2^20 boxes the float count of edges is off by more than the one
  // step that the comparisons below mend
  const long long k = fabsf(u) < 1048576.0f ? (long long)(int)floorf(u) : (long long)floor(x * invL);
  long long X = to_fixed(x, q) - k * L;
  X += X < 0 ? L : 0;
  X -= X >= L ? L : 0;
  return X;
}
__device__ __forceinline__ bool not_finite(double x) {
  return ((unsigned)__double2hiint(x) & 0x7ff00000u) == 0x7ff00000u;
}
__device__ __forceinline__ long long word64(double x, double y, double z, int t) {
  return t | (not_finite(x) || not_finite(y) || not_finite(z) ? POS64_BAD : 0ll);
}
__device__ __forceinline__ ipos4 make_pos64(double x, double y, double z, int t, int q, const Box64& b) {
  return ipos4{wrap64(x, q, b.L[0], b.invL[0], b.invLf[0]), wrap64(y, q, b.L[1], b.invL[1], b.invLf[1]),
               wrap64(z, q, b.L[2], b.invL[2], b.invLf[2]), word64(x, y, z, t)};
}
// axis a of a box with a long edge: where that one is long, the coordinate modulo
// 2^64, its coarse word to w
__device__ __forceinline__ long long wrap_long(double x, int q, const Box64& b, int a, long long& w) {
  if (b.Lc[a] < LONG64_EDGE) return wrap64(x, q, b.L[a], b.invL[a], b.invLf[a]);
  const double k = floor(x * b.invL[a]);
  const int c = (int)floor(ldexp(fma(-k, b.edge[a], x), q - LONG64_UNIT));
  w |= (long long)min(max(c, 0), 1023) << (32 + 10 * a);
  return (long long)((unsigned long long)to_fixed(x, q) - (unsigned long long)(long long)k * (unsigned long long)b.L[a]);
}
// difference of two wrapped coordinates, as the minimum image (edges are at
// least twice the list radius, so an entry's image is the nearest one)
__device__ __forceinline__ long long nearest(long long d, long long L) {
  const long long half = L >> 1;
  d -= d > half ? L : 0;
  d += d < -half ? L : 0;
  return d;
}
// the same on an axis of Lc units (out of line: inside the FP64 adjoint it cost 26
// registers): the coarse words hi and hj (at bit s) tell the image and whether the
// atoms are far apart (beyond any cutoff, which is below 4 units); the difference
// modulo 2^64 is the rest
static __device__ __noinline__ long long nearest_long(long long d, long long L, int Lc, int hi, int hj, int s) {
  if (Lc < LONG64_EDGE) return nearest(d, L);
  int dc = ((hj >> s) & 1023) - ((hi >> s) & 1023);
  const int k = dc > (Lc >> 1) ? 1 : (dc < -(Lc >> 1) ? -1 : 0);
  dc -= k * Lc;
  if (dc > 8 || dc < -8) return dc > 0 ? (1ll << 61) : -(1ll << 61);
  return (long long)((unsigned long long)d - (unsigned long long)(long long)k * (unsigned long long)L);
}

}  // namespace tgb
