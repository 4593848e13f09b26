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
__device__ __forceinline__ ipos4 make_pos64(double x, double y, double z, int t, int q, const Box64& b) {
  return ipos4{wrap64(x, q, b.L[0], b.invL[0], b.invLf[0]), wrap64(y, q, b.L[1], b.invL[1], b.invLf[1]),
               wrap64(z, q, b.L[2], b.invL[2], b.invLf[2]), t};
}
// difference of two wrapped coordinates, as the minimum image (edges are at
// least twice the list radius, so an entry's image is the nearest one)
__device__ __forceinline__ long long nearest(long long d, long long L) {
  const long long half = L >> 1;
  d -= d > half ? L : 0;
  d += d < -half ? L : 0;
  return d;
}

}  // namespace tgb
