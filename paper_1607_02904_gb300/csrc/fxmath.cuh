// Double-precision elementary functions in 64-bit integer arithmetic.
//
// GB300's FP64 pipe takes one warp instruction per 64 cycles and SM quarter
// (1.25 TFLOP/s on the chip, 1/62 of the FP32 rate), where the integer pipes
// take one per 1 to 2 cycles. An exponential of some 16 FP64 operations costs
// a warp 1,000 cycles there; the same function in fixed point, with 64-bit
// products from four 32-bit multiplies each, issues about 80 integer
// instructions and carries 60 or more bits where a double has 53.
//
// Values between the functions are a mantissa and an exponent (Mant: m in
// [2^63, 2^64) stands for m 2^(e - 63)) or signed fixed point with 57 fraction
// bits (base-2 logarithms, |value| < 64). The exponential and the logarithm
// use tables over 64 intervals and short polynomials inside one (Tang, ACM
// TOMS 15 (1989) 144 and 16 (1990) 378, in base 2 and fixed point); the
// reciprocal and the reciprocal square root refine the hardware's float
// approximation by one step of second order. Every function's relative error
// is below 2^-56 before its one rounding to double (the fixed-point logarithm's
// absolute error below 2^-55); the reciprocal and the square root of doubles are
// rounded correctly, as the operations that they stand for. Arguments outside a
// function's range (zero, subnormal, infinite, NaN, or too large for the
// fixed-point formats) take the CUDA functions or the FP64 formulas.
//
// Measured on GB300 against the CUDA functions: ten FP64 MD steps of 512,000 Si
// atoms 11.1 -> 5.7 ms, one evaluation of 4,096 atoms 65 -> 52 us, a fitting
// iteration of 24 cells with lambda3 4.27 -> 3.81 ms; errors as before.
//
// Compiles for the host too (without the fallbacks' CUDA intrinsics), where
// the arithmetic is checked against many digits.
#pragma once
#include <math.h>

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define TGB_FX __device__ __forceinline__
#define TGB_FX_CALL static __device__ __noinline__
#define TGB_FX_TABLE static __device__ const
#else
#define TGB_FX inline
#define TGB_FX_CALL inline
#define TGB_FX_TABLE static const
#endif

namespace tgb {
namespace fx {

// 2^(i/64) with 63 fraction bits
TGB_FX_TABLE uint64_t kExp2[64] = {
    0x8000000000000000ull, 0x8164d1f3bc030773ull, 0x82cd8698ac2ba1d7ull, 0x843a28c3acde4046ull,
    0x85aac367cc487b15ull, 0x871f61969e8d1010ull, 0x88980e8092da8527ull, 0x8a14d575496efd9aull,
    0x8b95c1e3ea8bd6e7ull, 0x8d1adf5b7e5ba9e6ull, 0x8ea4398b45cd53c0ull, 0x9031dc431466b1dcull,
    0x91c3d373ab11c336ull, 0x935a2b2f13e6e92cull, 0x94f4efa8fef70961ull, 0x96942d3720185a00ull,
    0x9837f0518db8a96full, 0x99e0459320b7fa65ull, 0x9b8d39b9d54e5539ull, 0x9d3ed9a72cffb751ull,
    0x9ef5326091a111aeull, 0xa0b0510fb9714fc2ull, 0xa27043030c496819ull, 0xa43515ae09e6809eull,
    0xa5fed6a9b15138eaull, 0xa7cd93b4e965356aull, 0xa9a15ab4ea7c0ef8ull, 0xab7a39b5a93ed337ull,
    0xad583eea42a14ac6ull, 0xaf3b78ad690a4375ull, 0xb123f581d2ac2590ull, 0xb311c412a9112489ull,
    0xb504f333f9de6484ull, 0xb6fd91e328d17791ull, 0xb8fbaf4762fb9ee9ull, 0xbaff5ab2133e45fbull,
    0xbd08a39f580c36bfull, 0xbf1799b67a731083ull, 0xc12c4cca66709456ull, 0xc346ccda24976407ull,
    0xc5672a115506daddull, 0xc78d74c8abb9b15dull, 0xc9b9bd866e2f27a3ull, 0xcbec14fef2727c5dull,
    0xce248c151f8480e4ull, 0xd06333daef2b2595ull, 0xd2a81d91f12ae45aull, 0xd4f35aabcfedfa1full,
    0xd744fccad69d6af4ull, 0xd99d15c278afd7b6ull, 0xdbfbb797daf23755ull, 0xde60f4825e0e9124ull,
    0xe0ccdeec2a94e111ull, 0xe33f8972be8a5a51ull, 0xe5b906e77c8348a8ull, 0xe8396a503c4bdc68ull,
    0xeac0c6e7dd24392full, 0xed4f301ed9942b84ull, 0xefe4b99bdcdaf5cbull, 0xf281773c59ffb13aull,
    0xf5257d152486cc2cull, 0xf7d0df730ad13bb9ull, 0xfa83b2db722a033aull, 0xfd3e0c0cf486c175ull,
};

// per i: c 2^53 with c the smallest integer >= 1024 / (1 + i/64), and
// -log2(c / 1024) with 57 fraction bits; load_log takes a pair by one 16-byte
// load, which its address has to be a multiple of
alignas(16) TGB_FX_TABLE uint64_t kLog2[128] = {
    0x8000000000000000ull, 0x0000000000000000ull, 0x7e20000000000000ull, 0x000ae67673c5254full,
    0x7c20000000000000ull, 0x0016b50e297afcceull, 0x7a60000000000000ull, 0x0021320bef2e08f8ull,
    0x7880000000000000ull, 0x002c99c4d80ce2adull, 0x76c0000000000000ull, 0x003768205f24a728ull,
    0x7520000000000000ull, 0x004195a2fe15dacdull, 0x7380000000000000ull, 0x004be78cb56ff742ull,
    0x71e0000000000000ull, 0x00565ee59de27448ull, 0x7040000000000000ull, 0x0060fcc133716a9bull,
    0x6ec0000000000000ull, 0x006aecb2a7b1d1caull, 0x6d40000000000000ull, 0x0074ff550e92b572ull,
    0x6be0000000000000ull, 0x007e5a5fcef4333dull, 0x6a80000000000000ull, 0x0087d42402259a88ull,
    0x6920000000000000ull, 0x00916d6e1559a4b7ull, 0x67c0000000000000ull, 0x009b271288e64106ull,
    0x6680000000000000ull, 0x00a41b2f34aebcb5ull, 0x6540000000000000ull, 0x00ad2b6bd1b86f6bull,
    0x6400000000000000ull, 0x00b6587b432e4750ull, 0x62c0000000000000ull, 0x00bfa3172c70b441ull,
    0x61a0000000000000ull, 0x00c819b97485f720ull, 0x6080000000000000ull, 0x00d0a978a14c0d9full,
    0x5f60000000000000ull, 0x00d952eb7a8ffc16ull, 0x5e40000000000000ull, 0x00e216ae2634459eull,
    0x5d20000000000000ull, 0x00eaf5626a31ebefull, 0x5c20000000000000ull, 0x00f2eeefbf237053ull,
    0x5b20000000000000ull, 0x00fafec54831f1a5ull, 0x5a20000000000000ull, 0x01032560e91e59deull,
    0x5920000000000000ull, 0x010b6344bc75ae70ull, 0x5820000000000000ull, 0x0113b8f7444275bbull,
    0x5740000000000000ull, 0x011b17e849adc261ull, 0x5640000000000000ull, 0x01239bb9203bcc33ull,
    0x5560000000000000ull, 0x012b23e51b39c7b0ull, 0x5480000000000000ull, 0x0132bfee370ee686ull,
    0x53a0000000000000ull, 0x013a703e50fa4df3ull, 0x52c0000000000000ull, 0x014235429d72a9ddull,
    0x5200000000000000ull, 0x0148eef19317990dull, 0x5120000000000000ull, 0x0150db96d04eaa35ull,
    0x5060000000000000ull, 0x0157b7eb8038faf3ull, 0x4fa0000000000000ull, 0x015ea4b771855cd6ull,
    0x4ee0000000000000ull, 0x0165a24a6d5cef3dull, 0x4e20000000000000ull, 0x016cb0f6865c8ea0ull,
    0x4d60000000000000ull, 0x0173d1102f2c0982ull, 0x4ca0000000000000ull, 0x017b02ee522efefeull,
    0x4be0000000000000ull, 0x018246ea6a6006abull, 0x4b40000000000000ull, 0x01886300713adfc4ull,
    0x4a80000000000000ull, 0x018fc924c89ac847ull, 0x49e0000000000000ull, 0x019602381211518aull,
    0x4940000000000000ull, 0x019c48d45f2b5251ull, 0x4880000000000000ull, 0x01a3e2f4ac43f603ull,
    0x47e0000000000000ull, 0x01aa482b35ca9cebull, 0x4740000000000000ull, 0x01b0bbae4995d670ull,
    0x46a0000000000000ull, 0x01b73dbe68b5a1bbull, 0x4620000000000000ull, 0x01bc7d3e94dedc4cull,
    0x4580000000000000ull, 0x01c31a27dd00b49cull, 0x44e0000000000000ull, 0x01c9c65c26a33233ull,
    0x4460000000000000ull, 0x01cf281f15f0be72ull, 0x43c0000000000000ull, 0x01d5f08f93f98892ull,
    0x4340000000000000ull, 0x01db694903d94b87ull, 0x42a0000000000000ull, 0x01e24ee8ae9f0c50ull,
    0x4220000000000000ull, 0x01e7df5fe538ab35ull, 0x41a0000000000000ull, 0x01ed7aa6fa358f0aull,
    0x4120000000000000ull, 0x01f320e8445b299full, 0x40a0000000000000ull, 0x01f8d24f150baeaaull,
};

struct Mant {
  uint64_t m;
  int e;
};

// ---------------------------------------------------------------- bits
#ifdef __CUDACC__
TGB_FX uint64_t bits_of(double x) { return (uint64_t)__double_as_longlong(x); }
TGB_FX double from_bits(uint64_t b) { return __longlong_as_double((long long)b); }
TGB_FX float f_of(uint32_t b) { return __uint_as_float(b); }
TGB_FX uint32_t u_of(float f) { return __float_as_uint(f); }
TGB_FX int clz64(uint64_t v) { return __clzll((long long)v); }
TGB_FX uint64_t ldt(const uint64_t* p) { return __ldg((const unsigned long long*)p); }
TGB_FX float rcp_f(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
TGB_FX float rsqrt_f(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
TGB_FX void load_log(int i, uint64_t& c, uint64_t& l) {
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(kLog2) + i);
  c = v.x;
  l = v.y;
}
#else
inline uint64_t bits_of(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
inline double from_bits(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
inline float f_of(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
inline uint32_t u_of(float f) { uint32_t b; std::memcpy(&b, &f, 4); return b; }
inline int clz64(uint64_t v) { return v ? __builtin_clzll(v) : 64; }
inline uint64_t ldt(const uint64_t* p) { return *p; }
inline float& host_jitter() { static float j = 0.0f; return j; }  // relative error put on the approximations
inline float rcp_f(float x) { return (1.0f / x) * (1.0f + host_jitter()); }
inline float rsqrt_f(float x) { return (1.0f / sqrtf(x)) * (1.0f + host_jitter()); }
inline void load_log(int i, uint64_t& c, uint64_t& l) { c = kLog2[2 * i]; l = kLog2[2 * i + 1]; }
#endif

// high 32 bits of a 32 x 32 product
TGB_FX uint32_t mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
// high 64 bits of a 64 x 64 product, without the low x low part: at most 3 too
// small
TGB_FX uint64_t mulhi(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
  const uint32_t bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (uint64_t)ah * bh + mulhi32(ah, bl) + mulhi32(al, bh);
}
// a * b for 32-bit a, without the 32 lowest bits
TGB_FX uint64_t mul32(uint32_t a, uint64_t b) {
  return (uint64_t)a * (uint32_t)(b >> 32) + mulhi32(a, (uint32_t)b);
}
// the same for signed b
TGB_FX int64_t mul32s(uint32_t a, int64_t b) {
  return (int64_t)((uint64_t)((int64_t)(int32_t)(b >> 32) * (int64_t)a)) + mulhi32(a, (uint32_t)b);
}
// v 2^s for -127 <= s <= 63 (shifts out to 0)
TGB_FX uint64_t shift(uint64_t v, int s) { return s >= 0 ? v << s : (s > -64 ? v >> -s : 0ull); }

// positive normal doubles (any sign bit is ignored)
TGB_FX int exponent(double x) { return (int)((bits_of(x) >> 52) & 0x7ff) - 1023; }
TGB_FX bool normal(double x) {
  const uint32_t e = (uint32_t)(bits_of(x) >> 52) & 0x7ff;
  return e - 1u < 0x7feu;
}
TGB_FX Mant unpack(double x) {
  const uint64_t b = bits_of(x);
  return Mant{(b << 11) | 0x8000000000000000ull, (int)((b >> 52) & 0x7ff) - 1023};
}
// rounded to nearest; below the normal range 0, above it infinity
TGB_FX double pack(Mant a) {
  const uint64_t r = ((a.m >> 10) + 1) >> 1;  // 53 bits, 2^53 after a carry
  const uint64_t b = ((uint64_t)(uint32_t)(a.e + 1022) << 52) + r;
  return a.e < -1022 ? 0.0 : from_bits(a.e > 1023 || b > 0x7ff0000000000000ull ? 0x7ff0000000000000ull : b);
}
TGB_FX double nan64() { return from_bits(0x7ff8000000000000ull); }
// v 2^-q, rounded to nearest (|v| > 0 or 0)
TGB_FX double from_fixed(int64_t v, int q) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = clz64(a);
  if (a == 0) return 0.0;
  const uint64_t b = bits_of(pack(Mant{a << z, 63 - z - q}));
  return from_bits(b | ((uint64_t)v & 0x8000000000000000ull));
}
TGB_FX Mant mul(Mant a, Mant b) {
  const uint64_t p = mulhi(a.m, b.m);  // in [2^62, 2^64)
  const int c = (int)(p >> 63);
  return Mant{c ? p : p << 1, a.e + b.e + c};
}

// ---------------------------------------------------------------- functions
// 2^z, z with 57 fraction bits
TGB_FX Mant exp2_fixed(int64_t z) {
  const int n = (int)(z >> 57);
  const uint64_t T = ldt(&kExp2[(int)(z >> 51) & 63]);
  const uint64_t R = ((uint64_t)z & ((1ull << 51) - 1)) << 13;  // r = R 2^-70 < 2^-6
  const uint32_t R32 = (uint32_t)(R >> 32);
  // 2^r - 1 = r (c1 + r (c2 + ...)), c_k = ln(2)^k / k!; from the fourth
  // coefficient on 32 bits carry enough
  uint32_t q = 0x15d87fe8u + (mulhi32(R32, 0x02861226u + (mulhi32(R32, 0x003ff980u) >> 6)) >> 6);
  q = 0x9d955b7eu + (mulhi32(R32, q) >> 6);                              // c4 + ..., 38 fraction bits
  const uint64_t q3 = 0x0e35846b82505fc6ull + (((uint64_t)R32 * q) >> 12);  // 64 fraction bits
  const uint64_t q2 = 0x3d7f7bff058b1d51ull + (mulhi(R, q3) >> 6);
  const uint64_t q1 = 0xb17217f7d1cf79acull + (mulhi(R, q2) >> 6);
  const uint64_t p = mulhi(R, q1) >> 6;
  return Mant{T + mulhi(T, p), n};
}
// log2 of a value with |exponent| <= 62, 57 fraction bits
TGB_FX int64_t log2_fixed(Mant a) {
  uint64_t c, l;
  load_log((int)(a.m >> 57) & 63, c, l);
  const uint64_t t = mul32((uint32_t)(c >> 32), a.m) - (1ull << 62);  // m c - 1 in [0, 2^-5.9), 62 bits
  const uint64_t R = (int64_t)t < 0 ? 0ull : t << 7;                  // t = R 2^-69
  const uint32_t R32 = (uint32_t)(R >> 32);
  // log2(1 + t) = t (k1 - t (k2 - t (k3 - ...))), k_j = log2(e) / j
  uint32_t q = 0x17154765u - (mulhi32(R32, 0x1484b13du) >> 5);
  q = 0x1a61762au - (mulhi32(R32, q) >> 5);
  q = 0x1ec709dcu - (mulhi32(R32, q) >> 5);
  q = 0x24eed8a2u - (mulhi32(R32, q) >> 5);                                // k5 - ..., 31 fraction bits
  const uint64_t q4 = 0x2e2a8eca5705fc2full - (((uint64_t)R32 * q) >> 5);  // 63 fraction bits
  const uint64_t q3 = 0x3d8e13b87407fae9ull - (mulhi(R, q4) >> 5);
  const uint64_t q2 = 0x5c551d94ae0bf85eull - (mulhi(R, q3) >> 5);
  const uint64_t q1 = 0xb8aa3b295c17f0bcull - (mulhi(R, q2) >> 5);
  const uint64_t p = mulhi(R, q1) >> 11;
  return (int64_t)((uint64_t)(int64_t)a.e << 57) + (int64_t)l + (int64_t)p;
}

// y0 (1 + E), y0 with 31 and E with 62 fraction bits: 63 bits. |E| < 2^-20, where
// E shifted by 21 still fits its word: the approximations are good to 2^-23 (what
// the PTX instructions state) and see their argument cut to 24 bits, 2^-22
// together. The terms of third order left out are below 2^-60.
TGB_FX uint64_t refine(uint32_t y0, int64_t E) {
  return ((uint64_t)y0 << 32) + (uint64_t)(mul32s(y0, (int64_t)((uint64_t)E << 21)) >> 19);
}
TGB_FX float inside(float y) { return fminf(fmaxf(y, 0.5f), 0.99999994f); }
// 1 / a
TGB_FX Mant rcp(Mant a) {
  // a float approximation of 1/m, m in [1, 2), inside [1/2, 1), as 31-bit fixed point
  const float y = inside(rcp_f(f_of(0x3f800000u | (uint32_t)((a.m >> 40) & 0x7fffffu))));
  const uint32_t y0 = ((u_of(y) & 0x7fffffu) | 0x800000u) << 7;
  const int64_t e = (int64_t)((1ull << 62) - mul32(y0, a.m));  // 1 - m y0
  const int32_t eh = (int32_t)(e >> 20);
  const uint64_t r = refine(y0, e + (((int64_t)eh * eh) >> 22));
  return Mant{(r >> 63) ? ~0ull : r << 1, -a.e - 1};
}
// 1 / sqrt(a)
TGB_FX Mant rsqrt(Mant a) {
  const int odd = a.e & 1;
  const uint64_t w = odd ? a.m : a.m >> 1;  // in [1, 4), 62 bits
  const float y = inside(rsqrt_f(f_of((odd ? 0x40000000u : 0x3f800000u) | (uint32_t)((a.m >> 40) & 0x7fffffu))));
  const uint32_t y0 = ((u_of(y) & 0x7fffffu) | 0x800000u) << 7;
  const uint64_t s = (uint64_t)y0 * y0;                     // exact, 62 bits
  const int64_t e = (int64_t)((1ull << 60) - mulhi(w, s));  // 1 - w y0^2, 60 bits
  const int32_t eh = (int32_t)(e >> 20);                    // 40 bits
  const uint64_t r = refine(y0, (e << 1) + (((int64_t)eh * eh * 3) >> 21));
  return Mant{(r >> 63) ? ~0ull : r << 1, -((a.e - odd) >> 1) - 1};
}

// ---------------------------------------------------------------- on doubles
// 1 / x, correctly rounded: the mantissas' quotient lies within 2^-6 of n or n + 1
// units, n its cut approximation, so that the sign of 2^106 - X (2 n + 1), X the
// mantissa of x as an integer, says which is nearer (its low 64 bits hold it; it
// is never 0)
TGB_FX_CALL double rcp(double x) {
  const Mant a = unpack(x);
  if (!normal(x) || a.e > 1021) return 1.0 / x;
  const Mant r = rcp(a);
  uint64_t n = r.m >> 11;
  n += (int64_t)((a.m >> 11) * (2 * n + 1)) < 0 ? 1 : 0;
  return from_bits((((uint64_t)(uint32_t)(r.e + 1022) << 52) + n) | (bits_of(x) & 0x8000000000000000ull));
}
TGB_FX_CALL double rsqrt(double x) {
  if (!(normal(x) && x > 0.0)) return 1.0 / ::sqrt(x);
  return pack(rsqrt(unpack(x)));
}
// sqrt(x), correctly rounded (in the same way: by the sign of 4 x - (2 n + 1)^2 in
// units of n squared)
TGB_FX_CALL double sqrt(double x) {
  if (!(normal(x) && x > 0.0)) return ::sqrt(x);
  const Mant a = unpack(x), s = mul(a, rsqrt(a));
  uint64_t n = s.m >> 11;
  n += (int64_t)(((a.m >> 11) << (54 + a.e - 2 * s.e)) - (2 * n + 1) * (2 * n + 1)) > 0 ? 1 : 0;
  return from_bits(((uint64_t)(uint32_t)(s.e + 1022) << 52) + n);
}
// x log2(e) with 57 fraction bits, |x| < 32
TGB_FX int64_t log2e_times(double x) {
  const Mant a = unpack(x);
  const uint64_t v = shift(mulhi(a.m, 0x5c551d94ae0bf85eull), a.e - 4);
  return (int64_t)bits_of(x) < 0 ? -(int64_t)v : (int64_t)v;
}
TGB_FX_CALL double exp(double x) {
  if (!(exponent(x) < 5)) return ::exp(x);
  if (exponent(x) < -60) return 1.0;
  return pack(exp2_fixed(log2e_times(x)));
}
TGB_FX_CALL double log(double x) {
  const int e = exponent(x);
  // between 1/2 and 2 the fixed point's absolute error is not a relative one
  if (!(x > 0.0 && e >= -60 && e <= 60) || e == 0 || e == -1) return ::log(x);
  const int64_t v = log2_fixed(unpack(x));
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = clz64(a);
  if (a == 0) return 0.0;
  const double y = pack(mul(Mant{a << z, 6 - z}, Mant{0xb17217f7d1cf79acull, -1}));  // times ln 2
  return from_bits(bits_of(y) | ((uint64_t)v & 0x8000000000000000ull));
}
// sin(pi x) and cos(pi x) for 0 <= x <= 1/2
TGB_FX_CALL void sincospi(double x, double* s, double* c) {
  if (!(x <= 0.5) || exponent(x) < -30) {
#ifdef __CUDACC__
    ::sincospi(x, s, c);
#else
    *s = ::sin(M_PI * x);
    *c = ::cos(M_PI * x);
#endif
    return;
  }
  // f = x or 1/2 - x, at most 1/4: sin(pi f) = f S(f^2), cos(pi f) = C(f^2)
  const bool swap = x > 0.25;
  Mant f = unpack(x);
  if (swap) {
    const uint64_t d = (1ull << 63) - (f.m >> (-1 - f.e));  // 1/2 - x, 64 bits
    const uint64_t d1 = d ? d : 1ull;
    const int z = clz64(d1);
    f = Mant{d1 << z, -1 - z};
  }
  const uint64_t h = shift(f.m, f.e + 2);  // f with 65 fraction bits
  const uint64_t v = mulhi(h, h);          // f^2 with 66
  // alternating series, 61 fraction bits
  uint64_t S = 0x0000000c52021090ull;
  S = 0x000001aaec32af93ull - (mulhi(v, S) >> 2);
  S = 0x00002df5b73e2aafull - (mulhi(v, S) >> 2);
  S = 0x0003d1e869a031acull - (mulhi(v, S) >> 2);
  S = 0x003c60e9fbd10e3full - (mulhi(v, S) >> 2);
  S = 0x02a0f0690fdcf037ull - (mulhi(v, S) >> 2);
  S = 0x132d2cce62bd85beull - (mulhi(v, S) >> 2);
  S = 0x519af19dd6ab8749ull - (mulhi(v, S) >> 2);
  S = 0xa55de7312df295f5ull - (mulhi(v, S) >> 2);
  S = 0x6487ed5110b4611aull - (mulhi(v, S) >> 2);
  uint64_t C = 0x00000001ef6e308dull;
  C = 0x0000004a831646beull - (mulhi(v, C) >> 2);
  C = 0x000009063161796cull - (mulhi(v, C) >> 2);
  C = 0x0000db7127a25894ull - (mulhi(v, C) >> 2);
  C = 0x000fce9c51bb1e61ull - (mulhi(v, C) >> 2);
  C = 0x00d368f95102545dull - (mulhi(v, C) >> 2);
  C = 0x0787d41a246eaebdull - (mulhi(v, C) >> 2);
  C = 0x2aba78fc797ff3f9ull - (mulhi(v, C) >> 2);
  C = 0x81e0f840dad61d9bull - (mulhi(v, C) >> 2);
  C = 0x9de9e64df22ef2d2ull - (mulhi(v, C) >> 2);
  C = 0x2000000000000000ull - (mulhi(v, C) >> 2);
  const double sv = pack(mul(f, Mant{S << 1, 1}));
  const int z = clz64(C);
  const double cv = pack(Mant{C << z, 2 - z});
  *s = swap ? cv : sv;
  *c = swap ? sv : cv;
}
// v a for a logarithm's magnitude v (57 fraction bits) and -30 <= a.e <= 5; false
// from lim (at most 62) on, where the product would leave the format
TGB_FX bool times(uint64_t v, Mant a, int lim, int64_t& z) {
  const uint64_t p = mulhi(v, a.m);  // 56 - a.e fraction bits
  const int up = a.e + 1;
  const uint64_t q = up < 0 ? p >> -up : p;
  z = (int64_t)(q << (up > 0 ? up : 0));
  return q < ((uint64_t)lim << 57) >> (up > 0 ? up : 0);
}
// b = (1 + (beta zeta)^n)^(-1/(2n)) and db/dzeta = -b u / (2 (1 + u) zeta) with
// u = (beta zeta)^n, for zeta > 0; false when an argument is outside the
// formats (the caller then takes the FP64 formulas)
TGB_FX_CALL bool bond(double zeta, double beta, double n, double ninv2, double* b, double* db) {
  const double bz = beta * zeta;
  const int ebz = exponent(bz), en = exponent(n), ei = exponent(ninv2);
  if (!(bz > 0.0 && n > 0.0 && normal(zeta)) || ebz < -60 || ebz > 60 || en < -30 || en > 5 || ei < -30 || ei > 5)
    return false;
  const int64_t lg = log2_fixed(unpack(bz));
  int64_t zu, zw;
  if (!times((uint64_t)(lg < 0 ? -lg : lg), Mant{unpack(n).m, en}, 62, zu)) return false;
  const Mant u = exp2_fixed(lg < 0 ? -zu : zu);
  // 1 + u
  const uint64_t one = 1ull << 62;
  const uint64_t s = u.e >= 0 ? (u.m >> 1) + (one >> u.e) : one + shift(u.m >> 1, u.e);
  const int c = (int)(s >> 63);
  const Mant opu{c ? s : s << 1, (u.e > 0 ? u.e : 0) + c};
  if (!times((uint64_t)log2_fixed(opu), Mant{unpack(ninv2).m, ei}, 62, zw)) return false;
  const Mant bm = exp2_fixed(-zw);
  Mant d = mul(mul(bm, u), rcp(mul(opu, unpack(zeta))));
  d.e -= 1;
  *b = pack(bm);
  *db = -pack(d);
  return true;
}

}  // namespace fx
}  // namespace tgb
