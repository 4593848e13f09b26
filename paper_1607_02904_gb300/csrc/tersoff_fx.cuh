// The FP64 path's terms in 64-bit integer arithmetic (tersoff_lanes64.cuh).
//
// Bound: one FP64 warp instruction occupies its SM quarter's pipe for 64
// cycles, an integer one for 1 to 2. So bond vectors, lengths, unit vectors,
// angles, the angular function, exponentials, logarithms and the bond order
// are formed in fixed point and mantissa-exponent pairs (fxmath.cuh, 57 bits
// and more), and doubles carry only the sums of Eq. 5-7: the zeta sums, the
// radial derivative and the force accumulation, 166 to 200 FP64 instructions
// per atom with four bonds where the FP64 formulas take 1,012.
#pragma once
#include "fxmath.cuh"
#include "internal.cuh"

namespace tgb {
namespace fx {

// high 64 bits of a signed product (to 3 units)
TGB_FX int64_t smulhi(int64_t a, int64_t b) {
  const uint64_t p = mulhi((uint64_t)a, (uint64_t)b);
  return (int64_t)(p - ((uint64_t)(a >> 63) & (uint64_t)b) - ((uint64_t)(b >> 63) & (uint64_t)a));
}
// pack for exponents known to lie in the normal range
TGB_FX double pack_in(Mant a) {
  return from_bits(((uint64_t)(uint32_t)(a.e + 1022) << 52) + (((a.m >> 10) + 1) >> 1));
}

struct Bond64 {
  int64_t ux, uy, uz;  // unit vector, 62 fraction bits
  Mant r, ri;          // length and its reciprocal
};
// from the bond vector with q fraction bits (not 0, components below 2^62). Its
// largest component is moved up to bit 62 first, so that the squares keep 60 bits
// at any length.
TGB_FX Bond64 bond64(int64_t dx, int64_t dy, int64_t dz, int q) {
  uint64_t ax = (uint64_t)(dx < 0 ? -dx : dx), ay = (uint64_t)(dy < 0 ? -dy : dy), az = (uint64_t)(dz < 0 ? -dz : dz);
  const int up = clz64(ax | ay | az | 1ull) - 1;
  ax <<= up;
  ay <<= up;
  az <<= up;
  const int qd = q + up;
  const uint64_t s = (mulhi(ax, ax) + mulhi(ay, ay) + mulhi(az, az)) | 1ull;  // 2 qd - 64 fraction bits
  const int z = clz64(s);
  Bond64 b;
  const Mant r2{s << z, 127 - z - 2 * qd};
  b.ri = rsqrt(r2);
  b.r = mul(r2, b.ri);
  const int sh = 63 - qd + b.ri.e;
  const int64_t wx = (int64_t)shift(mulhi(ax, b.ri.m), sh), wy = (int64_t)shift(mulhi(ay, b.ri.m), sh),
                wz = (int64_t)shift(mulhi(az, b.ri.m), sh);
  b.ux = dx < 0 ? -wx : wx;
  b.uy = dy < 0 ? -wy : wy;
  b.uz = dz < 0 ? -wz : wz;
  return b;
}

// g(theta) = gamma + (gamma c^2/d^2) t^2 q and dg/dcos = -2 gamma c^2 t q^2,
// t = h - cos, q = 1/(d^2 + t^2), for cos with 60 fraction bits
TGB_FX void angle64(const FxRec& p, int64_t cs, double& g, double& dg) {
  const int64_t t = p.h - cs;
  const uint64_t at = (uint64_t)(t < 0 ? -t : t) | (t == 0 ? 1ull : 0ull);
  const int z = clz64(at);
  const Mant tm{at << z, 3 - z};
  const Mant t2 = mul(tm, tm);
  const uint64_t den = p.d2 + shift(t2.m, t2.e + 1 - p.qden);  // 64 - qden fraction bits
  const int zd = clz64(den);
  const Mant q = rcp(Mant{den << zd, p.qden - 1 - zd});
  const Mant tq = mul(tm, q);
  g = p.gamma + pack_in(mul(mul(tq, tm), Mant{p.gc2d2, p.gc2d2_e}));
  const double d = pack_in(mul(mul(tq, q), Mant{p.g2c2, p.g2c2_e}));
  dg = from_bits(bits_of(d) | (~(uint64_t)t & 0x8000000000000000ull));
}

// Pair term of a bond of length r inside the cutoff: f_R, b f_A and
// -(1/2) f_A db/dzeta (each without f_C); false when zeta or a power of it is
// outside the formats.
TGB_FX bool pair64(const FxRec& p, uint64_t rm, int re, double zeta, double* fr, double* bfa, double* dz) {
  const int ez = exponent(zeta);
  if (!((int64_t)bits_of(zeta) > 0 && ez >= -30 && ez <= 29)) return false;
  const int64_t lz = log2_fixed(unpack(zeta));
  const int64_t lbz = lz + p.lgbeta;
  int64_t au, lb;
  if (!times((uint64_t)(lbz < 0 ? -lbz : lbz), Mant{p.n, p.n_e}, 30, au)) return false;  // |n log2(beta zeta)|
  const int64_t zu = lbz < 0 ? -au : au;
  const Mant u = exp2_fixed(zu);
  const uint64_t one = 1ull << 62;
  const uint64_t s = u.e >= 0 ? (u.m >> 1) + (one >> u.e) : one + shift(u.m >> 1, u.e);  // 1 + u
  const int c = (int)(s >> 63);
  const int64_t l1u = log2_fixed(Mant{c ? s : s << 1, (u.e > 0 ? u.e : 0) + c});
  if (!times((uint64_t)l1u, Mant{p.in2, p.in2_e}, 16, lb)) return false;  // log2(1 + u)/(2n)
  const int64_t z1 = (int64_t)shift(mulhi(rm, p.l1), re + p.l1_e - 5);
  const int64_t z2 = (int64_t)shift(mulhi(rm, p.l2), re + p.l2_e - 5);
  const Mant ba = exp2_fixed(p.lgB - z2 - lb);
  *fr = pack_in(exp2_fixed(p.lgA - z1));
  *bfa = -pack_in(ba);
  // (1/4) b |f_A| u / ((1 + u) zeta)
  *dz = pack_in(mul(ba, exp2_fixed(zu - l1u - lz - (2ll << 57))));
  return true;
}

}  // namespace fx
}  // namespace tgb
