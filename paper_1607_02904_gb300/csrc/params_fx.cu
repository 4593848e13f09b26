// Integer records of the FP64 path from the derived parameter records.
#include <cmath>

#include "internal.cuh"

namespace tgb {
namespace {

struct HostMant {
  unsigned long long m;
  int e;
};
// v > 0 in extended precision (at least 64 bits of mantissa where long double
// has them; a double's 53 are exact in either case)
HostMant mant(long double v) {
  int e;
  const long double f = frexpl(v, &e);  // [1/2, 1)
  return HostMant{(unsigned long long)ldexpl(f, 64), e - 1};
}
long long fixed57(long double v) { return llrintl(ldexpl(v, 57)); }

}  // namespace

// A table qualifies when every value fits its format with room for the sums
// that pair64 forms from them. Pair records (i,j,j): |log2| of A and B at most
// 24, of beta at most 30, lambda r log2(e) at most 20 inside the largest
// cutoff. Every record: |h| below 2, d^2 in [1/16, 2^40], gamma and c such
// that gamma c^2 and its quotient by d^2 are positive and normal.
void make_fx_records(Ctx* c) {
  c->h_fx.clear();
  const int ns = c->ns;
  const long double log2e = 1.0L / logl(2.0L);
  const double lim = 20.0 / (1.4427 * c->rmax_cut);
  bool ok = true;
  c->fx_cut_j = true;
  auto in = [&](double v, double lo, double hi) { ok = ok && v >= lo && v <= hi; };
  auto rec = [&](int i, int j, int k) { return &c->h_rec64[(size_t)((i * ns + j) * ns + k) * RSTRIDE]; };
  for (int i = 0; i < ns; ++i)
    for (int j = 0; j < ns; ++j)
      for (int k = 0; k < ns; ++k) {
        const double* o = rec(i, j, k);
        const double* p = rec(i, k, k);
        if (o[K_RIN3] != p[K_RIN3] || o[K_ROUT3] != p[K_ROUT3]) c->fx_cut_j = false;
        in(o[K_H], -2.0, 2.0);
        in(o[K_D2], 0.0625, std::ldexp(1.0, 40));
        in(o[K_GAMMA], std::ldexp(1.0, -60), std::ldexp(1.0, 60));
        in(o[K_GC2D2], std::ldexp(1.0, -60), std::ldexp(1.0, 100));
        in(o[K_G2C2], std::ldexp(1.0, -60), std::ldexp(1.0, 100));
        if (j == k) {
          in(o[K_A], std::ldexp(1.0, -24), std::ldexp(1.0, 24));
          in(o[K_B], std::ldexp(1.0, -24), std::ldexp(1.0, 24));
          in(o[K_BETA], std::ldexp(1.0, -30), std::ldexp(1.0, 30));
          in(o[K_LAM1], 0.01, lim);
          in(o[K_LAM2], 0.01, lim);
          in(o[K_N], 0.03, 30.0);
        }
        FxRec f{};
        if (ok) {
          const HostMant gc = mant(o[K_GC2D2]), g2 = mant(o[K_G2C2]);
          f.gamma = o[K_GAMMA];
          f.h = llrint(std::ldexp(o[K_H], 60));
          f.qden = (int)std::ceil(std::log2(o[K_D2] + 16.0));
          f.d2 = (unsigned long long)ldexpl((long double)o[K_D2], 64 - f.qden);
          f.gc2d2 = gc.m, f.gc2d2_e = gc.e;
          f.g2c2 = g2.m, f.g2c2_e = g2.e;
          if (j == k) {
            const HostMant l1 = mant(log2e * o[K_LAM1]), l2 = mant(log2e * o[K_LAM2]);
            const HostMant n = mant(o[K_N]), in2 = mant(0.5L / (long double)o[K_N]);
            f.hl1 = 0.5 * o[K_LAM1];
            f.hl2 = 0.5 * o[K_LAM2];
            f.l1 = l1.m, f.l1_e = l1.e;
            f.l2 = l2.m, f.l2_e = l2.e;
            f.n = n.m, f.n_e = n.e;
            f.in2 = in2.m, f.in2_e = in2.e;
            f.lgA = fixed57(log2e * logl((long double)o[K_A]));
            f.lgB = fixed57(log2e * logl((long double)o[K_B]));
            f.lgbeta = fixed57(log2e * logl((long double)o[K_BETA]));
          }
        }
        c->h_fx.push_back(f);
      }
  c->fx_ok = ok;
}

}  // namespace tgb
