// Parameter adjoint of the FP64 path: eight lanes per centre atom, one bond j
// per lane (tersoff_bwd.cu states the adjoint).
//
// Bound: the FP64 pipe (64 cycles per warp instruction), and before it
// parallelism. A thread per atom walked all z (z - 1) ordered triplets twice,
// so that a few thousand atoms left most of the chip idle, and added every
// field of every triplet to shared doubles that 32 lanes hit at once. Here the
// atom's bonds are formed once by the group, with their cutoff function and
// its derivatives (once per bond instead of twice per triplet, when f_C(r_ik)
// does not depend on j); each lane runs its own j's two K loops, keeps the sums
// of its (ti, tj) records in registers, and adds them once per bond to its own
// column of shared memory. The table constants that multiply a whole sum (c,
// d, gamma) are applied there, not per triplet. Blocks loop over the atoms, so
// the columns are summed over a block once.
// Measured: a fitting iteration of 24 cells (some 13,000 atoms, lambda3 on)
// 3.48 -> 1.69 ms, of which the adjoint had been 2.1 ms; SiC, 4,096 atoms,
// 2,462 -> 175 us, 512,000 atoms 11.1 -> 6.6 ms. (A large crystal of one species
// keeps a thread per atom: BWD64_ONE_MAX.)
#pragma once

namespace tgb {
namespace bwd {

constexpr int L64_BLOCK = 64;
constexpr int L64_W = 8;           // lanes per atom
constexpr int L64_SLOTS = 16;      // bonds kept per atom; longer lists form them in each loop
constexpr int L64_WORDS = 15;      // doubles per kept bond
constexpr int L64_GROUP = L64_SLOTS * L64_WORDS + 1;
constexpr int L64_PAIR = 8, L64_TRIP = 7;
// a column's doubles per (ti, tj): the pair fields, then the triplet sums per tk
template <int NT> constexpr int l64_per = L64_PAIR + NT * L64_TRIP;
template <int NT> constexpr size_t l64_dyn() {
  return sizeof(double) * ((size_t)(L64_BLOCK / L64_W) * L64_GROUP + (size_t)NT * NT * l64_per<NT> * L64_BLOCK);
}

struct BondC {
  BondD<double> b;
  Cut<double> f;  // of record (ti, t, t)
};

// What the loops need of one record besides the raw fields.
struct RecC {
  double ga, h, d2, id2, c2, k2, l3, R, D;  // k2 = -2 gamma c^2
  int m, expo;  // expo: the exponential factor or its lambda3-derivative can be other than 1 and 0
};

// One lane's bond qj of the centre atom: the sums of its records' fields.
// get(q, bond): false outside the filter radius.
template <int NT, class Get>
__device__ __forceinline__ void bond_adjoint64(const double* sraw, const RecC* rec, bool cut_j, int ns, int ti, double hE,
                                               int qj, int count, Get get, double* col) {
  BondC j;
  if (!get(qj, j)) return;
  const BondD<double>& bj = j.b;
  const int tj = bj.t;
  const int p = (ti * ns + tj) * ns + tj;
  const double rj = bj.r, rdj = bj.rd;
  const RecC* rj_ = rec + (ti * ns + tj) * ns;
  if (!(rj < rec[p].R + rec[p].D)) return;
  double zeta = 0.0, zd = 0.0;
  for (int qk = 0; qk < count; ++qk) {
    if (qk == qj) continue;
    BondC k;
    if (!get(qk, k)) continue;
    const RecC& c = rj_[k.b.t];
    if (!cut_j) k.f = cutoff_ad<double>(k.b.r, c.R, c.D);
    if (__double_as_longlong(k.f.fc) == 0) continue;  // beyond the cutoff
    const double cs = bj.ux * k.b.ux + bj.uy * k.b.uy + bj.uz * k.b.uz;
    const double csd = (bj.px * k.b.ux + bj.py * k.b.uy + bj.pz * k.b.uz) +
                       (k.b.px * bj.ux + k.b.py * bj.uy + k.b.pz * bj.uz);
    const double t = c.h - cs, t2 = t * t, iden = fx::rcp(c.d2 + t2);
    const double g = c.ga * fma(c.c2, t2 * c.id2 * iden, 1.0);
    const double dg = c.k2 * t * (iden * iden);
    double T0 = k.f.fc * g, T1 = k.f.dfc * k.b.rd * g + k.f.fc * dg * csd;
    if (c.expo) {
      const Expo<double> ex = expo_ad<double>(rj - k.b.r, c.l3, c.m);
      T1 = T1 * ex.x + T0 * ex.dx * (rdj - k.b.rd);
      T0 *= ex.x;
    }
    zeta += T0;
    zd += T1;
  }
  const Cut<double> fj = cut_j ? j.f : cutoff_ad<double>(rj, rec[p].R, rec[p].D);
  const double A = rec_val(sraw, p, TERSOFF_P_A), l1 = rec_val(sraw, p, TERSOFF_P_LAMBDA1);
  const double B = rec_val(sraw, p, TERSOFF_P_B), l2 = rec_val(sraw, p, TERSOFF_P_LAMBDA2);
  const double e1 = fx::exp(-l1 * rj), e2 = fx::exp(-l2 * rj);
  const double Ae1 = A * e1, Be2 = B * e2;
  const double Pv = fj.fc * Ae1, Pd1 = fj.dfc - l1 * fj.fc, Pd = Pd1 * Ae1;
  const double Qv = -fj.fc * Be2, Qd1 = fj.dfc - l2 * fj.fc, Qd = -Qd1 * Be2;
  const Bo<double> bo = bond_ad<double>(zeta, rec_val(sraw, p, TERSOFF_P_BETA), rec_val(sraw, p, TERSOFF_P_N));
  const double Pdbar = -0.5 * rdj;
  const double Qbar = hE * bo.b - 0.5 * bo.db * zd;
  const double Qdbar = -0.5 * bo.b * rdj;
  const double bbar = hE * Qv - 0.5 * Qd * rdj;
  const double dbbar = -0.5 * Qv * zd;
  double* const c0 = col + (size_t)(ti * NT + tj) * l64_per<NT> * L64_BLOCK;
  c0[0 * L64_BLOCK] += (hE * fj.fc + Pdbar * Pd1) * e1;                                          // A
  c0[1 * L64_BLOCK] += hE * (-rj * Pv) + Pdbar * (-fj.fc * Ae1 - rj * Pd);                       // lambda1
  c0[2 * L64_BLOCK] -= (Qbar * fj.fc + Qdbar * Qd1) * e2;                                        // B
  c0[3 * L64_BLOCK] += Qbar * (-rj * Qv) + Qdbar * (fj.fc * Be2 - rj * Qd);                      // lambda2
  c0[4 * L64_BLOCK] += (hE * fj.fc_R + Pdbar * (fj.dfc_R - l1 * fj.fc_R)) * Ae1 -
                       (Qbar * fj.fc_R + Qdbar * (fj.dfc_R - l2 * fj.fc_R)) * Be2;               // R
  c0[5 * L64_BLOCK] += (hE * fj.fc_D + Pdbar * (fj.dfc_D - l1 * fj.fc_D)) * Ae1 -
                       (Qbar * fj.fc_D + Qdbar * (fj.dfc_D - l2 * fj.fc_D)) * Be2;               // D
  c0[6 * L64_BLOCK] += bbar * bo.b_be + dbbar * bo.db_be;                                        // beta
  c0[7 * L64_BLOCK] += bbar * bo.b_n + dbbar * bo.db_n;                                          // n
  const double zbar = bbar * bo.db + dbbar * bo.ddb;
  const double zdbar = -0.5 * Qv * bo.db;
  if (zbar == 0.0 && zdbar == 0.0) return;
  double s[NT][L64_TRIP];
#pragma unroll
  for (int q = 0; q < NT; ++q)
#pragma unroll
    for (int x = 0; x < L64_TRIP; ++x) s[q][x] = 0.0;
  for (int qk = 0; qk < count; ++qk) {
    if (qk == qj) continue;
    BondC k;
    if (!get(qk, k)) continue;
    const RecC& c = rj_[k.b.t];
    if (!cut_j) k.f = cutoff_ad<double>(k.b.r, c.R, c.D);
    if (__double_as_longlong(k.f.fc) == 0) continue;
    const double cs = bj.ux * k.b.ux + bj.uy * k.b.uy + bj.uz * k.b.uz;
    const double csd = (bj.px * k.b.ux + bj.py * k.b.uy + bj.pz * k.b.uz) +
                       (k.b.px * bj.ux + k.b.py * bj.uy + k.b.pz * bj.uz);
    const double t = c.h - cs, t2 = t * t, den = c.d2 + t2, iden = fx::rcp(den), iden2 = iden * iden;
    const double x = t2 * c.id2 * iden, w = t * iden2;
    const double g = c.ga * fma(c.c2, x, 1.0), dg = c.k2 * w;
    const double dl = rj - k.b.r, dld = rdj - k.b.rd;
    Expo<double> ex{1.0, 0.0, 0.0, 0.0};
    if (c.expo) ex = expo_ad<double>(dl, c.l3, c.m);
    // T = F3 G X ; T_rate = F3' rd_k G X + F3 G' cs_rate X + F3 G X' dl_rate
    const double rdk = k.b.rd, fc = k.f.fc, dfc = k.f.dfc;
    const double zx = zbar * ex.x + zdbar * ex.dx * dld, dx = zdbar * ex.x;
    const double F3bar = g * zx + dx * dg * csd;
    const double F3dbar = dx * rdk * g;
    const double Gbar = fc * zx + dx * dfc * rdk;
    const double Gdbar = dx * fc * csd;
    const double Xbar = zbar * fc * g + zdbar * (dfc * rdk * g + fc * dg * csd);
    const double Xdbar = zdbar * fc * g * dld;
    double v[L64_TRIP];
    v[0] = F3bar * k.f.fc_R + F3dbar * k.f.dfc_R;
    v[1] = F3bar * k.f.fc_D + F3dbar * k.f.dfc_D;
    v[2] = Gbar;
    v[3] = Gbar * x - 2.0 * Gdbar * w;
    // d (times d): -t^2 (2 d^2 + t^2)/(d^2 den^2) and 4 t d^2 / den^3; h: w and
    // -(den - 4 t^2)/den^3
    v[4] = 4.0 * Gdbar * w * iden * c.d2 - Gbar * t2 * (c.d2 + den) * (c.id2 * iden2);
    v[5] = Gbar * w - Gdbar * (den - 4.0 * t2) * (iden2 * iden);
    v[6] = Xbar * ex.x_l + Xdbar * ex.dx_l;
#pragma unroll
    for (int q = 0; q < NT; ++q)
      if (NT == 1 || k.b.t == q) {
#pragma unroll
        for (int y = 0; y < L64_TRIP; ++y) s[q][y] += v[y];
      }
  }
#pragma unroll
  for (int q = 0; q < NT; ++q)
#pragma unroll
    for (int y = 0; y < L64_TRIP; ++y) c0[(L64_PAIR + q * L64_TRIP + y) * L64_BLOCK] += s[q][y];
}

template <int NT, bool BATCH>
__global__ void __launch_bounds__(L64_BLOCK, 3) k_bwd_lanes64(const __grid_constant__ BwdArgs<double> a, int cut_j) {
  constexpr int NREC = NT * NT * NT, PER = l64_per<NT>;
  __shared__ double sraw[NREC * NP];
  __shared__ RecC rec[NREC];
  __shared__ float sfilt[NT * NT];
  extern __shared__ __align__(16) unsigned char l64_dyn_[];
  double* const slots = reinterpret_cast<double*>(l64_dyn_);
  double* const cols = slots + (L64_BLOCK / L64_W) * L64_GROUP;
  const fwd::FwdArgs<double>& g = a.g;
  constexpr int ns = NT;
  for (int q = threadIdx.x; q < NREC * NP; q += L64_BLOCK) sraw[q] = a.raw[q];
  if (threadIdx.x < NT * NT) sfilt[threadIdx.x] = g.filt2[threadIdx.x];
  for (int q = 0; q < NT * NT * PER; ++q) cols[q * L64_BLOCK + threadIdx.x] = 0.0;
  __syncthreads();
  if (threadIdx.x < NREC) {
    const double* r = sraw + threadIdx.x * NP;
    RecC c;
    const double d = r[TERSOFF_P_D], cc = r[TERSOFF_P_C];
    c.ga = r[TERSOFF_P_GAMMA];
    c.h = r[TERSOFF_P_H];
    c.d2 = d * d;
    c.id2 = 1.0 / c.d2;
    c.c2 = cc * cc;
    c.k2 = -2.0 * c.ga * c.c2;
    c.l3 = r[TERSOFF_P_LAMBDA3];
    c.m = fwd::small_int(r[TERSOFF_P_M]);
    c.expo = c.l3 != 0.0 || c.m == 1;  // (m = 1: X_lambda3 = Delta at lambda3 = 0)
    c.R = r[TERSOFF_P_R];
    c.D = r[TERSOFF_P_D_CUT];
    rec[threadIdx.x] = c;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, q = lane & (L64_W - 1), gb = lane & ~(L64_W - 1);
  double* const my = slots + (threadIdx.x / L64_W) * L64_GROUP;
  double* const col = cols + threadIdx.x;
  constexpr int ATOMS = L64_BLOCK / L64_W;
  // warp-uniform loop: every lane takes part in the votes
  for (int it0 = blockIdx.x * ATOMS; it0 < g.n; it0 += gridDim.x * ATOMS) {
    const int item = it0 + threadIdx.x / L64_W;
    const bool have = item < g.n;
    const int i = have ? a.fine[item] : 0;
    ipos4 pi{};
    fwd::Shift<double, BATCH> sh;
    int ti = 0, c = 0;
    double gf0 = 0.0, gf1 = 0.0, gf2 = 0.0, hE = 0.0;
    const bool hasF = a.gF != nullptr;
    if (have) {
      pi = g.pos64[i];
      sh.load(g, i);
      ti = (int)pi.w;
      c = min(g.cnt[i], g.cap);
      hE = 0.5 * a.gE[a.atom_cell ? a.atom_cell[i] : 0];
      if (hasF) {
        gf0 = a.gF[3 * (size_t)i];
        gf1 = a.gF[3 * (size_t)i + 1];
        gf2 = a.gF[3 * (size_t)i + 2];
      }
    }
    // list entry s: bond data; false outside the filter radius
    auto from_list = [&](int s, BondC& k) -> bool {
      long long dx, dy, dz;
      int j, t;
      Bond<double>::fixed(g, sh, pi, g.nbr[(size_t)s * g.n + i], dx, dy, dz, j, t);
      if (!(fwd::coarse2(g, dx, dy, dz) <= sfilt[ti * ns + t])) return false;
      BondD<double>& b = k.b;
      const double x = fx::from_fixed(dx, g.fix64), y = fx::from_fixed(dy, g.fix64), z = fx::from_fixed(dz, g.fix64);
      const double r2 = x * x + y * y + z * z;
      const double ir = fx::rsqrt(r2);
      b.r = fx::sqrt(r2);
      b.ux = x * ir;
      b.uy = y * ir;
      b.uz = z * ir;
      double wx = 0.0, wy = 0.0, wz = 0.0;
      if (hasF) {
        wx = a.gF[3 * (size_t)j] - gf0;
        wy = a.gF[3 * (size_t)j + 1] - gf1;
        wz = a.gF[3 * (size_t)j + 2] - gf2;
      }
      b.rd = b.ux * wx + b.uy * wy + b.uz * wz;
      b.px = (wx - b.ux * b.rd) * ir;
      b.py = (wy - b.uy * b.rd) * ir;
      b.pz = (wz - b.uz * b.rd) * ir;
      b.t = t;
      const RecC& p = rec[(ti * ns + t) * ns + t];
      k.f = cutoff_ad<double>(b.r, p.R, p.D);
      return true;
    };
    // the group's bonds, eight list entries at a time
    int z = 0, cmax = c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    for (int c0 = 0; c0 < cmax; c0 += L64_W) {
      BondC k;
      const bool ok = c0 + q < c && from_list(c0 + q, k);
      const unsigned m = (__ballot_sync(0xffffffffu, ok) >> gb) & ((1u << L64_W) - 1u);
      const int at = z + __popc(m & ((1u << q) - 1u));
      if (ok && at < L64_SLOTS) {
        double* s = my + at * L64_WORDS;
        s[0] = k.b.ux;
        s[1] = k.b.uy;
        s[2] = k.b.uz;
        s[3] = k.b.r;
        s[4] = k.b.rd;
        s[5] = k.b.px;
        s[6] = k.b.py;
        s[7] = k.b.pz;
        fwd::put_int(s[8], k.b.t);
        s[9] = k.f.fc;
        s[10] = k.f.dfc;
        s[11] = k.f.fc_R;
        s[12] = k.f.fc_D;
        s[13] = k.f.dfc_R;
        s[14] = k.f.dfc_D;
      }
      z += __popc(m);
    }
    __syncwarp();
    if (z <= L64_SLOTS) {
      auto get = [&](int b, BondC& k) -> bool {
        const double* s = my + b * L64_WORDS;
        k.b.ux = s[0];
        k.b.uy = s[1];
        k.b.uz = s[2];
        k.b.r = s[3];
        k.b.rd = s[4];
        k.b.px = s[5];
        k.b.py = s[6];
        k.b.pz = s[7];
        k.b.t = fwd::get_int(s[8]);
        k.f.fc = s[9];
        k.f.dfc = s[10];
        k.f.fc_R = s[11];
        k.f.fc_D = s[12];
        k.f.dfc_R = s[13];
        k.f.dfc_D = s[14];
        return true;
      };
      for (int j = q; j < z; j += L64_W) bond_adjoint64<NT>(sraw, rec, cut_j != 0, ns, ti, hE, j, z, get, col);
    } else {
      for (int j = q; j < c; j += L64_W) bond_adjoint64<NT>(sraw, rec, cut_j != 0, ns, ti, hE, j, c, from_list, col);
    }
    __syncwarp();  // the slots are free for the next atom
  }
  __syncthreads();
  // the block's sums, with the constants of each record
  for (int w = threadIdx.x; w < NT * NT * PER; w += L64_BLOCK) {
    const double* s = cols + (size_t)w * L64_BLOCK;
    double v0 = 0.0, v1 = 0.0;
    for (int t = 0; t < L64_BLOCK; t += 2) {
      v0 += s[t];
      v1 += s[t + 1];
    }
    cols[(size_t)w * L64_BLOCK] = v0 + v1;  // (only this thread reads the column row)
  }
  __syncthreads();
  for (int w = threadIdx.x; w < NT * NT * PER; w += L64_BLOCK) {
    const int pr = w / PER, f = w % PER, ti = pr / NT, tj = pr % NT;
    const double v = cols[(size_t)w * L64_BLOCK];
    if (v == 0.0) continue;
    if (f < L64_PAIR) {
      constexpr int field[L64_PAIR] = {TERSOFF_P_A, TERSOFF_P_LAMBDA1, TERSOFF_P_B,    TERSOFF_P_LAMBDA2,
                                       TERSOFF_P_R, TERSOFF_P_D_CUT,   TERSOFF_P_BETA, TERSOFF_P_N};
      int fl = field[0];
#pragma unroll
      for (int y = 1; y < L64_PAIR; ++y) fl = f == y ? field[y] : fl;
      atomicAdd(&a.grad[((ti * ns + tj) * ns + tj) * NP + fl], v);
      continue;
    }
    const int tk = (f - L64_PAIR) / L64_TRIP, y = (f - L64_PAIR) % L64_TRIP;
    const int r = (ti * ns + tj) * ns + tk;
    double* const out = a.grad + r * NP;
    const RecC& c = rec[r];
    const double cc = sraw[r * NP + TERSOFF_P_C], d = sraw[r * NP + TERSOFF_P_D];
    switch (y) {
      case 0: atomicAdd(out + TERSOFF_P_R, v); break;
      case 1: atomicAdd(out + TERSOFF_P_D_CUT, v); break;
      case 2: atomicAdd(out + TERSOFF_P_GAMMA, v); break;
      case 3:
        atomicAdd(out + TERSOFF_P_GAMMA, c.c2 * v);
        atomicAdd(out + TERSOFF_P_C, 2.0 * c.ga * cc * v);
        break;
      case 4: atomicAdd(out + TERSOFF_P_D, -c.k2 / d * v); break;
      case 5: atomicAdd(out + TERSOFF_P_H, -c.k2 * v); break;
      default: atomicAdd(out + TERSOFF_P_LAMBDA3, v); break;
    }
  }
}

}  // namespace bwd
}  // namespace tgb
