// Force kernel of the FP64 path: one lane per bond, integer arithmetic.
//
// W lanes (4, 8 or 16) hold the bonds of one centre atom, one each; the other
// bonds' data arrive by warp shuffles (the paper's scheme (a), Sec. IV-B). The
// lane forms its bond, zeta over the other bonds (first K loop), the pair
// term, and, with the other bonds' dV/dzeta, the force on its neighbour
// (second K loop). The force on the atom is the negated group sum.
//
// Bound: issue and latency, with the FP64 pipe 62% busy. The terms are integer
// arithmetic (tersoff_fx.cuh) with some 40 FP64 instructions per lane. A thread
// per atom of the same arithmetic needs 168 registers for four bonds: 11 warps
// share an SM and 30% of the issue slots are taken (512,000 atoms, ten MD
// steps: 4.20 ms; 4,096 atoms, one evaluation: 51 us). A lane per bond needs
// 80 registers: 23 warps, half of the slots (3.85 ms, 32 us; the FP64 formulas
// with integer elementary functions 5.71 ms, 52 us). That is six blocks per SM,
// with the forces only; a launch bound of four (128 registers) 4.38 ms, five (96)
// 4.06, seven (72) 4.02, eight (64) 4.15. Instances whose shared memory leaves
// fewer blocks get their registers (lanes_blocks): 80 for all of them spilled 130
// to 690 bytes (4,096 atoms, one evaluation 32.8 -> 31.6 us; an evaluation with
// energy of 92,736 SiC atoms 259 -> 238).
// Lists of five to eight bonds take 8 lanes and of up to sixteen 16 lanes: 24
// fitting cells with lambda3 spend 77 and 68 us there, where a thread per atom
// with eight bonds in registers and with bonds in shared memory took 373 and
// 870.
//
// MODE 3: symmetric tables without lambda3 (each pair's g and dg/dcos serve
// both bonds). MODE 1: any other table inside the integer formats; every
// ordered triplet's three derivatives are kept in shared memory, where the
// partner lane reads them in the second loop.
//
// Items: atoms of a launch's bucket, or all. An atom with more bonds inside
// the cutoffs than lanes joins a block-local list and is done by 16 lanes, one
// with more than 16 by one thread over its list (the general path).
//
// LONG: boxes with an edge beyond 2,048 A (pos64.cuh), as instances for a run-time
// species count with energy and virial: the choice of the image inside the other
// instances cost 2.6% of ten MD steps of 512,000 atoms.
//
// Forces: per-slot stores into the receiving atoms' columns (gather scatter)
// or FP64 atomics, with the kmask bookkeeping of k_tersoff.
#pragma once
#include "tersoff_fwd.cuh"

namespace tgb {
namespace fwd {

constexpr int LBLOCK = 128;
constexpr int lanes_scratch(int W, int mode) {  // doubles per thread in dynamic shared memory
  return mode == 1 ? 3 * W : (W == 4 ? 0 : 2 * W);
}
// (the block-local rest runs with 16 lanes)
constexpr size_t lanes_dyn(int mode) { return sizeof(double) * LBLOCK * lanes_scratch(16, mode); }
// Blocks of an instance on one SM, for its launch bound and for grids of one wave:
// six, or what shared memory leaves (228 KB, 1 KB of it per block; the tables of
// several species, the sums over atoms, the scratch): 5 with energy sums and one or
// two species, 4 and 3 with lambda3, 3 and 2 for a run-time species count.
constexpr int LANES_BLOCKS = 6;
template <int NS, int MODE, bool BATCH, int EV> constexpr int lanes_blocks() {
  constexpr int SNS = NS > 0 ? NS : TERSOFF_MAX_SPECIES;
  constexpr size_t tables = NS == 1 ? 0 : (size_t)SNS * SNS * SNS * (sizeof(double) * RSTRIDE + sizeof(FxRec));
  constexpr size_t sums = EV >= 1 && !BATCH ? sizeof(double) * (7 * LBLOCK + 8 * (LBLOCK / 32)) : 0;
  constexpr int fit = (int)(233472 / (tables + sums + 512 + lanes_dyn(MODE) + 1024));
  return fit < LANES_BLOCKS ? fit : LANES_BLOCKS;
}

template <class T>
__device__ __forceinline__ T lsh(T v, int src) { return __shfl_sync(0xffffffffu, v, src); }
template <int W>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = 1; o < W; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// What every atom of a launch shares.
struct LaneEnv {
  const double* srec;   // double records
  const FxRec* frec;    // integer records
  const float* sfilt;   // squared filter radii
  int ns;
  bool slots, use_short, want_acc;
  double* scr;          // dynamic shared memory: word w of thread t at [w * LBLOCK + t]
  double* tsum;         // this thread's energy and virial sums (stride LBLOCK)
};

// One atom by W lanes. Every lane of the warp calls it; `have`: the group has
// an atom. Returns whether the atom is left (more bonds than lanes).
template <int NS, int W, int MODE, int BATCH, int EV, int LONG>
__device__ __forceinline__ bool lanes_atom(const FwdArgs<double>& a, const LaneEnv& v, int i, bool have) {
  const int lane = threadIdx.x & 31, q = lane & (W - 1), gb = lane & ~(W - 1);
  const int ns = NS > 0 ? NS : v.ns;
  int zl = 0, ti = 0;
  ipos4 pi{};
  Shift<double, BATCH, LONG> sh;
  if (have) {
    zl = a.zcnt[i];
    pi = a.pos64[i];
    ti = NS == 1 ? 0 : (int)pi.w;
    sh.load(a, i);
  }
  // a position that is not finite, of the atom or of one on its list, or a
  // neighbour at its own place: the lane has seen one
  bool odd = have && pos64_bad(pi);
  const uint32_t* list = a.shortl;
  int c = zl;
  bool left = have && v.use_short && (zl > a.zs_cap || zl > 64);
  if (have && !v.use_short) {
    list = a.nbr;
    c = min(a.cnt[i], a.cap);
  }
  // the lane's entry and its list slot
  uint32_t e = 0;
  int sl = -1, nb = 0;
  const bool filtered = have && !left && (!v.use_short || c > W);
  unsigned long long kept = 0ull;
  if (__any_sync(0xffffffffu, filtered)) {
    // keep the entries inside the cutoffs, W at a time; the loop runs to the
    // warp's longest list (every lane takes part in the votes)
    int nk = 0;
    const int cl = filtered ? c : 0;
    int cmax = cl;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cmax = max(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    for (int c0 = 0; c0 < cmax; c0 += W) {
      const int s = c0 + q;
      uint32_t es = 0;
      bool ok = false;
      if (s < cl) {
        es = list[(size_t)s * a.n + i];
        long long dx, dy, dz;
        int jj, tj;
        odd |= Bond<double>::fixed(a, sh, pi, es, dx, dy, dz, jj, tj);
        ok = coarse2(a, dx, dy, dz) <= v.sfilt[ti * ns + tj];
      }
      const unsigned m = (__ballot_sync(0xffffffffu, ok) >> gb) & ((1u << W) - 1u);
      const int cnt = __popc(m);
      // lane q receives the (q - nk)-th kept entry of this chunk
      const int want = q - nk;
      const bool take = want >= 0 && want < cnt;
      const int src = take ? (int)__fns(m, 0, want + 1) : 0;
      const uint32_t ein = __shfl_sync(0xffffffffu, es, gb + src);
      if (take) {
        e = ein;
        sl = c0 + src;
      }
      if (ok && s < 64) kept |= 1ull << s;
      nk += cnt;
    }
    if (filtered && nk > W) left = true;
    if (filtered) nb = nk;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) kept |= __shfl_xor_sync(0xffffffffu, kept, o);
  }
  if (have && !left && !filtered) {
    nb = c;
    if (q < c) {
      e = list[(size_t)q * a.n + i];
      sl = q;
    }
  }
  const bool act = have && !left;
  const bool mine = act && sl >= 0;
  // (read by every lane of the group before its first one writes it below)
  const unsigned long long was = v.slots && act && filtered ? a.kmask[i] : 0ull;
  __syncwarp();
  // forces through the fallback buffer while the gather still runs: it must
  // see zero in the atom's own slot and column (lanes take slots q, q + W, ...)
  if (act && !v.slots && !a.atomic_mode) {
    if (q == 0) store_slot<double>(a, a.own, (size_t)i, 0.0, 0.0, 0.0);
    const int zc = min(zl, a.zs_cap);
    for (int p = q; p < zc; p += W) store_slot<double>(a, a.contrib, (size_t)p * a.n + i, 0.0, 0.0, 0.0);
  }
  // 1. the lane's bond; entries outside the cutoffs take no part
  int j = i, tj = 0, rv = 0;
  if (v.slots && mine && !filtered) rv = (int)__ldg(&a.rev[(size_t)q * a.n + i]);
  long long bx = 0, by = 0, bz = 0;
  fx::Bond64 b{};
  double fc = 0.0, dfc = 0.0, r = 1.0;
  bool near = false, taper = false;
  if (mine) {
    odd |= Bond<double>::fixed(a, sh, pi, e, bx, by, bz, j, tj);
    if (coarse2(a, bx, by, bz) <= v.sfilt[ti * ns + tj]) {
      b = fx::bond64(bx, by, bz, a.fix64);
      odd |= b.r.e < -a.fix64 - 8;  // the zero vector's, far below one unit
      r = fx::pack_in(b.r);
      const double* pq = v.srec + rec_off<NS>(ns, ti, tj, tj);
      const long long rb = __double_as_longlong(r);  // positive doubles order like their bits
      // MODE 1: a three-body cutoff may lie beyond the pair's
      near = MODE == 1 || rb < __double_as_longlong(pq[K_ROUT2]);
      if (rb < __double_as_longlong(pq[K_ROUT2])) {
        fc = 1.0;
        if (rb > __double_as_longlong(pq[K_RIN2])) {
          taper = true;
          cutoff<double>(pq, K_PID2, K_DFC2, K_RIN2, K_ROUT2, K_ROUT2LO, r, fc, dfc);
        }
      }
    }
  }
  // the other bonds of the group: the first M lanes in rotation
  int M = W;
  if (W > 4) {
    M = act ? nb : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) M = max(M, __shfl_xor_sync(0xffffffffu, M, o));
  }
  auto partner = [&](int o) {
    int t = q + o;
    t -= t >= M ? M : 0;
    return t < W ? t : 0;
  };
  const bool wtaper = __any_sync(0xffffffffu, taper) || MODE == 1;
  const FxRec& p2 = v.frec[NS == 1 ? 0 : (ti * ns + tj) * ns + tj];
  double* const my = v.scr + threadIdx.x;
  // 2. first K loop
  double zeta = 0.0;
  constexpr int R = W == 4 && MODE == 3 ? 3 : 1;
  double g_[R], dg_[R];
  auto first = [&](int o, double& g, double& dg) {
    const int t = partner(o), src = gb + t;
    const long long kx = lsh((long long)b.ux, src), ky = lsh((long long)b.uy, src), kz = lsh((long long)b.uz, src);
    const bool kn = lsh((int)near, src) != 0;
    const double kf = wtaper ? lsh(fc, src) : 1.0;
    const int kt = NS == 1 ? 0 : lsh(tj, src);
    g = dg = 0.0;
    const bool both = near && kn && t != q;
    const FxRec& p3 = v.frec[NS == 1 ? 0 : (ti * ns + tj) * ns + kt];
    if (MODE == 3) {
      // without a branch (lanes without a bond compute on zeros), so that the
      // three pairs of four bonds overlap
      const long long cs = fx::smulhi(b.ux, kx) + fx::smulhi(b.uy, ky) + fx::smulhi(b.uz, kz);
      fx::angle64(p3, cs, g, dg);
      g = both ? g : 0.0;
      dg = both ? dg : 0.0;
      zeta = fma(kf, g, zeta);
      return;
    }
    const double kr = lsh(r, src), kd = lsh(dfc, src);
    double A1 = 0.0, A2 = 0.0, A3 = 0.0;
    if (both) {
      double f = kf, df = kd;
      const double* p3d = v.srec + rec_off<NS>(ns, ti, tj, kt);
      if (!a.cut_j)  // f_C(r_ik) depends on j
        cutoff<double>(p3d, K_PID3, K_DFC3, K_RIN3, K_ROUT3, K_ROUT3LO, kr, f, df);
      if (f != 0.0) {
        const long long cs = fx::smulhi(b.ux, kx) + fx::smulhi(b.uy, ky) + fx::smulhi(b.uz, kz);
        fx::angle64(p3, cs, g, dg);
        double ex = 1.0, dex = 0.0;
        const double l3 = p3d[K_LAM3];
        if (__double_as_longlong(l3) != 0) {
          const int m = small_int(p3d[K_M]);
          const double aa = l3 * (r - kr);
          double am1 = 1.0;
          for (int s = 1; s < m; ++s) am1 *= aa;
          ex = fx::exp(am1 * aa);
          dex = ex * p3d[K_M] * l3 * am1;
        }
        const double fg = f * g;
        zeta = fma(fg, ex, zeta);
        A1 = f * dg * ex;
        A2 = fg * dex;
        A3 = df * g * ex;
      }
    }
    // by the partner's lane, which reads them in the second loop
    my[(3 * t + 0) * LBLOCK] = A1;
    my[(3 * t + 1) * LBLOCK] = A2;
    my[(3 * t + 2) * LBLOCK] = A3;
  };
  if (W == 4) {
#pragma unroll
    for (int o = 1; o < 4; ++o) {
      double g, dg;
      first(o, g, dg);
      if (R == 3) {
        g_[R == 3 ? o - 1 : 0] = g;
        dg_[R == 3 ? o - 1 : 0] = dg;
      }
    }
  } else {
    for (int o = 1; o < M; ++o) {
      double g, dg;
      first(o, g, dg);
      if (MODE == 3) {
        my[(2 * o + 0) * LBLOCK] = g;
        my[(2 * o + 1) * LBLOCK] = dg;
      }
    }
  }
  // 3. pair level: ra = -dV/dr at fixed zeta
  double V = 0.0, ra = 0.0, dz = 0.0;
  if (near && fc != 0.0) {
    double fr, bfa;
    if (fx::pair64(p2, b.r.m, b.r.e, zeta, &fr, &bfa, &dz)) {
      ra = fma(p2.hl1, fr, p2.hl2 * bfa);
      if (EV >= 1) V = 0.5 * (fr + bfa);
      if (taper) {
        if (EV >= 1) V *= fc;
        ra = fma(fc, ra, -0.5 * dfc * (fr + bfa));
        dz *= fc;
      }
    } else {  // zeta = 0, or outside the formats
      double dVdr;
      pair_fc<double>(v.srec + rec_off<NS>(ns, ti, tj, tj), r, zeta, fc, dfc, V, dVdr, dz);
      ra = -dVdr;
    }
  }
  // 4. second K loop: F = (G - (u . G) u) / r + ra u
  const double ux = fx::from_fixed(b.ux, 62), uy = fx::from_fixed(b.uy, 62), uz = fx::from_fixed(b.uz, 62);
  double gx = 0.0, gy = 0.0, gz = 0.0;
  if (MODE == 1) __syncwarp();
  auto second = [&](int o, double g, double dg) {
    const int t = partner(o), src = gb + t;
    const double kx = lsh(ux, src), ky = lsh(uy, src), kz = lsh(uz, src);
    const double kdz = lsh(dz, src);
    double A;
    if (MODE == 3) {
      if (wtaper) {
        const double kf = lsh(fc, src);
        A = -fma(dz, kf, kdz * fc) * dg;
        ra = fma(-kdz * dfc, g, ra);
      } else {
        A = -(dz + kdz) * dg;
      }
    } else {
      if (t == q) return;
      // the partner's column, at this lane's place
      const double* their = v.scr + (threadIdx.x - q + t);
      const double B1 = their[(3 * q + 0) * LBLOCK], B2 = their[(3 * q + 1) * LBLOCK],
                   B3 = their[(3 * q + 2) * LBLOCK];
      A = -fma(dz, my[(3 * t) * LBLOCK], kdz * B1);
      ra -= fma(dz, my[(3 * t + 1) * LBLOCK], kdz * (B3 - B2));
    }
    gx = fma(A, kx, gx);
    gy = fma(A, ky, gy);
    gz = fma(A, kz, gz);
  };
  if (W == 4) {
#pragma unroll
    for (int o = 1; o < 4; ++o) second(o, g_[R == 3 ? o - 1 : 0], dg_[R == 3 ? o - 1 : 0]);
  } else {
    for (int o = 1; o < M; ++o)
      second(o, MODE == 3 ? my[(2 * o) * LBLOCK] : 0.0, MODE == 3 ? my[(2 * o + 1) * LBLOCK] : 0.0);
  }
  if (MODE == 1) __syncwarp();  // the columns are free for the next atom
  double fx_ = 0.0, fy_ = 0.0, fz_ = 0.0;
  if (near) {
    const double ri = fx::pack_in(b.ri);
    const double w = fma(-ri, fma(gx, ux, fma(gy, uy, gz * uz)), ra);
    fx_ = fma(ri, gx, w * ux);
    fy_ = fma(ri, gy, w * uy);
    fz_ = fma(ri, gz, w * uz);
  }
  // such an atom's energy and all forces of its terms are NaN
  if ((__ballot_sync(0xffffffffu, odd) >> gb) & ((1u << W) - 1u)) {
    V = fx_ = fy_ = fz_ = fx::nan64();
    near = true;
  }
  // 5. stores: the lane's neighbour force, the atom's own (lane 0)
  const double ox = -group_sum<W>(fx_), oy = -group_sum<W>(fy_), oz = -group_sum<W>(fz_);
  if (mine) {
    if (v.slots)
      store_slot<double>(a, a.contrib, filtered ? recv_slot(a, sl, i, j) : (size_t)rv * a.n + j, fx_, fy_, fz_);
    else if (near)
      atomic_add3(a.f, j, fx_, fy_, fz_);
  }
  if (act && q == 0) {
    if (v.slots)
      store_slot<double>(a, a.own, (size_t)i, ox, oy, oz);
    else
      atomic_add3(a.f, i, ox, oy, oz);
  }
  if (v.slots && act) {
    if (filtered) {
      // stored entries outside the cutoffs now: their receiving slots get zero
      // unless they hold zero already
      unsigned long long clr = was & ~kept;
      if (zl < 64) clr &= (1ull << zl) - 1ull;
      for (int s = q; s < 64; s += W)
        if ((clr >> s) & 1ull)
          store_slot<double>(a, a.contrib, recv_slot(a, s, i, entry_atom(a, a.shortl, s, i)), 0.0, 0.0, 0.0);
      if (q == 0) a.kmask[i] = kept;
    } else if (q == 0 && zl > 4) {
      a.kmask[i] = ~0ull;  // every entry written
    }
  }
  // 6. energy and virial
  if (EV >= 1) {
    double w[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    if (EV == 2 && near) {
      const double dx = fx::from_fixed(bx, a.fix64), dy = fx::from_fixed(by, a.fix64), dzz = fx::from_fixed(bz, a.fix64);
      w[0] = dx * fx_;
      w[1] = dy * fy_;
      w[2] = dzz * fz_;
      w[3] = dx * fy_;
      w[4] = dx * fz_;
      w[5] = dy * fz_;
    }
    if (v.want_acc && near) {
      v.tsum[0] += V;
      if (EV == 2 && (!LONG || a.virial))
        for (int p = 0; p < 6; ++p) v.tsum[(1 + p) * LBLOCK] += w[p];
    }
    if (a.eatom) {
      const double es = group_sum<W>(V);
      if (act && q == 0) a.eatom[i] = es;
    }
    if (BATCH) {
      for (int p = 0; p < 6; ++p) {
        const double s = group_sum<W>(w[p]);
        if (act && q == 0) a.vatom[6 * (size_t)i + p] = s;
      }
    }
  }
  return left && q == 0;
}

template <int NS, int W, int MODE, bool BATCH, int EV, int LONG>
__global__ void __launch_bounds__(LBLOCK, lanes_blocks<NS, MODE, BATCH, EV>()) k_lanes64(const __grid_constant__ FwdArgs<double> a) {
  static_assert(EV == 2 || !BATCH, "batches need the per-atom energy and virial");
  pdl_wait();
  constexpr int SNS = NS > 1 ? NS : (NS == 1 ? 1 : TERSOFF_MAX_SPECIES);
  constexpr int NREC = SNS * SNS * SNS;
  constexpr int FXW = (int)(sizeof(FxRec) / 8);
  __shared__ double srec_s[NS == 1 ? 1 : NREC * RSTRIDE];
  __shared__ unsigned long long sfx[NS == 1 ? 1 : NREC * FXW];
  __shared__ float sfilt[SNS * SNS];
  __shared__ int uni[5], over[2], over_a[LBLOCK / W], over_b[LBLOCK / W];
  __shared__ double tsum[7][LBLOCK];
  extern __shared__ __align__(16) unsigned char lanes_scr[];
  const int ns = NS > 0 ? NS : a.ns;
  if (NS != 1) {
    for (int q = threadIdx.x; q < ns * ns * ns * RSTRIDE; q += LBLOCK) srec_s[q] = a.rec[q];
    for (int q = threadIdx.x; q < ns * ns * ns * FXW; q += LBLOCK)
      sfx[q] = reinterpret_cast<const unsigned long long*>(a.fx)[q];
  }
  if (threadIdx.x < ns * ns) sfilt[threadIdx.x] = a.filt2[threadIdx.x];
  if (threadIdx.x < 5) {
    const int* src = threadIdx.x == 0   ? a.n_items
                     : threadIdx.x == 1 ? a.flags + FLAG_REV_MISS
                     : threadIdx.x == 2 ? a.flags + FLAG_DMAX
                     : threadIdx.x == 3 ? a.n_items2
                                        : a.n_items3;
    uni[threadIdx.x] = src ? *src : 0;
  }
  if (threadIdx.x < 2) over[threadIdx.x] = 0;
  LaneEnv v;
  v.want_acc = EV >= 1 && !BATCH && a.acc != nullptr;  // (a batch's sums are per system)
  if (v.want_acc)
    for (int q = 0; q < 7; ++q) tsum[q][threadIdx.x] = 0.0;
  __syncthreads();
  const int n1 = uni[0], n2 = uni[0] + uni[3];
  const int n_items = a.identity ? a.n : min(n2 + uni[4], a.n);
  v.srec = NS == 1 ? a.prm1 : srec_s;
  v.frec = NS == 1 ? &a.fx1 : reinterpret_cast<const FxRec*>(sfx);
  v.sfilt = sfilt;
  v.ns = ns;
  v.use_short = __int_as_float(uni[2]) <= a.dlim2;
  v.slots = !a.atomic_mode && v.use_short && uni[1] == 0;
  v.scr = reinterpret_cast<double*>(lanes_scr);
  v.tsum = &tsum[0][threadIdx.x];
  if (blockIdx.x == 0 && threadIdx.x == 0) a.flags[FLAG_EXTRA] = v.slots ? 0 : 1;
  constexpr int ATOMS = LBLOCK / W;
  for (int it0 = blockIdx.x * ATOMS; it0 < n_items; it0 += gridDim.x * ATOMS) {
    const int item = it0 + threadIdx.x / W;
    const bool have = item < n_items;
    const int i = !have ? 0
                  : a.identity ? item
                  : item < n1  ? a.order[item]
                  : item < n2  ? a.order2[item - n1]
                               : a.order3[item - n2];
    const bool left = lanes_atom<NS, W, MODE, BATCH, EV, LONG>(a, v, i, have);
    if (left) over_a[atomicAdd(&over[0], 1)] = i;
    // what did not fit: 16 lanes, then a thread each (the barrier's own count,
    // the same for every thread, decides)
    const int na = __syncthreads_count(left);
    if (na > 0) {
      if (W < 16) {
        for (int b0 = 0; b0 < na; b0 += LBLOCK / 16) {
          const int k = b0 + threadIdx.x / 16;
          const int i2 = k < na ? over_a[k] : 0;
          if (lanes_atom<NS, 16, MODE, BATCH, EV, LONG>(a, v, i2, k < na)) over_b[atomicAdd(&over[1], 1)] = i2;
        }
        __syncthreads();
      }
      const int* rest = W < 16 ? over_b : over_a;
      const int nr = W < 16 ? over[1] : na;
      if ((int)threadIdx.x < nr) {
        const int ig = rest[threadIdx.x];
        atomicAdd(&a.flags[FLAG_FALLBACK], 1);
        if (!v.slots && !a.atomic_mode) clear_slots<double>(a, ig);
        Shift<double, BATCH, LONG> sh;
        sh.load(a, ig);
        const int zl = a.zcnt[ig], ti = a.types[ig];
        const bool in_short = v.use_short && zl <= a.zs_cap;
        const uint32_t* list = in_short ? a.shortl : a.nbr;
        const int c = in_short ? zl : min(a.cnt[ig], a.cap);
        if (v.slots && !in_short) {
          atomicOr(&a.flags[FLAG_EXTRA_STICKY], 1);
          zero_stored<double>(a, ig, zl);
        }
        double eg = 0.0, w[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        general_atom<double, NS, MODE == 1, BATCH>(a, sh, v.srec, ig, ti, list, c, v.slots && in_short, false, 0ull, eg, w);
        if (v.slots && in_short) a.kmask[ig] = ~0ull;  // every entry written
        const ipos4 pg = a.pos64[ig];
        bool odd = pos64_bad(pg);
        for (int s = 0; s < c; ++s) {
          long long dx, dy, dz;
          int jj, tj;
          odd |= Bond<double>::fixed(a, sh, pg, list[(size_t)s * a.n + ig], dx, dy, dz, jj, tj) || (dx | dy | dz) == 0;
        }
        if (odd) {  // as in lanes_atom, the forces on its neighbours too
          eg = fx::nan64();
          for (int p = 0; p < 6; ++p) w[p] = eg;
          const bool st = v.slots && in_short;
          for (int s = 0; s < c; ++s) {
            const int jj = entry_atom(a, list, s, ig);
            if (st)
              store_slot<double>(a, a.contrib, recv_slot(a, s, ig, jj), eg, eg, eg);
            else
              atomic_add3(a.f, jj, eg, eg, eg);
          }
          if (st)
            store_slot<double>(a, a.own, (size_t)ig, eg, eg, eg);
          else
            atomic_add3(a.f, ig, eg, eg, eg);
        }
        if (EV >= 1) {
          if (a.eatom) a.eatom[ig] = eg;
          if (v.want_acc) {
            v.tsum[0] += eg;
            if (!LONG || a.virial)
              for (int p = 0; p < 6; ++p) v.tsum[(1 + p) * LBLOCK] += w[p];
          }
          if (BATCH)
            for (int p = 0; p < 6; ++p) a.vatom[6 * (size_t)ig + p] = w[p];
        }
      }
      __syncthreads();
      if (threadIdx.x < 2) over[threadIdx.x] = 0;
      __syncthreads();
    }
  }
  if (v.want_acc) {
    __syncthreads();
    block_reduce_sums<LBLOCK>(&tsum[0][threadIdx.x], a.acc);
  }
}

}  // namespace fwd
}  // namespace tgb
