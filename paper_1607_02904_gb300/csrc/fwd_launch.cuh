// Host-side instantiation and launch of the force kernel for one precision.
#pragma once
#include <algorithm>

#include "tersoff_lanes64.cuh"

namespace tgb {
namespace fwd {

template <class T> const T* rec_ptr(Ctx* c);
template <> inline const float* rec_ptr<float>(Ctx* c) { return c->d_rec32; }
template <> inline const double* rec_ptr<double>(Ctx* c) { return c->d_rec64; }
template <class T> const T* rec_host(Ctx* c);
template <> inline const float* rec_host<float>(Ctx* c) { return c->h_rec32.data(); }
template <> inline const double* rec_host<double>(Ctx* c) { return c->h_rec64.data(); }

// Atoms with more than 8 bonds inside the cutoffs (bucket 2), when they are
// over 0.5% of the atoms (e.g. SiC): the slot-cached wide kernel,
// beside the main launch (see launch_buckets). A grid of a few waves loops over the
// bucket (its size lives on the device).
template <class T, int NS, bool BATCH = false>
void launch_wide(Ctx* c, const FwdArgs<T>& a, cudaStream_t s) {
  FwdArgs<T> b2 = a;
  b2.order = c->d_bucket + 2 * (size_t)c->n;
  b2.n_items = c->d_flags + flag_bucket(2);
  b2.order2 = b2.order3 = nullptr;
  b2.n_items2 = b2.n_items3 = nullptr;
  b2.identity = 0;
  const size_t dyn = wide_slot_bytes(sizeof(T));
  const int cap = (c->n_sm > 0 ? c->n_sm : 152) * 8;
  const int need = (c->nbucket[2] + WIDE_BLOCK - 1) / WIDE_BLOCK + 1;
  const int grid = need < cap ? need : cap;
  void (*k)(FwdArgs<T>) =
      c->has_lam3 ? k_tersoff_wide<T, NS, true, BATCH> : k_tersoff_wide<T, NS, false, BATCH>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  k<<<grid, WIDE_BLOCK, dyn, s>>>(b2);
  c->launches++;
}

// Energy/virial mode of a force launch (the EV parameter of k_tersoff).
template <class T, bool BATCH>
int ev_mode(const FwdArgs<T>& a) {
  if (BATCH) return 2;
  if (a.acc != nullptr) return a.virial ? 2 : 1;
  return a.eatom != nullptr ? 1 : 0;
}

// MODE by the table: 1 with a lambda3 term, 2 symmetric without one, else 0.
template <class T, int NS, int ZC, bool BATCH, int EV>
void launch_mode(Ctx* c, const FwdArgs<T>& a, int grid, cudaStream_t s) {
  if (c->has_lam3)
    launch_pdl(k_tersoff<T, NS, ZC, 1, BATCH, false, EV>, grid, BLOCK, 0, s, a);
  else if (c->sym_table)
    launch_pdl(k_tersoff<T, NS, ZC, 2, BATCH, false, EV>, grid, BLOCK, 0, s, a);
  else
    launch_pdl(k_tersoff<T, NS, ZC, 0, BATCH, false, EV>, grid, BLOCK, 0, s, a);
}

// Grids are fixed by the atom count (the bucket sizes live on the device), so
// the launches can be captured in a CUDA graph and replayed across builds.
template <class T, int NS, int ZC, bool BATCH = false>
void launch_t(Ctx* c, const FwdArgs<T>& a, int grid, cudaStream_t s) {
  if (grid <= 0) return;
  if (sizeof(T) == 4 && NS == 1 && !BATCH && comp_atom_sums(c)) {
    launch_forward_cs(c, &a, ZC, grid, s);
    return;
  }
  // forces only, or energy without the virial (MD steps, with or without
  // thermo): the instances with less bookkeeping
  const int evm = ev_mode<T, BATCH>(a);
  if constexpr (ZC == 4 && !BATCH) {
    if (evm == 0) {
      launch_mode<T, NS, ZC, BATCH, 0>(c, a, grid, s);
      c->launches++;
      return;
    }
    if (evm == 1) {
      launch_mode<T, NS, ZC, BATCH, 1>(c, a, grid, s);
      c->launches++;
      return;
    }
  }
  launch_mode<T, NS, ZC, BATCH, 2>(c, a, grid, s);
  c->launches++;
}

// Launches per bucket (built with the list: the number of list entries inside
// the filter radii themselves, without the margin). Bucket 0 (at most 4) runs
// with register capacity 4. Bucket 1 (5 to 8) runs with capacity 8, on a side
// stream next to the main launch, when it holds over 5% of the atoms (e.g.
// SiC, where Si-Si second neighbours straddle the cutoff); otherwise it is
// appended to the capacity-4 launch. Every launch masks the stored short list
// (radius plus margin) by the cutoffs at each step; atoms with more entries
// inside than the capacity, and bucket 2, take the general path.
// Grid of a force launch: one thread per item, or (launch option) a number of
// waves of the blocks that fit on all SMs at once (resident blocks per SM from
// the kernel's launch bounds), the kernel looping over the items.
inline int force_grid(const Ctx* c, int zc, int evm) {
  const int full = (c->n + BLOCK - 1) / BLOCK;
  if (c->opt_waves <= 0 || c->n_sm <= 0) return full;
  // the blocks of this instance resident on one SM (its launch bound)
  const int resident = c->n_sm * fwd_min_blocks(zc <= 4 ? 4 : 8, zc <= 4 ? evm : 2,
                                                c->precision == TERSOFF_FP64);
  const int g = c->opt_waves * resident;
  return g < full ? g : full;
}

// The four-lane kernel takes the main launch when the launch option asks for
// it (tersoff_set_lanes(4), or the autotuner's choice) and the context is
// eligible (mixed path, one or two species, a single system). Automatic
// means one thread per atom: on the 512,000-atom Si benchmark the four-lane
// launch executes 43% more instructions at a 21% higher IPC and is slower.
template <class T, int NS, bool BATCH>
bool use_quad(const Ctx* c) {
  if (BATCH || sizeof(T) != 4 || NS < 1 || NS > 2 || comp_atom_sums(c) || c->n == 0) return false;
  return c->opt_quad == 1;
}

// The FP64 path's terms run one lane per bond (tersoff_lanes64.cuh) for tables
// inside the integer formats; other tables, and the ablation that sends every
// atom through Algorithm 2's loops, keep k_tersoff.
inline bool use_lanes64(const Ctx* c) { return c->fx_ok && !(c->ablate & TERSOFF_ABLATE_GENERAL); }

template <int NS, int W, bool BATCH, int EV, int LONG = 0>
void launch_lanes_ev(Ctx* c, const FwdArgs<double>& a, long long grid, cudaStream_t s) {
  const bool sym = c->sym_table;  // (false with a lambda3 term)
  void (*k)(FwdArgs<double>) = sym ? k_lanes64<NS, W, 3, BATCH, EV, LONG> : k_lanes64<NS, W, 1, BATCH, EV, LONG>;
  const size_t dyn = lanes_dyn(sym ? 3 : 1);
  const long long wave = (long long)(c->n_sm > 0 ? c->n_sm : 152) *
                         (sym ? lanes_blocks<NS, 3, BATCH, EV>() : lanes_blocks<NS, 1, BATCH, EV>());
  if (c->opt_waves > 0) grid = std::min(grid, c->opt_waves * wave);
  // with energy or virial sums one wave of looping blocks: each block adds its
  // totals to the accumulator once, and every such addition rounds at the
  // total's last place
  if (a.acc != nullptr) grid = std::min(grid, wave);
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
  launch_pdl(k, (int)grid, LBLOCK, dyn, s, a);
  c->launches++;
}
// items: about how many atoms the launch has (the device's counts decide; the
// kernel loops over what its grid does not cover)
template <int NS, int W, bool BATCH, int LONG>
void launch_lanes(Ctx* c, const FwdArgs<double>& a, long long items, cudaStream_t s) {
  constexpr int ATOMS = LBLOCK / W;
  const long long full = ((long long)c->n + ATOMS - 1) / ATOMS;
  long long grid = (items + ATOMS - 1) / ATOMS + (items < c->n ? 8 : 0);
  grid = std::max(1ll, std::min(grid, full));
  const int evm = ev_mode<double, BATCH>(a);
  if constexpr (W == 4 && !BATCH && !LONG) {
    if (evm == 0) return launch_lanes_ev<NS, W, BATCH, 0>(c, a, grid, s);
    if (evm == 1) return launch_lanes_ev<NS, W, BATCH, 1>(c, a, grid, s);
  }
  launch_lanes_ev<NS, W, BATCH, 2, LONG>(c, a, grid, s);
}

// LONG: boxes with a long edge, lanes only.
template <class T, int NS, bool BATCH = false, int LONG = 0>
void launch_buckets(Ctx* c, FwdArgs<T> a, cudaStream_t s) {
  constexpr bool D = sizeof(T) == 8;
  const bool lanes = LONG || (D && use_lanes64(c));
  if constexpr (!D) {
    if (use_quad<T, NS, BATCH>(c)) {
      TimedRegion tr(c, 0, s);
      const bool ev = a.acc != nullptr || a.eatom != nullptr;
      FwdArgs<T> aq = a;
      aq.identity = 1;
      launch_forward_quad(c, &aq, ev, s);
      // the atoms it left (more than four bonds inside the cutoffs, general
      // path): the per-thread kernel over the leftover list, one block per SM
      // looping over it; its last block zeroes the list's count
      FwdArgs<T> bl = a;
      bl.order = c->d_left;
      bl.n_items = c->d_flags + FLAG_LEFT;
      bl.order2 = bl.order3 = nullptr;
      bl.n_items2 = bl.n_items3 = nullptr;
      bl.identity = 0;
      bl.left_reset = 1;
      launch_t<T, NS, 8, BATCH>(c, bl, c->n_sm > 0 ? c->n_sm : 152, s);
      return;
    }
  }
  const int dec = bucket_decisions(c);
  const bool split1 = (dec & 1) != 0;
  const bool fork = split1 && c->side != nullptr;
  const bool wide = (dec & 2) != 0;
  // The wide launch runs next to the others, and starts first: it is one wave of
  // few warps, each a long serial chain (332 us of an evaluation of 2,097,152 SiC
  // atoms when it followed the main launch). Evaluation 1,211 -> 1,134 us; a
  // first evaluation of 197,432 atoms with its list build 613 -> 566 us.
  const bool fork2 = wide && c->side != nullptr && !lanes;
  cudaStream_t s2 = s, s3 = s;
  if (fork || fork2) cudaEventRecord(c->ev_fork, s);
  if (fork2) {
    cudaStreamWaitEvent(c->side2, c->ev_fork, 0);
    s3 = c->side2;
  }
  if (fork) {
    cudaStreamWaitEvent(c->side, c->ev_fork, 0);
    s2 = c->side;
  }
  if constexpr (!LONG) {
    if (wide && !lanes) launch_wide<T, NS, BATCH>(c, a, s3);
  }
  if (split1) {
    FwdArgs<T> b1 = a;
    b1.order = c->d_bucket + 1 * (size_t)c->n;
    b1.n_items = c->d_flags + flag_bucket(1);
    b1.order2 = b1.order3 = nullptr;
    b1.n_items2 = b1.n_items3 = nullptr;
    b1.identity = 0;
    if constexpr (D) {
      if (lanes) launch_lanes<NS, 8, BATCH, LONG>(c, b1, c->nbucket[1], s2);
    }
    if constexpr (!LONG) {
      if (!lanes) launch_t<T, NS, 8, BATCH>(c, b1, force_grid(c, 8, ev_mode<T, BATCH>(a)), s2);
    }
  }
  // bucket 0, then bucket 1 (unless split off), then bucket 2 (general path)
  FwdArgs<T> b0 = a;
  b0.order = c->d_bucket;
  b0.n_items = c->d_flags + flag_bucket(0);
  b0.order2 = split1 ? nullptr : c->d_bucket + 1 * (size_t)c->n;
  b0.n_items2 = split1 ? nullptr : c->d_flags + flag_bucket(1);
  b0.order3 = wide ? nullptr : c->d_bucket + 2 * (size_t)c->n;
  b0.n_items3 = wide ? nullptr : c->d_flags + flag_bucket(2);
  // all buckets in one launch: atoms in index order (spatial order, and no
  // indirection); atoms with longer lists take the masked or general path
  b0.identity = (split1 || wide) ? 0 : 1;
  {
    TimedRegion tr(c, 0, s);
    if constexpr (D) {
      if (lanes) {
        long long items = c->n;
        if (split1) items -= c->nbucket[1];
        if (wide) items -= c->nbucket[2];
        launch_lanes<NS, 4, BATCH, LONG>(c, b0, items, s);
        if (wide) {
          FwdArgs<T> b2 = a;
          b2.order = c->d_bucket + 2 * (size_t)c->n;
          b2.n_items = c->d_flags + flag_bucket(2);
          b2.identity = 0;
          launch_lanes<NS, 16, BATCH, LONG>(c, b2, c->nbucket[2], s);
        }
      }
    }
    if constexpr (!LONG) {
      if (!lanes) launch_t<T, NS, 4, BATCH>(c, b0, force_grid(c, 4, ev_mode<T, BATCH>(a)), s);
    }
    if (fork2) {
      cudaEventRecord(c->ev_join2, c->side2);
      cudaStreamWaitEvent(s, c->ev_join2, 0);
    }
  }
  if (fork) {
    cudaEventRecord(c->ev_join, c->side);
    cudaStreamWaitEvent(s, c->ev_join, 0);
  }
}

template <class T>
FwdArgs<T> make_args(Ctx* c, double* f, double* acc, double* eatom, bool virial = true) {
  FwdArgs<T> a;
  a.virial = virial ? 1 : 0;
  a.n = c->n;
  a.cap = c->cap;
  a.ns = c->ns;
  a.nbr = c->d_nbr;
  a.cnt = c->d_cnt;
  a.pos32 = c->d_pos32;
  a.posq = c->d_posq;
  a.rec = rec_ptr<T>(c);
  for (int q = 0; q < RSTRIDE; ++q) a.prm1[q] = rec_host<T>(c)[q];
  a.filt2 = c->d_filt32;
  set_pos64(c, a);
  if constexpr (sizeof(T) == 8) {
    if (c->fx_ok) a.fx1 = c->h_fx[0];
    a.fx = c->d_fx;
    a.cut_j = c->fx_cut_j ? 1 : 0;
  }
  a.near2 = c->d_near32;
  const double scale = ldexp(1.0, c->grid.fix_shift);
  for (int q = 0; q < 3; ++q) {
    a.h[q] = (float)c->grid.h[q];
    a.hq[q] = (int)llrint(c->grid.h[q] * scale);
  }
  a.qinv = ldexpf(1.0f, -c->grid.fix_shift);
  a.types = c->d_types;
  a.shortl = c->d_short;
  a.zcnt = c->d_zcnt;
  a.zs_cap = c->zs_cap;
  // ablation ABLATE_NO_SHORT: the stored short list is never valid
  a.dlim2 = (c->ablate & 1) ? -1.0f : (float)(0.25 * c->margin * c->margin);
  a.all_general = (c->ablate & 2) ? 1 : 0;
  a.f = f;
  a.contrib = c->d_contrib;
  a.rev = c->d_rev;
  a.kmask = c->d_kmask;
  a.atomic_mode = (c->scatter_atomic || comp_atom_sums(c)) ? 1 : 0;
  a.own = c->d_own;
  a.acc = acc;
  a.eatom = eatom;
  a.flags = c->d_flags;
  a.sys = c->d_sys;
  a.atom_sys = c->d_atom_sys;
  a.vatom = c->d_vatom;
  a.order = c->d_bucket;
  a.n_items = c->d_flags + flag_bucket(0);
  a.order2 = a.order3 = nullptr;
  a.n_items2 = a.n_items3 = nullptr;
  a.identity = 1;
  a.left = c->d_left;
  a.left_reset = 0;
  return a;
}

// Ablation TERSOFF_ABLATE_FASTFWD: the fast-forward lane scheme over the full
// skin list, one launch over all atoms in index order.
template <class T, int NS>
void launch_ffwd(Ctx* c, const FwdArgs<T>& a, cudaStream_t s) {
  const int grid = (c->n + BLOCK - 1) / BLOCK;
  TimedRegion tr(c, 0, s);
  if (c->has_lam3)
    k_tersoff_ffwd<T, NS, true><<<grid, BLOCK, 0, s>>>(a);
  else
    k_tersoff_ffwd<T, NS, false><<<grid, BLOCK, 0, s>>>(a);
  c->launches++;
}

// One translation unit per species count and path (fwd_f32.cu and the
// fwd_f64*.cu files) instantiates this.
template <class T, int NS>
int launch_species(Ctx* c, double* f, double* acc, double* eatom, cudaStream_t s, bool virial) {
  FwdArgs<T> a = make_args<T>(c, f, acc, eatom, virial);
  if (c->ablate & TERSOFF_ABLATE_FASTFWD)
    launch_ffwd<T, NS>(c, a, s);
  else
    launch_buckets<T, NS>(c, a, s);
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

// Batch of systems: the same bucketed launches as for one system (register
// capacity 4 for the atoms with at most 4 bonds inside the cutoffs, capacity
// 8 on the side stream for those with 5 to 8 when they are over 5%, the
// slot-cached wide kernel for the rest when they are over 0.5%), with
// per-system shifts and per-atom energy and virial for the per-system sums;
// runtime species count.
template <class T>
int launch_batch(Ctx* c, double* f, cudaStream_t s) {
  // energy and virial come from the per-atom stores: no block reduction
  FwdArgs<T> a = make_args<T>(c, f, nullptr, c->d_eatom);
  if (c->n > 0) launch_buckets<T, 0, true>(c, a, s);
  TGB_CUDA(c, cudaGetLastError());
  return TERSOFF_OK;
}

}  // namespace fwd
}  // namespace tgb
