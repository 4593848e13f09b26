// Velocity-Verlet steps of small systems in one resident kernel.
//
// Bound: latency. A step of a few hundred to some ten thousand atoms is two
// short dependent passes (kick, drift and pack; forces); as graph nodes they
// cost a launch each, and with displacement-triggered rebuilds a decision
// kernel and a conditional node more: 23 us per step at 216 atoms, 28 at
// 32,000, against 13.5 and 21.1 here (100 steps with energies at 1000 K, their
// rebuilds included; 8.5 and 12.8 on steps without either). Here the blocks stay
// on the chip, one atom per thread, and a barrier over the grid separates the
// passes. The kernel returns at the step
// whose rebuild is due (a displacement beyond half the skin, or the fixed
// period); the host enqueues the build and the rest.
//
// The arithmetic is that of k_step and k_tersoff (the same device functions);
// positions change while the kernel runs, so they are read past the read-only
// cache (Shift KIND 2).
//
// The barrier. Up to 16 blocks (2,048 atoms) form one cluster and use its
// hardware barrier. More blocks count arrivals in global memory: the launch is
// cooperative (all blocks are on the chip), every wait is bounded, and a wait
// that runs out raises FLAG_MD_TIMEOUT and ends the kernel (the other blocks'
// waits then run out too); the host restores the call's start and runs its steps
// by launches.
#include "step.cuh"
#include "tersoff_fwd.cuh"

namespace tgb {

fwd::FwdArgs<float> resident_args(Ctx* c);  // fwd_f32.cu

namespace {

using fwd::BLOCK;

struct ResidentArgs {
  double *x, *v;
  const double* f;
  double dt;
  int s0, s1;    // steps s0 .. s1 - 1 in full
  int resume;    // step s0 has been drifted (its rebuild follows): forces first
  int tail;      // then drift step s1 without packing (a rebuild follows)
  int on_skin;   // stop before the forces of a step with displacement^2 > lim2
  float lim2;
  double* rows;  // thermo accumulation rows or null
  double* snap;  // receives the state that step 0 starts from
  int* flags;
  int polls;  // of a wait before it gives up
};

// Barrier over the blocks of the one cluster, and the same words.
__device__ __forceinline__ void cluster_barrier(const int* flags, int* words) {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (threadIdx.x < 2) words[threadIdx.x] = *(const volatile int*)(flags + (threadIdx.x == 0 ? FLAG_DMAX : FLAG_REV_MISS));
  __syncthreads();
}

// Barrier over the grid; then the words every block needs: the running
// displacement and whether a short-list entry lacks its reverse. False: a wait
// ran out.
__device__ __forceinline__ bool grid_barrier(int* flags, unsigned target, int polls, int* words) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    int* bar = flags + FLAG_MD_BAR;
    atomicAdd(bar, 1);
    int spins = 0;
    unsigned have;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(have) : "l"(bar) : "memory");
    } while ((int)(have - target) < 0 && ++spins < polls);
    const bool ok = (int)(have - target) >= 0;
    if (!ok) atomicExch(flags + FLAG_MD_TIMEOUT, 1);
    __threadfence();
    words[0] = *(volatile int*)(flags + FLAG_DMAX);
    words[1] = *(volatile int*)(flags + FLAG_REV_MISS);
    words[2] = ok ? 1 : 0;
  }
  __syncthreads();
  return words[2] != 0;
}

template <int NS, int MODE, int EV, bool CLUSTER>
__global__ void __launch_bounds__(BLOCK, 6)
    k_md_resident(const __grid_constant__ fwd::FwdArgs<float> a, const __grid_constant__ PackArgs pk,
                  const __grid_constant__ GatherArgs ga, const __grid_constant__ Coef cf,
                  const __grid_constant__ ResidentArgs r) {
  constexpr int SNS = NS > 1 ? NS : (NS == 1 ? 1 : TERSOFF_MAX_SPECIES);
  constexpr int SREC = NS == 1 ? 1 : SNS * SNS * SNS * RSTRIDE;
  __shared__ float srec_s[SREC], sfilt[SNS * SNS], snear[SNS * SNS];
  __shared__ int words[3];
  __shared__ float2 tsum[7][BLOCK];
  const int ns = NS > 0 ? NS : a.ns;
  if (NS != 1)
    for (int q = threadIdx.x; q < ns * ns * ns * RSTRIDE; q += BLOCK) srec_s[q] = a.rec[q];
  if (threadIdx.x < ns * ns) {
    sfilt[threadIdx.x] = a.filt2[threadIdx.x];
    snear[threadIdx.x] = a.near2[threadIdx.x];
  }
  // a wait of an earlier launch of the call gave up: its steps will be run again
  // (step 0's launch goes on in any case: it writes the snapshot)
  if (!CLUSTER && r.s0 > 0 && *(const volatile int*)(r.flags + FLAG_MD_TIMEOUT)) return;
  if (threadIdx.x == 0) {
    words[0] = r.flags[FLAG_DMAX];
    words[1] = r.flags[FLAG_REV_MISS];
  }
  __syncthreads();
  fwd::ItemEnv<float> v{NS == 1 ? a.prm1 : srec_s, sfilt, snear, ns, 0, 0, a.n, true, true, EV >= 1,
                        &tsum[0][threadIdx.x]};
  const int i = blockIdx.x * BLOCK + threadIdx.x;
  const bool first = blockIdx.x == 0 && threadIdx.x == 0;
  unsigned target = 0;
  int s = r.s0;
  for (;; ++s) {
    if (!(r.resume && s == r.s0)) {
      if (s == r.s1 && !r.tail) break;
      const int pack = s < r.s1;
      float d2 = 0.0f, kef = 0.0f;
      double ke = 0.0;
      if (i < a.n) {
        if (s == 0)
          step_atom<false>(pk, ga, 0, r.x, r.v, r.f, cf, r.dt, 1, pack, false, r.snap, i, d2, ke, kef);
        else
          step_atom<true>(pk, ga, 1, r.x, r.v, r.f, cf, r.dt, 2, pack, EV >= 1, nullptr, i, d2, ke, kef);
      }
      if (pack) track_max(pk, d2);
      if (EV >= 1 && s > 0)  // of step s - 1
        block_sum_add_f(kef, r.rows + ACC_LEN * (size_t)(s - 1) + 7 * ACC_STRIDE);
      if (!pack) break;  // the rebuild's kernels follow
      target += gridDim.x;
      if (CLUSTER)
        cluster_barrier(r.flags, words);
      else if (!grid_barrier(r.flags, target, r.polls, words))
        return;
    }
    const float dmax2 = __int_as_float(words[0]);
    if (r.on_skin && dmax2 > r.lim2) {
      if (first) r.flags[FLAG_MD_HALT] = 1;
      break;
    }
    v.use_short = dmax2 <= a.dlim2;
    v.slots = v.use_short && words[1] == 0;
    if (first) r.flags[FLAG_EXTRA] = v.slots ? 0 : 1;
    if (EV >= 1)
      for (int q = 0; q < 7; ++q) fwd::sum_zero(tsum[q][threadIdx.x]);
    fwd::force_items<float, NS, 4, MODE, 2, false, EV>(a, v, i, gridDim.x * BLOCK);
    if (EV >= 1) {
      __syncthreads();
      fwd::block_reduce_sums(&tsum[0][threadIdx.x], r.rows + ACC_LEN * (size_t)s);
    }
    target += gridDim.x;
    if (CLUSTER)
      cluster_barrier(r.flags, words);
    else if (!grid_barrier(r.flags, target, r.polls, words))
      return;
  }
  if (first) r.flags[FLAG_MD_STEP] = s;
}

template <int NS, int EV, bool CL> void* kernel_of(const Ctx* c) {
  return c->has_lam3    ? (void*)k_md_resident<NS, 1, EV, CL>
         : c->sym_table ? (void*)k_md_resident<NS, 2, EV, CL>
                        : (void*)k_md_resident<NS, 0, EV, CL>;
}
template <int EV, bool CL> void* kernel_ns(const Ctx* c) {
  return c->ns == 1 ? kernel_of<1, EV, CL>(c) : c->ns == 2 ? kernel_of<2, EV, CL>(c) : kernel_of<0, EV, CL>(c);
}
int blocks_of(const Ctx* c) { return (c->n + BLOCK - 1) / BLOCK; }
bool one_cluster(const Ctx* c) { return blocks_of(c) <= 16; }
void* kernel(const Ctx* c, bool rows) {
  return one_cluster(c) ? (rows ? kernel_ns<1, true>(c) : kernel_ns<0, true>(c))
                        : (rows ? kernel_ns<1, false>(c) : kernel_ns<0, false>(c));
}
// the launch: one cluster of all blocks, or a cooperative grid
struct Config {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1] = {};
  Config(const Ctx* c, cudaStream_t s) {
    cfg.gridDim = dim3(blocks_of(c));
    cfg.blockDim = dim3(BLOCK);
    cfg.stream = s;
    if (one_cluster(c)) {
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cfg.gridDim.x;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    } else {
      at[0].id = cudaLaunchAttributeCooperative;
      at[0].val.cooperative = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

}  // namespace

// The mixed path's gathered forces in the one launch per step that small
// systems take (no bucket on a kernel of its own), up to the sizes given with
// RESIDENT_MAX_ATOMS.
bool resident_fits(Ctx* c, bool whole, bool rows) {
  if (c->precision != TERSOFF_MIXED || c->n_sys > 0 || c->scatter_atomic || c->ablate || c->opt_quad == 1 ||
      c->opt_waves > 0 || c->n_sm <= 0 || c->n > RESIDENT_MAX_ATOMS ||
      (whole && !one_cluster(c)) || bucket_decisions(c) != 0)
    return false;
  void* k = kernel(c, rows);
  if (one_cluster(c)) {
    Config g(c, nullptr);
    int fit = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, k, &g.cfg) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return fit >= 1;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, BLOCK, 0) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (long long)blocks_of(c) <= (long long)per_sm * c->n_sm;
}

int launch_resident(Ctx* c, double* x, double* v, const double* f, double dt, int s0, int s1, bool resume, bool tail,
                    bool on_skin, float lim2, double* rows, double* snap, cudaStream_t s) {
  fwd::FwdArgs<float> a = resident_args(c);
  PackArgs pk = make_pack(c, true);
  GatherArgs ga = make_gather(c);
  Coef cf = c->coef;
  ResidentArgs r{x, v, f, dt, s0, s1, resume, tail, on_skin, lim2, rows, snap, c->d_flags, c->md_wait};
  TGB_CUDA(c, cudaMemsetAsync(c->d_flags + FLAG_MD_HALT, 0, sizeof(int) * 2 * FLAG_STRIDE, s));  // and the barrier
  void* args[] = {&a, &pk, &ga, &cf, &r};
  Config g(c, s);
  TGB_CUDA(c, cudaLaunchKernelExC(&g.cfg, kernel(c, rows != nullptr), args));
  c->launches++;
  return TERSOFF_OK;
}

}  // namespace tgb
