// Temporally blocked step with one site per thread: many steps per launch.
//
// A block holds one or more pieces (Piece, thread t0 + j holds the piece's site j): whole
// lattices (rings), or stretches of longer ones with c_max ksteps halo sites on each side.
// Every thread keeps its site's Q populations in registers.  One step: collide, write the
// Q - 1 moving planes to the exchange area in shared memory (double-buffered by step
// parity), one block barrier, read plane i from the thread holding site x - c_i of the
// piece (its ends wrap: the periodic ring, or for a stretch values that travel c_max sites
// per step and stop short of the stored middle).
//
// Lattices with reservoir ends: the piece's nodes may include the fixed ones (j <= 0,
// j >= N - 1 and c_max ghosts beyond each end).  They collide the values they hold and
// then hold f^eq of the end's density, so from the third step on their exchange values,
// in both parities, do not change.
//
// When and why.  FP64 storage by default (also with reservoir ends): the fixed-point
// collision needs many warps to hide its latencies, which the register-resident kernel's
// several sites per thread leave no registers for (8 warps an SM against 24 here), and a
// single lattice is spread over the SMs instead of sitting on one or two.  FP32 storage
// when the batch is too small to give every SM a full register-resident block
// (choose_blocked in lbks_plan.h, setup_blocked): one 4096-site lattice takes 0.18 us per
// step in stretches over 64 SMs against 0.88 us in one block, 2^18 sites 0.88 against
// 1.12 us; 2^20 sites 3.1 against 2.2 us, so large FP32 batches stay register-resident.
// Not for scaled FP16, whose results depend on where launches end (rounded there).
// Per step and stretch: the halos cost 2 c_max k of NT sites, a launch 1.5 to 2 us in all.
// Measured (GB300): one 4096-site D1Q7 FP64 lattice 16.8 -> 0.87 us per step (stretches of
// 32 sites, 16 steps per launch; bound by the latency of one warp's collision), the
// 4096-lattice FP64 ensemble 615 -> 253 us per step, 3.7e10 site-updates/s (128 threads, 2
// steps per launch; bound by the integer pipe, 65 % busy), 122 front lattices 9.8 -> 2.2 us per
// step (over clusters), 24 FP32 lattices 0.87 -> 0.37 us per step.
#include "lbks_collapse.cuh"
#include "lbks_device.cuh"
#include "lbks_plan.h"

namespace lbks {

namespace {

using plan::kBlockedPieces;

// The next launch's blocks may be scheduled from this many steps before the end.  Earlier,
// they fill the SMs' free slots around the running blocks, unevenly (an SM with fewer of
// these gets more of those, up to five instead of four on a batch of 3.6 blocks an SM:
// 3.4 instead of 2.4 us per step); at the last step, a small batch waits for the launch.
constexpr int kNextGrid = 2;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void store_cluster(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// NTM: the most threads a block of this instance has.
template <int Q, int ST, int NTM> struct BlockedCfg {
  // Row of the exchange area, a compile-time stride: a column per thread.  FP64: and, for
  // each piece, c_max on either side of its own, where the threads at the piece's other end
  // put the values that wrap, so that every access is one address plus an immediate and no
  // registers are held for the neighbours.  FP32 has the registers: the six neighbours'
  // columns are computed once, which takes fewer instructions per step.
  static constexpr bool kGuard = ST == kF64;
  static constexpr int kXS = NTM + (kGuard ? 2 * cmax_of(Q) * kBlockedPieces : 0);
};

// ONE: every bundle holds one piece.  MINB: blocks an SM has to hold, which sets the
// register budget: 80 in FP64 (24 warps), 64 in FP32 where SMs are to be filled; FP64 batches
// of at most a block per SM take what the compiler wants instead (about 126), which shortens the
// one warp per scheduler's chain by 4 to 6 %.  Where a block holds several runs, their fixed-point
// constants lie in shared memory and are read every step: in registers (uniform ones where the
// block has one run) they were spilled, 152 bytes a thread (122 front lattices 2.70 -> 2.44 us
// per step).
// CLU: the blocks of a cluster hold lattices together (plan_clusters), without halos: a portion's
// edge values are also stored into the guard columns of the block that holds its neighbour
// (st.shared::cluster; the portion itself where a lattice lies in one block), and the step's barrier is
// the cluster's.  For FP64 batches with lattices longer than a block: their stretches cost up
// to two thirds more sites in halos, and launches that end block by block every 4 to 16
// steps.  The cluster barrier adds 0.25 us to a step's latency (1.13 against 0.87 us with one
// block an SM), which other blocks of the SM cover; 122 front lattices 2.83 -> 2.24 us per
// step, single lattices stay in stretches.
template <int Q, int ST, int NTM, int MINB, bool RES, bool ONE, bool CLU = false>
__global__ void __launch_bounds__(NTM, MINB)
    blocked_step_kernel(Arena src, Arena dst, const RunDesc* __restrict__ runs, const Piece* __restrict__ pieces,
                        const int2* __restrict__ bundles, int ksteps) {
  using T = typename StorageType<ST>::type;
  using CT = typename StorageType<ST>::compute;
  constexpr int C = cmax_of(Q), XS = BlockedCfg<Q, ST, NTM>::kXS;
  constexpr bool kGuard = BlockedCfg<Q, ST, NTM>::kGuard;
  __shared__ CT ex[2][Q - 1][XS];  // [step parity][plane i - 1]
  // (the pieces are written once, before any launch)
  const int t = threadIdx.x;
  int p = blockIdx.x, q = 0;
  if constexpr (!ONE) {
    const int2 bd = bundles[blockIdx.x];
    p = bd.x;
    for (int u = 1; u < bd.y; ++u)
      if (t >= pieces[bd.x + u].t0) q = u;
    p += q;
  }
  const Piece pc = pieces[p];
  const int n = pc.n, j = t - pc.t0;
  const bool active = j < n && (!CLU || bundles[blockIdx.x].y > 0);
  wait_prior_grid();
  const RunDesc& d = runs[pc.run];
  int x = (int)pc.x0 + j;  // run-local site (N <= 2^30)
  bool fixed = false;
  if constexpr (RES) fixed = x <= 0 || x >= (int)d.N - 1;
  else if (x >= (int)d.N) x -= (int)d.N;
  CT g[Q];
  if (active) {
    const T* fs = static_cast<const T*>(src.f) + d.off + x;
#pragma unroll
    for (int i = 0; i < Q; ++i, fs += src.plane) g[i] = *fs;
  }
  const Coef<CT, Q> k = load_coef<CT, Q>(d);
  __shared__ FixCoef held[(ST == kF64 && !ONE) ? kBlockedPieces : 1];
  if constexpr (ST == kF64 && !ONE) {
    if (j == 0) held[q] = d.fix;
    __syncthreads();
  }
  CT* const own = &ex[0][0][t + (kGuard ? C * (2 * q + 1) : 0)];
  int from[Q];  // plane i's new value: the column of the thread holding x - c_i, less this one's
#pragma unroll
  for (int i = 1; i < Q; ++i) {
    const int c = (i + 1) / 2;
    from[i] = (i & 1) ? (j >= c ? -c : n - c) : (j + c < n ? c : c - n);
  }
  uint32_t edge = 0;  // where this thread's values that leave the portion go, in the cluster's shared memory
  if constexpr (CLU) {
    const bool right = j >= n - C;
    const int to = right ? pc.pad_ : pc.halo;
    edge = map_to_rank(smem_addr(&ex[0][0][(to & 0xffff) + (right ? j - n : j)]), (uint32_t)to >> 16);
    cluster_barrier();  // every block runs before another writes into it
  }
  for (int s = 0; s < ksteps; ++s) {
    if (s == ksteps - kNextGrid || (s == 0 && ksteps < kNextGrid)) allow_next_grid();
    CT* const xs = own + (s & 1) * (Q - 1) * XS;
    if (active && (!RES || !fixed || s < 3)) {
      if constexpr (ST == kF64) collide<Q>(g, ONE ? k.fix : held[q], &d);
      else collide<Q>(g, k);
#pragma unroll
      for (int i = 1; i < Q; ++i) {
        const int c = (i + 1) / 2;
        CT* const w = xs + (i - 1) * XS;
        *w = g[i];
        // the last c sites' right-moving values enter at the piece's start, and so on
        if (kGuard && ((i & 1) ? j >= n - c : j < c)) {
          if constexpr (CLU)
            store_cluster(edge + (uint32_t)((((s & 1) * (Q - 1) + i - 1) * XS) * sizeof(CT)), g[i]);
          else
            w[(i & 1) ? -n : n] = g[i];
        }
      }
      if constexpr (RES) {
        if (fixed) {
          const double rb = x <= 0 ? d.rho_left : d.rho_right;
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            double v = __fma_rn(d.B[i], __dmul_rn(rb, rb), __dmul_rn(d.A[i], rb));
            if (i == 0) v = __dsub_rn(v, d.rhobar);
            g[i] = static_cast<CT>(v);
          }
        }
      }
    }
    // (double-buffered: a block writes parity s again only after all have passed s + 1's)
    if constexpr (CLU) cluster_barrier();
    else __syncthreads();
    if (active && !fixed) {
#pragma unroll
      for (int i = 1; i < Q; ++i) g[i] = xs[(i - 1) * XS + (kGuard ? -speed(i) : from[i])];
    }
  }
  if (active && j >= pc.st_lo && j < pc.st_hi) {
    T* fd = static_cast<T*>(dst.f) + d.off + x;
#pragma unroll
    for (int i = 0; i < Q; ++i, fd += dst.plane) *fd = g[i];
  }
}

// The tau = 1 collapse in the same form: one value per thread, its 2 c_max neighbours read
// from the exchange area each step (with the guard columns for wrapping ends).  FP64
// storage, FP32 batches too small for the register-resident collapse, and reservoir ends
// (the fixed nodes keep their values, put in both parities once).  Z: the operations that
// add zero are left out (collapse_site's ZB, and ZR in FP64).  FP64 is bound by the
// FP64 pipe, so what counts is to use every SM's: one 4096-site lattice 25 -> 1.0 us per
// step (0.85 with Z), 24 lattices 25 -> 3.9 (2.9), the 4096-lattice ensemble 442 -> 418 (303);
// FP32, 24 lattices: 1.02 -> 0.34 us (0.31), one lattice 0.57 -> 0.20 (300 lattices: 1.03
// either way, so larger batches stay register-resident).
template <int C, int ST, bool RES, bool ONE, bool Z>
__global__ void __launch_bounds__(512, 2)
    blocked_collapse_kernel(Arena src, Arena dst, const RunDesc* __restrict__ runs, const Piece* __restrict__ pieces,
                            const int2* __restrict__ bundles, int ksteps) {
  using T = typename StorageType<ST>::type;
  using CT = typename StorageType<ST>::compute;
  constexpr int XS = 512 + 2 * C * kBlockedPieces;
  __shared__ CT ex[2][XS];
  const int t = threadIdx.x;
  int p = blockIdx.x, q = 0;
  if constexpr (!ONE) {
    const int2 bd = bundles[blockIdx.x];
    p = bd.x;
    for (int u = 1; u < bd.y; ++u)
      if (t >= pieces[bd.x + u].t0) q = u;
    p += q;
  }
  const Piece pc = pieces[p];
  const int n = pc.n, j = t - pc.t0;
  const bool active = j < n;
  wait_prior_grid();
  const RunDesc& d = runs[pc.run];
  int x = (int)pc.x0 + j;
  bool fixed = false;
  if constexpr (RES) fixed = x <= 0 || x >= (int)d.N - 1;
  else if (x >= (int)d.N) x -= (int)d.N;
  CT v = CT(0);
  if (active) v = static_cast<CT>(static_cast<const T*>(src.f)[d.off + x]);
  const CollapseCoef<CT, C> k = load_collapse_coef<CT, C>(d);
  CT* const own = &ex[0][t + C * (2 * q + 1)];
  const bool last = j >= n - C, first = j < C;  // these also enter at the other end
  for (int s = 0; s < ksteps; ++s) {
    if (s == ksteps - kNextGrid || (s == 0 && ksteps < kNextGrid)) allow_next_grid();
    CT* const xs = own + (s & 1) * XS;
    if (active && (!RES || !fixed || s < 2)) {
      *xs = v;
      if (last) xs[-n] = v;
      if (first) xs[n] = v;
    }
    __syncthreads();
    if (active && !fixed) {
      CT dl[C + 1], dr[C + 1];
      dl[0] = dr[0] = CT(0);
#pragma unroll
      for (int c = 1; c <= C; ++c) {
        dl[c] = xs[-c];
        dr[c] = xs[c];
      }
      v = collapse_site<CT, C, Z, Z && ST == kF64>(v, dl, dr, k);
    }
  }
  if (active && !fixed && j >= pc.st_lo && j < pc.st_hi) static_cast<T*>(dst.f)[d.off + x] = static_cast<T>(v);
}

template <int Q, int ST, bool RES, int NTM>
cudaError_t launch_n(const ResidentLaunch& L, cudaStream_t s) {
  constexpr int MINB = (ST == kF64 ? 768 : 1024) / NTM;
  if (L.one)
    return launch_early(blocked_step_kernel<Q, ST, NTM, MINB, RES, true>, L.nbundles, L.NT, 0, s, L.src, L.dst, L.runs,
                        L.pieces, L.bundles, L.ksteps);
  return launch_early(blocked_step_kernel<Q, ST, NTM, MINB, RES, false>, L.nbundles, L.NT, 0, s, L.src, L.dst, L.runs,
                      L.pieces, L.bundles, L.ksteps);
}

// The exchange area is sized by the instance, and FP64's would otherwise bound the blocks
// per SM: 128 threads (21 KB), 256 (34 KB) and 384 (46 KB).
template <int Q, int ST, bool RES>
cudaError_t launch_t(const ResidentLaunch& L, cudaStream_t s) {
  if constexpr (ST == kF64) {
    if (L.NT <= 128 && L.one && L.spread)
      return launch_early(blocked_step_kernel<Q, ST, 128, 1, RES, true>, L.nbundles, L.NT, 0, s, L.src, L.dst, L.runs,
                          L.pieces, L.bundles, L.ksteps);
    if (L.NT <= 128) return launch_n<Q, ST, RES, 128>(L, s);
    if (L.NT <= 256) return launch_n<Q, ST, RES, 256>(L, s);
    return launch_n<Q, ST, RES, 384>(L, s);
  } else {
    return launch_n<Q, ST, RES, 512>(L, s);
  }
}

template <int Q, bool RES, int NTM>
cudaError_t launch_cluster_n(const ResidentLaunch& L, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)L.nbundles);
  cfg.blockDim = dim3((unsigned)L.NT);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)L.cl;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, blocked_step_kernel<Q, kF64, NTM, 768 / NTM, RES, false, true>, L.src, L.dst, L.runs,
                            L.pieces, L.bundles, L.ksteps);
}

template <int Q, bool RES>
cudaError_t launch_cluster_t(const ResidentLaunch& L, cudaStream_t s) {
  if (L.storage != kF64 || L.one || L.nbundles % L.cl || L.cl > 8 || L.NT > 384) return cudaErrorInvalidValue;
  if (L.NT <= 128) return launch_cluster_n<Q, RES, 128>(L, s);
  if (L.NT <= 256) return launch_cluster_n<Q, RES, 256>(L, s);
  return launch_cluster_n<Q, RES, 384>(L, s);
}

template <int Q, int ST, bool RES, bool Z>
cudaError_t launch_collapse_z(const ResidentLaunch& L, cudaStream_t s) {
  constexpr int C = cmax_of(Q);
  if (L.one)
    return launch_early(blocked_collapse_kernel<C, ST, RES, true, Z>, L.nbundles, L.NT, 0, s, L.src, L.dst, L.runs,
                        L.pieces, L.bundles, L.ksteps);
  return launch_early(blocked_collapse_kernel<C, ST, RES, false, Z>, L.nbundles, L.NT, 0, s, L.src, L.dst, L.runs,
                      L.pieces, L.bundles, L.ksteps);
}

template <int Q, int ST, bool RES>
cudaError_t launch_collapse_t(const ResidentLaunch& L, cudaStream_t s) {
  return L.zb ? launch_collapse_z<Q, ST, RES, true>(L, s) : launch_collapse_z<Q, ST, RES, false>(L, s);
}

#define LBKS_BLOCKED_DISPATCH(OP)                                                    \
  do {                                                                               \
    if (Q == 5 && storage == kF64) { constexpr int Qc = 5, STc = kF64; OP; }         \
    if (Q == 5 && storage == kF32) { constexpr int Qc = 5, STc = kF32; OP; }         \
    if (Q == 7 && storage == kF64) { constexpr int Qc = 7, STc = kF64; OP; }         \
    if (Q == 7 && storage == kF32) { constexpr int Qc = 7, STc = kF32; OP; }         \
  } while (0)

}  // namespace

bool blocked_supported(int Q, int storage, int NT) {
  return (Q == 5 || Q == 7) && (storage == kF64 || storage == kF32) && NT >= 32 && NT <= 512 && NT % 32 == 0;
}

cudaError_t launch_blocked(const ResidentLaunch& L, bool reservoir, cudaStream_t s) {
  const int Q = L.Q, storage = L.storage;
  if (!blocked_supported(Q, storage, L.NT)) return cudaErrorInvalidValue;
  if (L.nbundles == 0) return cudaSuccess;
  if (L.collapse) {
    if (reservoir) LBKS_BLOCKED_DISPATCH(return (launch_collapse_t<Qc, STc, true>(L, s)));
    else LBKS_BLOCKED_DISPATCH(return (launch_collapse_t<Qc, STc, false>(L, s)));
    return cudaErrorInvalidValue;
  }
  if (L.NT > (storage == kF64 ? 384 : 512)) return cudaErrorInvalidValue;
  if (L.cl > 1) {
    if (Q == 5) return reservoir ? launch_cluster_t<5, true>(L, s) : launch_cluster_t<5, false>(L, s);
    return reservoir ? launch_cluster_t<7, true>(L, s) : launch_cluster_t<7, false>(L, s);
  }
  if (reservoir) LBKS_BLOCKED_DISPATCH(return (launch_t<Qc, STc, true>(L, s)));
  else LBKS_BLOCKED_DISPATCH(return (launch_t<Qc, STc, false>(L, s)));
  return cudaErrorInvalidValue;
}

}  // namespace lbks
