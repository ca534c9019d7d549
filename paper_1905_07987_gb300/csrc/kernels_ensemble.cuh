// Ensembles of uneven elastic grids advanced together: one persistent launch per phase of the step for
// all runs.  The work of the runs is concatenated (the predictor's blocks of cells, the corrector's cells, faces of
// one direction for the Riemann solver); each work item finds its run by binary search in the
// prefix offsets of the run table and is processed by the same device function as in the
// per-context kernels, with that run's step arguments (from device memory).  Blocks and warps
// loop over the concatenated items (grid sized by the SM count), so small runs share the GPU with
// large ones inside one launch.  No block waits for another.
#pragma once
#include "kernels.cuh"
#include "kernels_ck_fx.cuh"
#include "step_scalars.cuh"

namespace ader {

// Largest r with off[r] <= item (off[0] = 0, off[nr] = total, item < total).
__device__ __forceinline__ int ens_find(const long long* off, int nr, long long item) {
  int lo = 0, hi = nr - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= item) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

template <int N, bool MIXED, bool PIC>
struct EnsCfg {
  static constexpr int TPB = MIXED ? CfgEM<N, PIC>::TPB : CfgE<N>::TPB;
  static constexpr int MINB = MIXED ? CfgEM<N, PIC>::MINB : CfgE<N>::MINB;
  static constexpr int CPB = MIXED ? CfgEM<N, PIC>::CPB : CfgE<N>::CPB;
  static constexpr size_t SMEM = MIXED ? CfgEM<N, PIC>::SMEM : CfgE<N>::SMEM;
  static_assert(CPB == ck_cells_per_block(N), "the host counts the blocks of each run");
};

// The it-th predictor block of all runs (PIC: Picard predictor, otherwise Cauchy-Kowalevski).
template <int N, bool MIXED, bool PIC>
__device__ __forceinline__ void ens_predictor_block(const StepArgs* R, const EnsTable& E,
                                                    const Tables& T, const TablesF& F,
                                                    long long it) {
  const int r = ens_find(E.blk0, E.nr, it);
  const long long c0 = (it - E.blk0[r]) * EnsCfg<N, MIXED, PIC>::CPB;
  if constexpr (MIXED) predictor_elastic_mixed_block<N, PIC>(R[r], T, F, c0);
  else predictor_elastic_block<N, PIC>(R[r], T, F.el, c0);
  __syncthreads();  // the next block of cells reuses the shared memory
}

template <int N, bool MIXED, bool PIC>
__global__ void __launch_bounds__(EnsCfg<N, MIXED, PIC>::TPB, EnsCfg<N, MIXED, PIC>::MINB)
    k_ens_predictor(const StepArgs* __restrict__ R, const __grid_constant__ EnsTable E,
                    const __grid_constant__ Tables T, const __grid_constant__ TablesF F) {
  const long long total = E.blk0[E.nr];
  for (long long it = blockIdx.x; it < total; it += gridDim.x)
    ens_predictor_block<N, MIXED, PIC>(R, E, T, F, it);
}

template <class P, int D, int N>
__global__ void __launch_bounds__(128) k_ens_riemann(const StepArgs* __restrict__ R,
                                                     const __grid_constant__ EnsTable E,
                                                     const __grid_constant__ Tables T, int d) {
  const long long total = E.face0[d][E.nr];
  const int lane = threadIdx.x & 31;
  for (long long w = (long long)blockIdx.x * 4 + (threadIdx.x >> 5); w < total;
       w += (long long)gridDim.x * 4) {
    const int r = ens_find(E.face0[d], E.nr, w);  // the same for the whole warp
    riemann_face<P, D, N>(R[r], T, d, E.phioff[d][r], w - E.face0[d][r], lane);
  }
}

// The corrector of all runs in groups of CPB concatenated cells, as the per-context kernel's blocks; a
// group that spans runs is taken run by run.  A run's weights are formed when a block comes to it.
// (One cell at a time left half to seven eighths of the threads idle at orders 1 to 4.)
template <int N, int CPB, int NT>
__device__ __forceinline__ void ens_corrector(const StepArgs* R, const EnsTable& E,
                                              SmemC<Elastic, 3, N, CPB>& S) {
  const long long total = E.cell0[E.nr];
  int run = -1, Ew = 0;
  for (long long b = (long long)blockIdx.x * CPB; b < total; b += (long long)gridDim.x * CPB) {
    const long long end = b + CPB < total ? b + CPB : total;
    for (long long c = b; c < end;) {
      const int r = ens_find(E.cell0, E.nr, c);
      const long long e = CPB == 1 || E.cell0[r + 1] > end ? end : E.cell0[r + 1];
      // (with groups of one cell keeping the weights gains nothing)
      if (CPB == 1 || r != run) Ew = corrector_weights<3, N + 1>(R[r], S.w, threadIdx.x);
      run = r;
      corrector_cells<Elastic, 3, N, CPB, NT>(R[r], S, Ew, E.phioff[1][r], E.phioff[2][r],
                                              c - E.cell0[r], (int)(e - c), threadIdx.x);
      c = e;
    }
  }
}

template <int N>
__global__ void __launch_bounds__(CfgC<Elastic, 3, N>::TPB)
    k_ens_corrector(const StepArgs* __restrict__ R, const __grid_constant__ EnsTable E) {
  using X = CfgC<Elastic, 3, N>;
  __shared__ SmemC<Elastic, 3, N, X::CPB> S;
  ens_corrector<N, X::CPB, X::TPB>(R, E, S);
}

// One step of every run: dt, predictor (`blocks` of them), Riemann per direction, corrector, time
// advance.
template <int N, bool MIXED, bool PIC>
cudaError_t ens_step_n(const StepArgs* R, const EnsTable& E, const Tables& T, const TablesF& F,
                       long long blocks, cudaStream_t s) {
  using G = EnsCfg<N, MIXED, PIC>;
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(k_ens_predictor<N, MIXED, PIC>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)G::SMEM);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
  cudaError_t e = launch_ens_dt(R, E.nr, s);
  if (e != cudaSuccess) return e;
  k_ens_predictor<N, MIXED, PIC><<<(unsigned)blocks, G::TPB, G::SMEM, s>>>(R, E, T, F);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  for (int d = 0; d < 3; ++d) {
    k_ens_riemann<Elastic, 3, N><<<152 * 16, 128, 0, s>>>(R, E, T, d);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  k_ens_corrector<N><<<152 * 8, CfgC<Elastic, 3, N>::TPB, 0, s>>>(R, E);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return launch_ens_advance(R, E.nr, s);
}

}  // namespace ader

namespace ader {

// ---- one persistent launch for whole steps ----------------------------------------------------
// Grid-wide barrier of a cooperative launch (every block resident): blocks arrive on a counter,
// the last one resets it and advances the generation; the others poll the generation at most
// `limit` times.  A wait that runs out returns false (the caller latches ST_TIMEOUT and leaves);
// the other blocks then run out at the same barrier, so no block waits forever.  The state is
// zeroed by the host before every launch.
struct GridBar {
  unsigned count;
  unsigned gen;
};

__device__ __forceinline__ bool grid_sync(GridBar* b, unsigned nblocks, long long limit) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    volatile unsigned* vg = &b->gen;
    const unsigned g = *vg;
    __threadfence();
    if (atomicAdd(&b->count, 1u) == nblocks - 1) {
      b->count = 0;
      __threadfence();
      atomicAdd(&b->gen, 1u);
    } else {
      long long i = 0;
      while (*vg == g) {
        if (i++ >= limit) {
          ok = 0;
          break;
        }
        __nanosleep(100);
      }
    }
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

// Cells of a group of the fused launch's corrector: a round of the predictor's threads.
template <int N>
__host__ __device__ constexpr int ens_fused_corrector_cells(int threads) {
  return threads < 2 * CfgC<Elastic, 3, N>::LINES ? 1 : threads / CfgC<Elastic, 3, N>::LINES;
}

// `steps` steps of every run in one launch: per step the time-step finalisation, the predictor
// over the concatenated cells, the Riemann solver over the concatenated faces of all directions,
// the corrector over groups of the concatenated cells and the time advance, separated by
// grid-wide barriers.  Rsteps: the runs' step arguments of each step ([steps][nr]).
template <int N, bool MIXED>
__global__ void __launch_bounds__(EnsCfg<N, MIXED, true>::TPB, EnsCfg<N, MIXED, true>::MINB)
    k_ens_fused(const StepArgs* __restrict__ Rsteps, const __grid_constant__ EnsTable E,
                const __grid_constant__ Tables T, const __grid_constant__ TablesF F, int steps,
                GridBar* bar, long long limit) {
  using P = Elastic;
  constexpr int D = 3;
  constexpr int TPB = EnsCfg<N, MIXED, true>::TPB;
  extern __shared__ __align__(16) double fsm[];
  const unsigned nb = gridDim.x;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  bool ok = true;
  for (int s = 0; s < steps && ok; ++s) {
    const StepArgs* R = Rsteps + (long long)s * E.nr;
    if (blockIdx.x == 0 && (int)threadIdx.x < E.nr) dt_finalize_one(R[threadIdx.x]);
    if (!(ok = grid_sync(bar, nb, limit))) break;
    for (long long it = blockIdx.x; it < E.blk0[E.nr]; it += nb)
      ens_predictor_block<N, MIXED, true>(R, E, T, F, it);
    if (!(ok = grid_sync(bar, nb, limit))) break;
    {
      const long long nf0 = E.face0[0][E.nr], nf1 = E.face0[1][E.nr];
      const long long nft = nf0 + nf1 + (D == 3 ? E.face0[2][E.nr] : 0);
      const long long wpb = TPB / 32;
      for (long long w = (long long)blockIdx.x * wpb + wib; w < nft; w += (long long)nb * wpb) {
        const int d = w < nf0 ? 0 : (w < nf0 + nf1 ? 1 : 2);
        const long long wd = w - (d == 0 ? 0 : (d == 1 ? nf0 : nf0 + nf1));
        const int r = ens_find(E.face0[d], E.nr, wd);  // the same for the whole warp
        riemann_face<P, D, N>(R[r], T, d, E.phioff[d][r], wd - E.face0[d][r], lane);
      }
    }
    if (!(ok = grid_sync(bar, nb, limit))) break;
    {
      // over the predictor's shared memory
      constexpr int CPB = ens_fused_corrector_cells<N>(TPB);
      ens_corrector<N, CPB, TPB>(R, E, *reinterpret_cast<SmemC<P, D, N, CPB>*>(fsm));
    }
    if (!(ok = grid_sync(bar, nb, limit))) break;
    if (blockIdx.x == 0 && (int)threadIdx.x < E.nr) advance_one(R[threadIdx.x].dev, 0);
    // the next step's finalisation (block 0, same threads) follows the advance in program order
  }
  if (!ok && threadIdx.x == 0)
    for (int r = 0; r < E.nr; ++r) atomicOr(&Rsteps[r].dev->status, ST_TIMEOUT);
}

// Launch `steps` steps of every run as one cooperative kernel (after zeroing the barrier).
template <int N, bool MIXED>
cudaError_t ens_fused_n(const StepArgs* R, const EnsTable& E, const Tables& T, const TablesF& F,
                        int steps, GridBar* bar, long long limit, int blocks_per_sm,
                        cudaStream_t s) {
  using G = EnsCfg<N, MIXED, true>;
  constexpr size_t SC = sizeof(SmemC<Elastic, 3, N, ens_fused_corrector_cells<N>(G::TPB)>);
  constexpr size_t SMEM = G::SMEM > SC ? G::SMEM : SC;
  static int max_bps = 0;
  if (!max_bps) {
    cudaError_t e = cudaFuncSetAttribute(k_ens_fused<N, MIXED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e != cudaSuccess) return e;
    int nbk = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nbk, k_ens_fused<N, MIXED>, G::TPB, SMEM);
    if (e != cudaSuccess) return e;
    max_bps = nbk < 1 ? 1 : nbk;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int bps = blocks_per_sm < 1 ? 1 : (blocks_per_sm > max_bps ? max_bps : blocks_per_sm);
  cudaError_t e = cudaMemsetAsync(bar, 0, sizeof(GridBar), s);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(sms * bps));
  cfg.blockDim = dim3(G::TPB);
  cfg.dynamicSmemBytes = SMEM;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_ens_fused<N, MIXED>, R, E, T, F, steps, bar, limit);
}

}  // namespace ader
