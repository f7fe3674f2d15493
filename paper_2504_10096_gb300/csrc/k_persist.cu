// Persistent Krylov steps for one small problem.
//
// A Lanczos step of a problem of a few thousand rows is a chain of short phases -- the
// structured product (tiles, then the block-row reduction), two Gram-Schmidt passes (dots,
// then the update), the second product on the folded path, the norm and the new basis
// vector -- each far too small to fill the GPU, so with one kernel per phase the launch
// and drain gaps cost more than the work.  Here one cooperative launch runs all the steps of
// a restart cycle: every CTA loops over the units of a phase (the same bodies and unit
// decomposition as the per-phase kernels, bse_phases.cuh, so the result is the same bits),
// and the phases are separated by a grid barrier.  The state machine is the device-resident
// KState: the step loop stops when the subspace is full, a breakdown asks the host for a fresh
// vector, or the problem is done; the restart itself stays with the per-phase kernels.
//
// What bounds it: the latency of a phase's loads and of its barrier (1.1-2 us), and in larger problems
// the integer pipe in the tiles.  Per step: TDA N = 2000, complex128, 36 us (tiles 14, reduction 2.3, dots
// 2 x 2.5, updates 2 x 4.5, normalisation 2.6, the rest barriers), 82 us with FP64-pipe tiles; PH
// N = 3000 99 us (tiles 2 x 30), 225 before.
//
// The grid barrier counts arrivals; every wait is bounded (about a second of polling), after
// which the CTA raises the barrier's error flag and returns, and the others' waits expire in turn,
// so a wait can never hang the device.  The launch is
// cooperative, so all CTAs are resident together.
#include <algorithm>
#include <cstddef>

#include "fx_phases.cuh"
#include "grid_sync.cuh"

namespace bse {
namespace {

constexpr int PS_THREADS = 256;
// One CTA per SM: two of 128 registers a thread spill in the product's row loop (measured, PH
// N = 3000: 473 ms against 311; TDA N = 2000: 81 against 53).
constexpr int PS_RING = 8192;              // two (TDA: four) tile rows per warp in flight (16 KiB: no faster)

// The FP64 tiles (a few, if any, beside fixed-point ones) stay out of line: their registers would be
// spilled around the other phases.
template <typename ST, typename R, bool HASB>
__device__ __noinline__ void ps_tiles(const Prob* probs, const TileJob* jobs, int njobs, int mode, int bid, int nblk,
                                      unsigned char* sm) {
  using CT = typename Acc<R>::T;
  CT* xc = reinterpret_cast<CT*>(sm);
  CT(*red)[TS] = reinterpret_cast<CT(*)[TS]>(xc + 2 * TS);
  prod_tiles_body<ST, R, HASB, true>(probs, jobs, njobs, mode, GenericIO{}, 1, bid, nblk, xc, xc + TS, red);
}

template <typename ST, typename R, bool HASB>
__global__ void __launch_bounds__(PS_THREADS, 1)
k_steps_persist(const Prob* __restrict__ probs, const TileJob* __restrict__ jobs, int njobs, int nfx, int steps,
                GridBar* gb) {
  constexpr bool FX = std::is_same<ST, double2>::value;
  extern __shared__ __align__(128) unsigned char psm[];
  __shared__ int s_ok;
  // every CTA keeps its own copy of the problem's description and state and advances the state
  // itself (the same numbers everywhere): no read of it has to cross the GPU
  __shared__ KState s_st;
  __shared__ Prob s_p;
  const int bid = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned int nblk = gridDim.x;
  unsigned int gen = 0;
  KState* const gst = probs[0].st;
  if (tid == 0) {
    s_p = probs[0];
    s_st = *gst;
    s_p.st = &s_st;
  }
  const int ph = HASB ? 1 : 0;
  // the fixed-point product's row rings and barriers keep their place (complex128); the rest of
  // the shared memory is carved per phase
  FxPipe pipe;
  unsigned char* rest = psm;
  if constexpr (FX) {
    fx_init(*reinterpret_cast<FxShared<PS_RING>*>(psm));
    rest += offsetof(FxShared<PS_RING>, x);
  }
  __syncthreads();
  const Prob& p = s_p;
  const KState* st = &s_st;
  const int nslab = (int)(p.Npad / p.slab), nch = dot_chunks(p.nT);
  const GenericIO io{};
  using CT = typename Acc<R>::T;
  ST* cf = reinterpret_cast<ST*>(rest);
  ST(*ured)[32] = reinterpret_cast<ST(*)[32]>(cf + 2 * MAXM + 2);
  CT(*grp)[REDUCE_ROWS] = reinterpret_cast<CT(*)[REDUCE_ROWS]>(rest);
  for (int s = 0; s < steps; ++s) {
    if (!kactive(st)) break;                          // the same state in every CTA
#pragma unroll 1
    for (int prod = 0; prod < (HASB ? 2 : 1); ++prod) {
      const int mode = !HASB ? PM_STEP_A : (prod ? PM_STEP_MPLUS : PM_STEP_MMINUS);
      // the tiles: the fixed-point ones (complex128), then the others
      if constexpr (FX)
        if (nfx > 0)
          fx_tiles_body<HASB, true>(&s_p, jobs, nfx, p.nq, mode, io, 1, bid, nblk, *reinterpret_cast<FxShared<PS_RING>*>(psm),
                                    pipe, p.err);
      if (njobs > nfx) ps_tiles<ST, R, HASB>(&s_p, jobs + nfx, njobs - nfx, mode, bid, nblk, rest);
      if (!grid_sync(gb, nblk, gen, &s_ok)) return;
      for (int u = bid; u < REDUCE_UNITS * p.nT; u += nblk) prod_reduce_body<ST, R, true>(&s_p, mode, io, u, 0, grp);
      if (!grid_sync(gb, nblk, gen, &s_ok)) return;
      if (prod) break;
      const CgsSet cs = cgs_set(p, st, ph, 0);
      const int nset = cs.nm + cs.nt;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        // tasks go round the CTAs first: neighbours share an SM's schedulers as little as possible
        for (int t = bid + nblk * warp; t < nset * nch; t += nblk * (PS_THREADS / 32))
          cgs_dot_task<ST, true>(p, st, cs, ph, 0, 0, pass, t % nset, t / nset);
        if (!grid_sync(gb, nblk, gen, &s_ok)) return;
        for (int u = bid; u < nslab; u += nblk) {
          cgs_update_unit<ST, true>(p, st, ph, pass, 0, 0, u, cf, ured);
          __syncthreads();
        }
        if (!grid_sync(gb, nblk, gen, &s_ok)) return;
      }
    }
    // the new basis vector by the warps that have rows, and beside it the end of the step by the last
    // warp: the rows go by a copy of the index the step's end advances
    KState now;
    now.j = st->j;
    __syncthreads();
    const bool endw = warp == PS_THREADS / 32 - 1;
    double b2 = 0.0;
    const int64_t r0 = ((int64_t)bid + (int64_t)nblk * warp) * 32;
    if (endw || r0 < p.Npad) b2 = norm_sum<true>(p, ph);
    if (r0 < p.Npad && b2 > 0.0 && isfinite(b2)) {
      const R inv = (R)rsqrt(b2);
      for (int64_t r = r0; r < p.Npad; r += (int64_t)nblk * PS_THREADS)
        normalize_row<ST, true>(p, &now, ph, 0, r + lane, inv);
    }
    if (endw && lane == 0) finish_one<true>(s_p, ph, 0, 0, b2, bid == 0);
    if (!grid_sync(gb, nblk, gen, &s_ok)) return;
  }
  __syncthreads();
  if (bid == 0 && tid == 0) *gst = s_st;
}

template <typename ST, typename R, bool HASB>
size_t persist_smem() {
  using CT = typename Acc<R>::T;
  const size_t prod = (size_t)10 * TS * sizeof(CT);
  const size_t red = (size_t)REDUCE_GROUPS * REDUCE_ROWS * sizeof(CT);
  const size_t upd = (size_t)(2 * MAXM + 2) * sizeof(ST) + (size_t)8 * 32 * sizeof(ST);
  const size_t rest = std::max(std::max(prod, red), upd);
  if (!std::is_same<ST, double2>::value) return rest;
  return std::max(sizeof(FxShared<PS_RING>), offsetof(FxShared<PS_RING>, x) + rest);
}

template <typename ST, typename R, bool HASB>
int persist_grid() {
  static PerDevice<int> grid;
  const int dev = current_device();
  return grid.get(dev, [&] {
    const size_t sm = persist_smem<ST, R, HASB>();
    if (sm > 48 * 1024)
      cudaFuncSetAttribute(k_steps_persist<ST, R, HASB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    int occ = 0, nsm = 0, coop = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_steps_persist<ST, R, HASB>, PS_THREADS, sm);
    cudaGetLastError();
    return (coop && occ >= 1) ? nsm : 0;    // one CTA per SM: every CTA resident
  });
}

template <typename ST, typename R, bool HASB>
int launch_persist_t(const Prob* dprobs, const TileJob* jobs, int njobs, int nfx, int steps, GridBar* gb,
                     cudaStream_t s) {
  const int grid = persist_grid<ST, R, HASB>();
  if (grid <= 0) return 1;
  if (cudaMemsetAsync(gb, 0, sizeof(GridBar), s) != cudaSuccess) return -1;
  const size_t sm = persist_smem<ST, R, HASB>();
  void* args[] = {(void*)&dprobs, (void*)&jobs, (void*)&njobs, (void*)&nfx, (void*)&steps, (void*)&gb};
  count_launch();
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_steps_persist<ST, R, HASB>, dim3(grid),
                                                    dim3(PS_THREADS), args, sm, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  return 0;
}

}  // namespace

template <typename ST, typename R>
int launch_steps_persist(const Prob* dprobs, const TileJob* jobs, int njobs, int nfx, bool ph, int steps,
                         GridBar* gb, cudaStream_t s) {
  return ph ? launch_persist_t<ST, R, true>(dprobs, jobs, njobs, nfx, steps, gb, s)
            : launch_persist_t<ST, R, false>(dprobs, jobs, njobs, nfx, steps, gb, s);
}

template int launch_steps_persist<double2, double>(const Prob*, const TileJob*, int, int, bool, int, GridBar*,
                                                   cudaStream_t);
template int launch_steps_persist<float2, float>(const Prob*, const TileJob*, int, int, bool, int, GridBar*,
                                                 cudaStream_t);

}  // namespace bse
