// Kernels of the fixed-point complex128 product (fx_phases.cuh): the tile kernel and the packing
// of the limbs.
#include <algorithm>

#include "fx_phases.cuh"

namespace bse {
namespace {

constexpr int FX_RING = 8192;   // two (TDA: four) rows per warp, two CTAs per SM

template <bool HASB>
__global__ void __launch_bounds__(FX_THREADS, 2)
k_prod_tiles_fx(const Prob* __restrict__ probs, const TileJob* __restrict__ jobs, int njobs, int nq, int mode,
                GenericIO io, int strided) {
  extern __shared__ __align__(128) unsigned char fxsm[];
  FxShared<FX_RING>& sh = *reinterpret_cast<FxShared<FX_RING>*>(fxsm);
  fx_init(sh);
  __syncthreads();
  dep_begin();
  clock_start(probs[0].clock);
  FxPipe pipe;
  fx_tiles_body<HASB, false>(probs, jobs, njobs, nq, mode, io, strided, blockIdx.x, gridDim.x, sh, pipe, probs[0].err);
}

// One CTA per tile (I, J >= I): the scale from the largest component, the choice between the
// fixed-point and the FP64 kernel (FX_SPREAD), and the limbs (zeros on the matrix diagonal).  The tile's
// second reading comes from L2.
template <bool HASB>
__global__ void __launch_bounds__(256)
k_fx_pack(const double2* __restrict__ A, const double2* __restrict__ B, int64_t N, int nT, int4* __restrict__ Af,
          int4* __restrict__ Bf, int* __restrict__ texp) {
  const int I = blockIdx.y, J = blockIdx.x;
  if (J < I) return;
  const int64_t t = (int64_t)I * nT - (int64_t)I * (I - 1) / 2 + (J - I);
  const double2* a = A + t * (TS * TS);
  const double2* b = HASB ? B + t * (TS * TS) : nullptr;
  __shared__ unsigned int smx[8], smn[8];
  __shared__ int weak[2][2][TS];       // of the rows and columns: neither matrix strong, not both
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto off_diag = [&](int e) { return I != J || (e >> 7) != (e & (TS - 1)); };
  // high words of the magnitudes; 1 for a subnormal that has none
  auto mag = [](double v) { return max(hi_abs(v), __double2loint(v) ? 1u : 0u); };
  weak[0][tid >> 7][tid & (TS - 1)] = weak[1][tid >> 7][tid & (TS - 1)] = 0;
  const int nr = (int)min((int64_t)TS, N - (int64_t)I * TS), nc = (int)min((int64_t)TS, N - (int64_t)J * TS);
  unsigned int m = 0, mn = 0xffffffffu;
  for (int e = tid; e < TS * TS; e += 256) {
    const double2 v = a[e];
    unsigned int t = max(mag(v.x), mag(v.y));
    if (HASB) {
      const double2 w = b[e];
      t = max(t, max(mag(w.x), mag(w.y)));
    }
    if (off_diag(e)) m = max(m, t);
    if ((e >> 7) < nr && (e & (TS - 1)) < nc) mn = min(mn, t);
  }
  m = __reduce_max_sync(0xffffffffu, m);
  mn = __reduce_min_sync(0xffffffffu, mn);
  if (lane == 0) {
    smx[warp] = m;
    smn[warp] = mn;
  }
  __syncthreads();
  for (int w = 0; w < 8; ++w) {
    m = max(m, smx[w]);
    mn = min(mn, smn[w]);
  }
  const int ex = max(1, (int)(m >> 20));
  for (int e = tid; e < TS * TS; e += 256) {
    double2 v = a[e], w = HASB ? b[e] : make_double2(0.0, 0.0);
    if (!off_diag(e)) v = w = make_double2(0.0, 0.0);
    Af[t * (TS * TS) + e] = fx_entry(v, ex);
    if (HASB) Bf[t * (TS * TS) + e] = fx_entry(w, ex);
    // entries that are not strong (the matrix diagonal never is)
    const unsigned int hv = max(hi_abs(v.x), hi_abs(v.y)), hw = HASB ? max(hi_abs(w.x), hi_abs(w.y)) : hv;
    const int r = e >> 7, c = e & (TS - 1);
    if (r < nr && c < nc && min(hv, hw) + (FX_STRONG << 20) < m) {
      atomicAdd(&weak[1][0][r], 1);
      atomicAdd(&weak[1][1][c], 1);
      if (max(hv, hw) + (FX_STRONG << 20) < m) {
        atomicAdd(&weak[0][0][r], 1);
        atomicAdd(&weak[0][1][c], 1);
      }
    }
  }
  __syncthreads();
  const int top = __reduce_max_sync(0xffffffffu, weak[0][tid >> 7][tid & (TS - 1)]);
  const int top2 = __reduce_max_sync(0xffffffffu, weak[1][tid >> 7][tid & (TS - 1)]);
  __syncthreads();
  if (lane == 0) {
    smx[warp] = top;
    smn[warp] = top2;
  }
  __syncthreads();
  // (a tile of zeros adds nothing; high words compare magnitudes to a few units of 2^-20)
  if (tid == 0) {
    const bool in_range = ex >= 256 && ex <= 1792;
    unsigned int w = 0, w2 = 0;
    for (int k = 0; k < 8; ++k) {
      w = max(w, smx[k]);
      w2 = max(w2, smn[k]);
    }
    texp[t] = m == 0 ? 1 : (in_range && m <= mn + (FX_SPREAD << 20) ? ex | (int)(w << FX_WEAK | w2 << FX_WEAK2) : -1);
  }
}

}  // namespace

// Bands per tile: the fewest row steps on the busiest SM, a unit of TS / nq rows costing about 16
// rows more (staging, the column sums).
int fx_bands(int ntiles) {
  int best = 1;
  int64_t cost = INT64_MAX;
  for (int nq = 1; nq <= 8; nq *= 2) {
    const int64_t c = (((int64_t)ntiles * nq + num_sms() - 1) / num_sms()) * (TS / nq + 16);
    if (c < cost) { cost = c; best = nq; }
  }
  return best;
}

// two CTAs per SM (96 KiB of shared memory and 128 registers a thread each)
int product_fx_occupancy() {
  static PerDevice<bool> opt_in;
  opt_in.get(current_device(), [] {
    cudaFuncSetAttribute(k_prod_tiles_fx<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxShared<FX_RING>));
    cudaFuncSetAttribute(k_prod_tiles_fx<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxShared<FX_RING>));
    return true;
  });
  return 2;
}

void launch_product_fx(const Prob* dprobs, const TileJob* jobs, int njobs, int nfx, int nq, int nprob, int maxnT,
                       int mode, const GenericIO* io_host, bool hasB, ProdShape shape, cudaStream_t s) {
  GenericIO io{};
  if (io_host) io = *io_host;
  if (nfx > 0) {
    count_launch();
    const int grid = product_grid(product_fx_occupancy(), shape, nfx * nq);
    if (hasB) launch_dep(k_prod_tiles_fx<true>, grid, FX_THREADS, sizeof(FxShared<FX_RING>), s, dprobs, jobs, nfx, nq, mode, io, shape.strided);
    else launch_dep(k_prod_tiles_fx<false>, grid, FX_THREADS, sizeof(FxShared<FX_RING>), s, dprobs, jobs, nfx, nq, mode, io, shape.strided);
  }
  if (njobs > nfx) launch_tiles_f64(dprobs, jobs + nfx, njobs - nfx, mode, io, hasB, shape, nfx == 0, s);
  launch_prod_reduce_f64(dprobs, nprob, maxnT, mode, io, s);
}

void launch_fx_pack(const double2* A, const double2* B, int64_t N, int nT, int4* Afx, int4* Bfx, int* texp,
                    cudaStream_t s) {
  count_launch();
  if (B) k_fx_pack<true><<<dim3(nT, nT), 256, 0, s>>>(A, B, N, nT, Afx, Bfx, texp);
  else k_fx_pack<false><<<dim3(nT, nT), 256, 0, s>>>(A, B, N, nT, Afx, nullptr, texp);
}

}  // namespace bse
