// dvm_euler1d.cu -- the Euler sub-steps of a short 1D problem (MUSCL of Section
// 4.3.2, limited or not): one cluster of at most 8 CTAs holds the whole tube in
// shared memory through all sub-steps of a kinetic step.
//
// Bound by latency: a sub-step of a few hundred cells is microseconds of
// dependent arithmetic (FP64 above all), and the grid barrier of the larger
// kernels with its loads and stores of the state through L2 costs as much
// again.  Here the cells a neighbour needs and the CTA's alpha are written
// straight into the other CTAs' shared memory and the hardware's cluster
// barrier ends the sub-step.  More cells per CTA than 64 would wait for one SM's FP64 pipe
// longer than the grid barrier costs.  200 cells, 9 sub-steps: FP64 98 -> 60 us;
// whole steps of 32 velocities, 16 / 200 / 512 cells: FP64 104 / 107 / 113 -> 71 /
// 72 / 86 us, FP32 53 / 47 / 52 -> 28 / 28 / 33 us.
#include <cooperative_groups.h>

#include <algorithm>

#include "dvm_euler64.cuh"
#include "dvm_internal.cuh"
#include "dvm_math.cuh"

namespace dvm {
namespace {

namespace cg = cooperative_groups;

constexpr int kClusterMax = 8;    // CTAs (the portable cluster size)
constexpr int kClusterCells = 64; // cells per CTA at most

// halved split fluxes (F +- alpha W) / 2 and half the limited slope of halved
// differences
__device__ __forceinline__ void split_half(const double* W, double al, double* gp, double* gm) {
  split64<1>(W, W[0] != 0.0 ? rcp64(W[0]) : 0.0, 0, al, gp, gm);
}
__device__ __forceinline__ void split_half(const float* W, float al, float* gp, float* gm) {
  float F[3];
  euler_flux<float, 1>(W, 0, F);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float f = 0.5f * F[k];
    gp[k] = fmaf(0.5f * al, W[k], f);
    gm[k] = fmaf(-0.5f * al, W[k], f);
  }
}
template <bool LIMITED> __device__ __forceinline__ double half_slope_of(double a, double b) { return half_slope<LIMITED>(a, b); }
template <bool LIMITED> __device__ __forceinline__ float half_slope_of(float a, float b) {
  return 0.5f * slope<float, LIMITED>(a, b);
}
// maxima of values >= 0 as integers (an FP64 comparison costs more)
__device__ __forceinline__ double max_bits(double a, double b) {
  return __longlong_as_double(max(__double_as_longlong(a), __double_as_longlong(b)));
}
__device__ __forceinline__ float max_bits(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double warp_max(double a) {
  for (int o = 16; o > 0; o >>= 1) a = max_bits(a, __shfl_xor_sync(0xffffffffu, a, o));
  return a;
}
__device__ __forceinline__ float warp_max(float a) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(a)));
}
__device__ __forceinline__ double alpha_1d(const double* W) {
  double a[2];
  alpha64<1>(W, a);
  return a[0];
}
__device__ __forceinline__ float alpha_1d(const float* W) {
  float a[3];
  state_alpha_of<1>(W, a);
  return a[0];
}

template <typename TF, bool LIMITED>
__global__ void __launch_bounds__(256) k_euler1d(Geom g, DevPtrs p) {
  constexpr int NM = 3, M = kClusterCells;
  __shared__ TF s_w[2][NM][M + 4], s_g[2 * NM][M + 4], s_f[NM][M + 1];
  __shared__ TF s_al[2][2 * kClusterMax];  // maxima of the two warps of cells of every CTA
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int nx = g.nx[0], tid = threadIdx.x, NT = blockDim.x;
  const int b0 = (int)((long long)rank * nx / C), m = (int)((long long)(rank + 1) * nx / C) - b0;
  const bool outflow = g.bc[0] == DVM_BC_OUTFLOW;
  const long long nc = g.nc;
  for (int i = tid; i < m + 4; i += NT) {
    const int c = bc_cell(b0 + i - 2, nx, g.bc[0]);
#pragma unroll
    for (int k = 0; k < NM; ++k) s_w[0][k][i] = ((const TF*)p.W0)[k * nc + c];
  }
  // the neighbours that need this CTA's first and last cells (none beyond an
  // outflow end, whose two ghosts are copies)
  const int lrank = rank > 0 ? rank - 1 : (outflow ? -1 : C - 1);
  const int rrank = rank + 1 < C ? rank + 1 : (outflow ? -1 : 0);
  const int ml = lrank < 0 ? 0 : (int)((long long)(lrank + 1) * nx / C) - (int)((long long)lrank * nx / C);
  double ad = __longlong_as_double((long long)__ldcg(p.aslot));
  const double a0 = ad;
  __shared__ TF s_kk;
  __shared__ int s_flags;  // bit 0: last sub-step, bit 1: no wave
  const int fk = tid / (m + 1), ff = tid - fk * (m + 1);
  double t = 0.0;
  int s = 0;
  bool last = false;
  cl.sync();  // every CTA runs before its shared memory is written
  for (;; ++s) {
    const int cur = s & 1;
    // length of the sub-step (Eq. Time2) by the last warp, which has no cells,
    // while the others form the split fluxes
    if (tid == NT - 1) {
      double dtE = 0.0;
      int flags = 0;
      if (g.forced_sub > 0) {
        dtE = g.dt / g.forced_sub;
        flags = s + 1 == g.forced_sub;
      } else if (!(ad > 0.0)) {
        flags = 2;
        if (rank == 0) set_status(p.status, DVM_ERR_NONPHYSICAL);
      } else {
        const double cfl = sizeof(TF) == 8 ? __ddiv_rn(__dmul_rn(0.5, g.dx), ad)
                                           : (double)__fdiv_rn(0.5f * (float)g.dx, (float)ad);
        const double rem = __dsub_rn(g.dt, t);
        flags = cfl >= rem;
        dtE = flags ? rem : cfl;
      }
      t = __dadd_rn(t, dtE);
      s_kk = sizeof(TF) == 8 ? (TF)(dtE / g.dx) : (TF)((float)dtE / (float)g.dx);
      s_flags = flags;
    }
    const TF al = (TF)ad;
    if (tid < m + 4) {
      const int i = tid;
      TF W[NM], gp[NM], gm[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) W[k] = s_w[cur][k][i];
      split_half(W, al, gp, gm);
#pragma unroll
      for (int k = 0; k < NM; ++k) s_g[k][i] = gp[k], s_g[NM + k][i] = gm[k];
    }
    __syncthreads();
    if (s_flags & 2) return;
    last = s_flags & 1;
    const TF kk = s_kk;
    // psi between cells f - 1 and f (entries f + 1 and f + 2)
    if (fk < NM) {
      const int k = fk, f = ff;
      const TF *gp = s_g[k] + f, *gm = s_g[NM + k] + f;
      const TF sp = half_slope_of<LIMITED>(gp[1] - gp[0], gp[2] - gp[1]);
      const TF sm = half_slope_of<LIMITED>(gm[2] - gm[1], gm[3] - gm[2]);
      s_f[k][f] = (gp[1] + gm[2]) + (sp - sm);
    }
    __syncthreads();
    TF a = TF(0);
    if (tid < m) {
      TF W[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        W[k] = fma(-kk, s_f[k][tid + 1] - s_f[k][tid], s_w[cur][k][tid + 2]);
        s_w[cur ^ 1][k][tid + 2] = W[k];
      }
      if (!last) {
        if (tid < 2 && lrank >= 0) {
          TF* o = cl.map_shared_rank(&s_w[cur ^ 1][0][0], lrank) + ml + 2 + tid;
#pragma unroll
          for (int k = 0; k < NM; ++k) o[k * (M + 4)] = W[k];
        }
        if (tid >= m - 2 && rrank >= 0) {
          TF* o = cl.map_shared_rank(&s_w[cur ^ 1][0][0], rrank) + tid - (m - 2);
#pragma unroll
          for (int k = 0; k < NM; ++k) o[k * (M + 4)] = W[k];
        }
        if (tid == 0 && lrank < 0)
#pragma unroll
          for (int k = 0; k < NM; ++k) s_w[cur ^ 1][k][0] = s_w[cur ^ 1][k][1] = W[k];
        if (tid == m - 1 && rrank < 0)
#pragma unroll
          for (int k = 0; k < NM; ++k) s_w[cur ^ 1][k][m + 2] = s_w[cur ^ 1][k][m + 3] = W[k];
        a = alpha_1d(W);
      }
    }
    if (last) break;
    if (s + 1 >= g.m_cap) {
      if (rank == 0 && tid == 0) set_status(p.status, DVM_ERR_CFL);
      cl.sync();  // (no CTA leaves before the others' writes to it)
      break;
    }
    if (tid < kClusterCells) {  // (two warps hold the cells)
      a = warp_max(a);
      if ((tid & 31) < C) *cl.map_shared_rank(&s_al[cur ^ 1][2 * rank + (tid >> 5)], tid & 31) = a;
    }
    cl.sync();
    TF v = TF(0);
    for (int r = 0; r < 2 * C; ++r) v = max_bits(v, s_al[cur ^ 1][r]);
    ad = (double)v;
  }
  const int n = s + 1;  // (a thread's own cell)
  TF* dst = (TF*)((n & 1) ? p.W1 : p.W0);
  if (tid < m)
#pragma unroll
    for (int k = 0; k < NM; ++k) dst[k * nc + b0 + tid] = s_w[n & 1][k][tid + 2];
  if (rank == 0 && tid == 0) {
    *p.msub = n;
    p.alpha[0] = a0;
    p.alpha[1] = p.alpha[2] = 0.0;
  }
}

template <typename TF, bool LIMITED>
cudaError_t launch_t(const Geom& g, const DevPtrs& p, cudaStream_t s) {
  const int C = std::min(kClusterMax, g.nx[0] / 2), most = (g.nx[0] + C - 1) / C;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)std::min(256, std::max(64, (3 * (most + 1) + 31) / 32 * 32)));
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_euler1d<TF, LIMITED>, g, p);
}

}  // namespace

bool euler1d_eligible(const Geom& g) {
  return g.d == 1 && g.scheme != DVM_HOFKS_WENO && g.nx[0] >= 2 && g.nx[0] <= kClusterMax * kClusterCells;
}

cudaError_t launch_euler1d(const Geom& g, const DevPtrs& p, bool limited, cudaStream_t s) {
  if (g.precision == DVM_F64) return limited ? launch_t<double, true>(g, p, s) : launch_t<double, false>(g, p, s);
  return limited ? launch_t<float, true>(g, p, s) : launch_t<float, false>(g, p, s);
}

}  // namespace dvm
