// dvm_euler64.cu -- the Euler sub-steps of 1D and 2D problems in FP64 (MUSCL of
// Section 4.3.2, limited or not): one cooperative launch for all sub-steps of a
// kinetic step, a grid barrier between them.
//
// Bound by the FP64 pipe: GB300 issues 2 FP64 lanes per clock and SM, so a
// sub-step costs its FP64 instructions per warp x 16 clocks on the busiest SM.
// Hence (1) every face flux is evaluated once, one thread per (face,
// component), instead of by both of its cells; (2) split fluxes only on the
// cross the faces need, not on the corners; (3) quotients share a reciprocal
// (third-order Newton iteration on the hardware seed) and one residual
// correction instead of a full division each; (4) the tile is sized at creation
// so that the tiles fill the SMs evenly and the warps are full; (5) with the
// halved split fluxes g = (F +- alpha W) / 2 the limited slope of Eq. discmom
// enters as a b / (a + b), saving the constants.  About 330 FP64 instructions
// per cell and sub-step against 720 in the two-phase kernel.  A kinetic step's
// sub-steps: 2D 256^2 1981 -> 978 us, 100^2 with 100 sub-steps 3184 -> 1317 us,
// 1D 200 cells (9 sub-steps) 195 -> 98 us.
#include <math.h>

#include <algorithm>

#include "dvm_euler64.cuh"
#include "dvm_internal.cuh"
#include "dvm_math.cuh"

namespace dvm {
namespace {

constexpr int kE64Threads = 256;

struct Tile64 {
  int tx, ty;        // cells of a tile
  int ntx, ntiles;   // tiles per row, in all
};

// doubles of shared memory: states of the cross, split fluxes along x and y,
// face fluxes along x and y
__host__ __device__ inline int smem64(int d, int tx, int ty) {
  const int nm = d + 2;
  int n = nm * tx * ty + nm * 4 * ty + 2 * nm * (tx + 4) * ty + nm * (tx + 1) * ty;
  if (d == 2) n += nm * 4 * tx + 2 * nm * tx * (ty + 4) + nm * tx * (ty + 1);
  return n;
}

template <int D, bool LIMITED>
__global__ void __launch_bounds__(kE64Threads) k_euler64(Geom g, DevPtrs p, Tile64 T) {
  constexpr int NM = D + 2;
  extern __shared__ double s_e64[];
  __shared__ double s_max[2][kE64Threads / 32], s_t[4];
  __shared__ int s_flags;
  const int TX = T.tx, TY = T.ty, tid = threadIdx.x, NT = blockDim.x;
  const int nint = TX * TY, nxh = 4 * TY, nyh = D == 2 ? 4 * TX : 0, ns = nint + nxh + nyh;
  const int gxs = (TX + 4) * TY, gys = D == 2 ? TX * (TY + 4) : 0;
  const int fxs = (TX + 1) * TY, fys = D == 2 ? TX * (TY + 1) : 0;
  double* s_w = s_e64;                       // [NM][ns]
  double* s_gx = s_w + NM * ns;              // [2 NM][TY][TX + 4]
  double* s_gy = s_gx + 2 * NM * gxs;        // [2 NM][TY + 4][TX]
  double* s_fx = s_gy + 2 * NM * gys;        // [NM][TY][TX + 1]
  double* s_fy = s_fx + NM * fxs;            // [NM][TY + 1][TX]
  const int Nx = g.nx[0], Ny = D == 2 ? g.nx[1] : 1;
  const long long nc = g.nc;
  const unsigned long long nb = gridDim.x;
  // every launch of a handle completes whole generations of the barrier, and
  // none can end before this block arrives
  unsigned long long target = 0;
  if (tid == 0) target = ld_acquire_u64(p.gbar) / nb * nb;
  double t = 0.0, a0[2] = {0.0, 0.0};
  int s = 0;
  for (;; ++s) {
    const double* src = (const double*)((s & 1) ? p.W1 : p.W0);
    double* dst = (double*)((s & 1) ? p.W0 : p.W1);
    // the sub-step's alpha and length (Eq. Time2) by thread 0 while the others
    // stage the first tile's states
    if (tid == 0) {
      double ad[3], asum = 0.0;
      for (int d = 0; d < 3; ++d) ad[d] = __longlong_as_double((long long)__ldcg(p.aslot + (s % 3) * 3 + d));
      for (int d = 0; d < D; ++d) asum = __dadd_rn(asum, ad[d]);
      if (s == 0) a0[0] = ad[0], a0[1] = ad[1];
      if (blockIdx.x == 0)
        for (int d = 0; d < 3; ++d) p.aslot[((s + 2) % 3) * 3 + d] = 0ull;
      double dtE = 0.0;
      int flags = 0;
      if (g.forced_sub > 0) {
        dtE = g.dt / g.forced_sub;
        flags = s + 1 == g.forced_sub;
      } else if (!(asum > 0.0)) {
        flags = 2;
        if (blockIdx.x == 0) set_status(p.status, DVM_ERR_NONPHYSICAL);
      } else {
        const double cfl = __ddiv_rn(__dmul_rn(0.5, g.dx), asum), rem = __dsub_rn(g.dt, t);
        flags = cfl >= rem;
        dtE = flags ? rem : cfl;
      }
      t = __dadd_rn(t, dtE);
      s_t[0] = ad[0], s_t[1] = ad[1], s_t[2] = dtE / g.dx;
      s_flags = flags;
    }
    double amax[2] = {0.0, 0.0};
    bool last = false;
    for (int tile = blockIdx.x; tile < T.ntiles; tile += gridDim.x) {
      const int x0 = tile % T.ntx * TX, y0 = tile / T.ntx * TY;
      // states of the tile and its cross-shaped halo
      for (int i = tid; i < ns; i += NT) {
        int lx, ly;
        if (i < nint) {
          ly = i / TX, lx = i - ly * TX;
        } else if (i < nint + nxh) {
          const int h = (i - nint) & 3;
          ly = (i - nint) >> 2, lx = h < 2 ? h - 2 : TX + h - 2;
        } else {
          const int h = (i - nint - nxh) / TX;
          lx = i - nint - nxh - h * TX, ly = h < 2 ? h - 2 : TY + h - 2;
        }
        const long long c = bc_cell(x0 + lx, Nx, g.bc[0]) + (D == 2 ? (long long)Nx * bc_cell(y0 + ly, Ny, g.bc[1]) : 0);
#pragma unroll
        for (int k = 0; k < NM; ++k) s_w[k * ns + i] = __ldcg(src + k * nc + c);
      }
      __syncthreads();
      const int flags = s_flags;
      if (flags & 2) return;
      last = flags & 1;
      const double al[2] = {s_t[0], s_t[1]}, kk = s_t[2];
      for (int i = tid; i < ns; i += NT) {
        double W[NM], gp[NM], gm[NM];
#pragma unroll
        for (int k = 0; k < NM; ++k) W[k] = s_w[k * ns + i];
        const double r = W[0] != 0.0 ? rcp64(W[0]) : 0.0;
        int lx, ly, dirs;
        if (i < nint) {
          ly = i / TX, lx = i - ly * TX, dirs = 3;
        } else if (i < nint + nxh) {
          const int h = (i - nint) & 3;
          ly = (i - nint) >> 2, lx = h < 2 ? h - 2 : TX + h - 2, dirs = 1;
        } else {
          const int h = (i - nint - nxh) / TX;
          lx = i - nint - nxh - h * TX, ly = h < 2 ? h - 2 : TY + h - 2, dirs = 2;
        }
        if (dirs & 1) {
          split64<D>(W, r, 0, al[0], gp, gm);
          double* o = s_gx + ly * (TX + 4) + lx + 2;
#pragma unroll
          for (int k = 0; k < NM; ++k) o[k * gxs] = gp[k], o[(NM + k) * gxs] = gm[k];
        }
        if (D == 2 && (dirs & 2)) {
          split64<D>(W, r, 1, al[1], gp, gm);
          double* o = s_gy + (ly + 2) * TX + lx;
#pragma unroll
          for (int k = 0; k < NM; ++k) o[k * gys] = gp[k], o[(NM + k) * gys] = gm[k];
        }
      }
      __syncthreads();
      // psi_{j+1/2} = g+_j + slope/2 (g+) + g-_{j+1} - slope/2 (g-), one thread
      // per face and component
      const int nf = NM * (fxs + fys);
      for (int i = tid; i < nf; i += NT) {
        const bool isx = i < NM * fxs;
        const int e = isx ? i : i - NM * fxs;
        const int per = isx ? fxs : fys;
        const int k = e / per, f = e - k * per;
        int at, st;  // cell j of the face in its split-flux array
        const double *gp, *gm;
        if (isx) {
          const int ly = f / (TX + 1);
          at = ly * (TX + 4) + (f - ly * (TX + 1)) + 1;
          st = 1;
          gp = s_gx + k * gxs, gm = s_gx + (NM + k) * gxs;
        } else {
          at = f + TX;
          st = TX;
          gp = s_gy + k * gys, gm = s_gy + (NM + k) * gys;
        }
        const double p0 = gp[at - st], p1 = gp[at], p2 = gp[at + st];
        const double m1 = gm[at], m2 = gm[at + st], m3 = gm[at + 2 * st];
        const double sp = half_slope<LIMITED>(p1 - p0, p2 - p1), sm = half_slope<LIMITED>(m2 - m1, m3 - m2);
        (isx ? s_fx : s_fy)[e] = (p1 + m2) + (sp - sm);
      }
      __syncthreads();
      for (int i = tid; i < nint; i += NT) {
        const int ly = i / TX, lx = i - ly * TX;
        const int x = x0 + lx, y = y0 + ly;
        if (x >= Nx || y >= Ny) continue;
        double Wn[NM];
        const long long c = x + (long long)Nx * y;
#pragma unroll
        for (int k = 0; k < NM; ++k) {
          const double* fx = s_fx + k * fxs + ly * (TX + 1) + lx;
          double acc = fx[1] - fx[0];
          if (D == 2) {
            const double* fy = s_fy + k * fys + i;
            acc += fy[TX] - fy[0];
          }
          Wn[k] = fma(-kk, acc, s_w[k * ns + i]);
          dst[k * nc + c] = Wn[k];
        }
        if (!last) {
          double a[2];
          alpha64<D>(Wn, a);
          amax[0] = fmax(amax[0], a[0]);
          if (D == 2) amax[1] = fmax(amax[1], a[1]);
        }
      }
      __syncthreads();
    }
    if (last) break;
    // the maxima as bit patterns (they are >= 0): integer reductions
#pragma unroll
    for (int d = 0; d < D; ++d) {
      for (int o = 16; o > 0; o >>= 1) amax[d] = fmax(amax[d], __shfl_xor_sync(0xffffffffu, amax[d], o));
      if ((tid & 31) == 0) s_max[d][tid >> 5] = amax[d];
    }
    __syncthreads();
    if (tid == 0) {
      for (int d = 0; d < D; ++d) {
        double v = 0.0;
        for (int w = 0; w < NT / 32; ++w) v = fmax(v, s_max[d][w]);
        atomicMax(p.aslot + ((s + 1) % 3) * 3 + d, (unsigned long long)__double_as_longlong(v));
      }
    }
    if (s + 1 >= g.m_cap) {
      if (blockIdx.x == 0 && tid == 0) set_status(p.status, DVM_ERR_CFL);
      break;
    }
    // grid barrier: arrive with a release, wait (bounded) for this generation
    if (tid == 0) {
      target += nb;
      __threadfence();
      asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p.gbar), "l"(1ull) : "memory");
      int good = 1;
      const long long c0 = clock64();
      while (ld_acquire_u64(p.gbar) < target) {
        if (clock64() - c0 > (1LL << 31)) {
          set_status(p.status, DVM_ERR_TIMEOUT);
          good = 0;
          break;
        }
      }
      s_flags = good ? 0 : 2;
    }
    __syncthreads();
    if (s_flags & 2) return;
    __syncthreads();
  }
  if (blockIdx.x == 0 && tid == 0) {
    *p.msub = s + 1;
    p.alpha[0] = a0[0];
    p.alpha[1] = a0[1];
    p.alpha[2] = 0.0;
  }
}

// The tile whose busiest SM has the fewest FP64 instructions per sub-step, in
// warps x instructions: states 45 each, faces 24, updates with alpha 90, and
// 120 a tile for its barriers; at most 100 KB of shared memory.  Up to 4000
// candidates, so once per handle (searched at every launch, a step outside a graph cost the
// host 16 us instead of 10).
Tile64 best_tile64(const Geom& g, int sms) {
  const int nm = g.d + 2;
  auto warps = [](int n) { return (n + 31) / 32; };
  Tile64 best{};
  long long cost = 0;
  for (int ty = 1; ty <= (g.d == 2 ? std::min(32, g.nx[1]) : 1); ++ty)
    for (int tx = std::min(4, g.nx[0]); tx <= std::min(128, g.nx[0]); ++tx) {
      if (smem64(g.d, tx, ty) * 8 > 100 * 1024) break;
      const int ntx = (g.nx[0] + tx - 1) / tx, nty = g.d == 2 ? (g.nx[1] + ty - 1) / ty : 1;
      const long long tiles = (long long)ntx * nty;
      const int ns = tx * ty + 4 * ty + (g.d == 2 ? 4 * tx : 0);
      const int nf = nm * ((tx + 1) * ty + (g.d == 2 ? tx * (ty + 1) : 0));
      const long long c = (tiles + sms - 1) / sms * (45 * warps(ns) + 24 * warps(nf) + 90 * warps(tx * ty) + 120);
      if (!best.tx || c < cost || (c == cost && tiles < best.ntiles)) best = {tx, ty, ntx, (int)tiles}, cost = c;
    }
  return best;
}

Tile64 tile64(const Geom& g) {
  const int tx = g.euler_tile[0], ty = g.euler_tile[1], ntx = (g.nx[0] + tx - 1) / tx;
  return {tx, ty, ntx, ntx * ((g.nx[1] + ty - 1) / ty)};
}

template <int D, bool LIMITED>
cudaError_t launch_t(const Geom& g, const DevPtrs& p, cudaStream_t s, bool prepare, int* blocks, cudaEvent_t started) {
  const Tile64 T = tile64(g);
  const size_t smem = sizeof(double) * smem64(D, T.tx, T.ty);
  auto* k = k_euler64<D, LIMITED>;
  const int items = std::max((D + 2) * ((T.tx + 1) * T.ty + (D == 2 ? T.tx * (T.ty + 1) : 0)), 64);
  const int threads = std::min(kE64Threads, (items + 31) / 32 * 32);
  if (prepare) {
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    int per_sm = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem);
    *blocks = (int)std::min<long long>((long long)sms * std::max(per_sm, 1), T.ntiles);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)g.euler_blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  if (started) {
    attr[1].id = cudaLaunchAttributeLaunchCompletionEvent;
    attr[1].val.launchCompletionEvent.event = started;
    attr[1].val.launchCompletionEvent.flags = 0;
  }
  cfg.attrs = attr;
  cfg.numAttrs = started ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k, g, p, T);
}

}  // namespace

void euler64_tile(Geom* g) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const Tile64 T = best_tile64(*g, sms);
  g->euler_tile[0] = T.tx, g->euler_tile[1] = T.ty;
}

cudaError_t launch_euler64(const Geom& g, const DevPtrs& p, bool limited, cudaStream_t s, bool prepare, int* blocks,
                           cudaEvent_t started) {
  if (g.d == 1)
    return limited ? launch_t<1, true>(g, p, s, prepare, blocks, started) : launch_t<1, false>(g, p, s, prepare, blocks, started);
  return limited ? launch_t<2, true>(g, p, s, prepare, blocks, started) : launch_t<2, false>(g, p, s, prepare, blocks, started);
}

}  // namespace dvm
