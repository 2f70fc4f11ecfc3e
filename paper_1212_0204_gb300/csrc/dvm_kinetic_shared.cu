// dvm_kinetic_shared.cu -- launch of the kinetic pass with CTA-shared source
// rows (dvm_shared_kernel.cuh): which configurations take it, its velocity
// splits and its folded chunks.
#include <math.h>

#include <algorithm>

#include "dvm_shared_kernel.cuh"

namespace dvm {
namespace {

// Slot rows per CTA at most, so that the shared memory leaves room for as many
// CTAs as the registers do (FP64 two, HOFKS three, FKS four).
int max_rows(const Geom& g) { return g.precision == DVM_F64 ? 36 : 40; }

constexpr int kMaxSplits = 40;

int form_of(const Geom& g) {
  if (g.scheme == DVM_FKS) return kFormFks;
  return g.lin_slice && !g.learn ? kFormP : kFormFull;
}

bool any_outflow(const Geom& g) {
  bool o = false;
  for (int i = 0; i < g.d; ++i) o |= g.bc[i] == DVM_BC_OUTFLOW;
  return o;
}

// Shared memory of a CTA at most: two CTAs per SM.
constexpr size_t kMaxSmem = 113 * 1024;

// ky per folded chunk: equal chunks, a multiple of 4 (the staged block), whose
// rows (16 + the range of delta over the chunk) fit max_rows, or fewer rows
// where the tables of a long velocity axis or of a narrow box (32 columns reach
// many 16-row blocks) leave no room for these.  rows = 0 where not even chunks
// of 24 rows fit.  The HOFKS slots count as the full form's, so that the shape
// does not change with the learned path.
SharedLaunch shape_of(const Geom& g, int splits) {
  SharedLaunch sl;
  sl.splits = splits;
  sl.blocks = std::min((30 + g.nx[0]) / g.nx[0] + 1, (g.nx[1] + kShTY - 1) / kShTY);
  const int q = std::min(g.p, kMaxV1);  // (a chunk is no longer than the axis)
  const int W = g.precision == DVM_F64 ? ShShape<double>::W : ShShape<float>::W;
  for (int top = max_rows(g); top >= 24; top -= 4) {
    const int most = q == 1 ? top - kShTY : ((top - kShTY - 3) * q) & ~3;
    const int chunks = (g.nv[1] + most - 1) / most;
    sl.kc = ((g.nv[1] + chunks - 1) / chunks + 3) & ~3;
    sl.rows = kShTY + (q == 1 ? sl.kc : (sl.kc + q - 1) / q + 2);
    if (shared_smem(g, g.scheme == DVM_FKS ? kFormFks : kFormFull, sl.rows, sl.blocks, W) <= kMaxSmem) return sl;
  }
  sl.rows = 0;
  return sl;
}

// One thread per cell: the parameter rows into the layouts of fold_shared.
template <int D, int FORM>
__global__ void __launch_bounds__(256) k_shared_fold(Geom g, DevPtrs p) {
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const long long nc = g.nc;
  if (c >= nc) return;
  const float4* __restrict__ pg = (const float4*)p.prm;
  float r[16];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 v = __ldg(pg + q * nc + c);
    r[4 * q] = v.x, r[4 * q + 1] = v.y, r[4 * q + 2] = v.z, r[4 * q + 3] = v.w;
  }
  const float lam = r[row_lam()], L = r[row_L()], h = r[row_h(D)];
  const float ux = r[row_u(0)], uy = r[row_u(1)], uz = D == 3 ? r[row_u(2)] : 0.f;
  const float *nu = r + row_nu(D, 0), *mu = r + row_mu(D, 0);
  float4* __restrict__ o = (float4*)p.wprm + c;
  if constexpr (FORM == kFormFks) {
    o[0] = make_float4(L, h, ux, uy);
    o[nc] = D == 3 ? make_float4(uz, mu[0], mu[1], mu[2]) : make_float4(mu[0], mu[1], mu[2], mu[3]);
    if (D == 3) o[2 * nc] = make_float4(mu[3], mu[4], 0.f, 0.f);
  } else {
    o[0] = make_float4(lam, L, h, uy);
    if constexpr (FORM == kFormP) {
      float P[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) P[i] = fmaf(lam, nu[i], mu[i]);
      o[nc] = make_float4(ux, uz, P[0], P[1]);
      o[2 * nc] = make_float4(P[2], P[3], P[4], 0.f);
    } else if constexpr (D == 3) {
      o[nc] = make_float4(ux, uz, lam * nu[0], lam * nu[1]);
      o[2 * nc] = make_float4(lam * nu[2], lam * nu[3], lam * nu[4], mu[0]);
      o[3 * nc] = make_float4(mu[1], mu[2], mu[3], mu[4]);
    } else {
      o[nc] = make_float4(ux, lam * nu[0], lam * nu[1], lam * nu[2]);
      o[2 * nc] = make_float4(lam * nu[3], mu[0], mu[1], mu[2]);
      o[3 * nc] = make_float4(mu[3], 0.f, 0.f, 0.f);
    }
  }
}

template <typename TS, int D, int FORM, bool P1, bool OUT, bool FLUSH = false>
void launch_one(const Geom& g, const DevPtrs& p, int splits, cudaStream_t s, bool prepare) {
  constexpr int MINB = sizeof(TS) == 8 ? 2 : (FORM == kFormFks ? 4 : 3);
  auto* k = k_kpass_shared<TS, D, FORM, P1, OUT, FLUSH, MINB>;
  const SharedLaunch sl = shape_of(g, splits);
  if (prepare) {
    // the most any configuration takes, so that handles do not lower it for
    // one another
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxSmem);
    return;
  }
  if constexpr (sizeof(TS) != 8) k_shared_fold<D, FORM><<<(unsigned)((g.nc + 255) / 256), 256, 0, s>>>(g, p);
  const long long cols = (long long)g.nx[0] * ((g.nx[1] + kShTY - 1) / kShTY);
  const dim3 grid((unsigned)((cols + 31) / 32), (unsigned)(g.nx[2] * splits));
  k<<<grid, ShShape<TS>::T, shared_smem(g, FORM, sl.rows, sl.blocks, ShShape<TS>::W), s>>>(g, p, sl);
}

template <typename TS, int D, int FORM>
void launch_form(const Geom& g, const DevPtrs& p, int splits, cudaStream_t s, bool prepare) {
  const bool out = any_outflow(g);
  if constexpr (sizeof(TS) != 8)
    if (window_eligible(g)) {
      launch_one<TS, D, FORM, true, false, true>(g, p, splits, s, prepare);
      return;
    }
  if constexpr (FORM == kFormP) {
    launch_one<TS, D, FORM, true, false>(g, p, splits, s, prepare);  // periodic, p = 1
  } else {
    if (g.p == 1 && !out) launch_one<TS, D, FORM, true, false>(g, p, splits, s, prepare);
    else if (g.p == 1) launch_one<TS, D, FORM, true, true>(g, p, splits, s, prepare);
    else if (!out) launch_one<TS, D, FORM, false, false>(g, p, splits, s, prepare);
    else launch_one<TS, D, FORM, false, true>(g, p, splits, s, prepare);
  }
}

template <typename TS>
void launch_ts(const Geom& g, const DevPtrs& p, int splits, int form, cudaStream_t s, bool prepare) {
  if (g.d == 2) {
    if (form == kFormFks) launch_form<TS, 2, kFormFks>(g, p, splits, s, prepare);
    else launch_form<TS, 2, kFormFull>(g, p, splits, s, prepare);
  } else {
    if (form == kFormFks) launch_form<TS, 3, kFormFks>(g, p, splits, s, prepare);
    else if (form == kFormP) {
      if constexpr (sizeof(TS) != 8) launch_form<TS, 3, kFormP>(g, p, splits, s, prepare);
    } else launch_form<TS, 3, kFormFull>(g, p, splits, s, prepare);
  }
}

void launch_shared_form(const Geom& g, const DevPtrs& p, int splits, int form, cudaStream_t s, bool prepare) {
  if (g.precision == DVM_F64) launch_ts<double>(g, p, splits, form, s, prepare);
  else if (g.precision == DVM_F32) launch_ts<float>(g, p, splits, form, s, prepare);
  else launch_ts<__nv_bfloat16>(g, p, splits, form, s, prepare);
}

}  // namespace

// 2D and 3D, with 32-bit byte offsets within a velocity, a grid within the
// launch limits and tables within the shared memory, where the 16-row columns are at least half full (a box flat in
// y wastes threads that the per-cell pass does not).
bool shared_eligible(const Geom& g) {
  if (g.d < 2 || g.nc >= (1LL << 28) || g.nx[2] > 65535 / kMaxSplits) return false;
  const long long ty = (g.nx[1] + kShTY - 1) / kShTY;
  return 2LL * g.nx[1] >= ty * kShTY && shape_of(g, 1).rows > 0;
}

// Velocity splits (ranges of the (kx, kz) pairs): the c <= 40 with the least
// estimated time of its CTAs, ceil(pairs / c) + 0.3 pairs long each (0.3 for the
// tables and partial sums).  Periodic: full waves of resident CTAs plus a last
// one of k per SM at (k / resident)^0.7 of the full rate.  Outflow (the CTAs at
// the boundary take longer) and FP64 (the Euler sub-steps beside it want the
// same pipe): the CTAs counted as spread evenly plus half a CTA.  Times half
// the partial sums' share of the traffic; where the tiles alone fill the chip
// many times over, c <= 4 (their memory); 2D periodic HOFKS c <= 6 p, for the step
// waits for the 1/p as many Euler sub-steps beside it and the CTAs take their
// SMs; 2D FP32 at least pairs / kShRun, for a split's sums are FP32 and the splits
// are added in FP64.  Step of the implosion 200^2 x 30^2, c = 5, 8, 15, 30: 339, 287, 253, 260
// us (with every value beyond the domain addressed by itself; 207 us at c = 10 since); FKS
// 200^2 x 20^2, c = 4, 7, 12: 65, 54, 63 us; FP64 HOFKS 100^2 x 40^2, c = 10, 20, 40:
// 1471, 1163, 1124 us; HOFKS 64^2 x 25^2, c = 6, 12, 25: 126, 135, 138 us.
int shared_splits(const Geom& g, int sms) {
  const long long tiles = ((long long)g.nx[0] * ((g.nx[1] + kShTY - 1) / kShTY) + 31) / 32 * g.nx[2];
  const int pairs = g.nv[0] * g.nv[2];
  const bool fks = g.scheme == DVM_FKS, f64 = g.precision == DVM_F64, even = f64 || any_outflow(g);
  const int per_sm = f64 ? 2 : (fks ? 4 : 3);
  int most = tiles >= 8LL * sms ? 4 : kMaxSplits;
  if (g.d == 2 && !fks && !even) most = std::min(most, 6 * g.p);
  const int least = g.d == 2 && !f64 ? (pairs + kShRun - 1) / kShRun : 1;
  static_assert(kMaxV1 <= kMaxSplits * kShRun, "every x axis can be split into short runs");
  int best = least;
  double cost = 1e30;
  for (int c = least; c <= std::max(most, least) && c <= pairs; ++c) {
    const long long slots = (long long)sms * per_sm, ctas = tiles * c, full = ctas / slots, rest = ctas % slots;
    const double k = (double)((rest + sms - 1) / sms) / per_sm;
    const double waves = even ? (double)ctas / slots + 0.5 : (double)full + (rest ? pow(k, 0.3) : 0.0);
    const double t = waves * ((pairs + c - 1) / c + 0.3) * (1.0 + (fks ? 1 : 2) * (g.d + 2) * c / (double)g.nvel);
    if (t < cost * 0.999) cost = t, best = c;
  }
  return best;
}

int shared_rows(const Geom& g) { return shape_of(g, 1).rows; }

void shared_prepare(const Geom& g) {
  DevPtrs none{};
  // the forms with and without the learned path
  Geom l = g;
  l.learn = 1;
  launch_shared_form(g, none, 1, form_of(g), nullptr, true);
  launch_shared_form(l, none, 1, form_of(l), nullptr, true);
}

void launch_shared(const Geom& g, const DevPtrs& p, int splits, cudaStream_t s) {
  launch_shared_form(g, p, splits, form_of(g), s, false);
}

}  // namespace dvm
