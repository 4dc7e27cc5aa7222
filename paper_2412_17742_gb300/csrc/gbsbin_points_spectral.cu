// One detector group (arXiv:2412.17742, Sec. VIII, total photon-number distribution; Sec. III
// Eq. q_d with a single group): D(w) = w I, and XA = I - Sigma^{-1} is Hermitian, so
//
//   K(w) = I - w XA = Q (I - w Lambda) Q^H,  XA = Q Lambda Q^H with Lambda real,
//   log det K(w) = sum_i Log(1 - w lambda_i),
//   gamma^T K(w)^{-1} w X gamma = sum_i g_i w / (1 - w lambda_i),  g_i = (Q^T gamma)_i (Q^H X gamma)_i.
//
// The host diagonalises XA once per state (gbsbin_host_eigen.cpp).  Every |lambda_i| < 1, so each
// factor has a positive real part and the sum of principal logarithms is the branch continuous
// from w = 0.  A grid point costs O(n): TP lanes share the n factors, each multiplying its own (the
// exponent taken out every fourth factor, the arguments summed in FP32, which fixes the winding
// of the product's logarithm), then a butterfly.  G = q(w)/q(1) is formed from the product itself,
// sqrt(prod (1 - lambda_i) / prod (1 - w lambda_i)) times exp of the displacement terms'
// difference, so no logarithm of the size of log q is rounded on the way.
//
// All of it is FP64, for plans of either arithmetic: at n = 512 and 86 points it is 44,000
// factors of ~8 FP64 operations, which 152 SMs at 2 operations a clock finish in ~1200 clocks.
// What bounds a launch is the FP64 latency of one warp's chain (n / TP factors, the butterfly, the root) on
// small grids and the FP64 rate on large ones, so a point takes a CTA or a warp while that leaves SMs to
// fill and one thread on large grids, where a warp then takes the roots of 32 points at once.  Before, a CTA or warp per point eliminated the Hessenberg
// form of XA, n serial steps of O(n): 614 us at n = 512 with 86 points in FP64. The whole
// table, transform included, took 642 us and takes 18.5 us, 17.6 of them on the host's side of the call.
#include <cuda_runtime.h>

#include "gbsbin_device.cuh"
#include "gbsbin_df.cuh"
#include "gbsbin_internal.h"

namespace gbsbin {
namespace {

constexpr int kSpectralThreads = 128;

struct Partial {                                // a share of the factors
  double2 prod, ex;
  int e2;
  float args;
};

__device__ __forceinline__ void join(Partial& p, const Partial& q, bool disp) {
  p.prod = ArF64::mul(p.prod, q.prod);
  p.e2 += q.e2 + ArF64::normalise(p.prod);
  p.args += q.args;
  if (disp) p.ex = ArF64::add(p.ex, q.ex);
}

// One point by TP consecutive threads (thread r of the team; TP = kSpectralThreads: the whole CTA, through
// shared memory); every thread of the block calls it, teams past the last point with live = false.
template <int TP, bool DISP>
__device__ __forceinline__ void spectral_point(const PointArgs& a, long long e, int r, bool live) {
  const double2 w = grid_root(a.tw, a.grid, 0, live ? point_digit(e, a.grid, 0) : 0);
  const double rt0 = a.sp[0], e0 = a.sp[1], lam_min = a.sp[4], lam_max = a.sp[5];   // (the loads pass under the product)
  const double2 ex0 = make_double2(a.sp[2], a.sp[3]);
  Partial p{ArF64::one(), ArF64::zero(), 0, 0.f};
  int since = 0;
  for (int i = r; i < a.n; i += TP) {
    const double lam = a.lam[i];
    const double2 z = make_double2(fma(-w.x, lam, 1.0), -w.y * lam);
    p.prod = ArF64::mul(p.prod, z);
    p.args += atan2f((float)z.y, (float)z.x);
    if (++since == 4) {                         // |z| < 2 and > 1 - |lambda|
      p.e2 += ArF64::normalise(p.prod);
      since = 0;
    }
    if (DISP) p.ex = ArF64::fma(a.gq[i], ArF64::recip(z), p.ex);
  }
  p.e2 += ArF64::normalise(p.prod);
#pragma unroll
  for (int o = (TP < 32 ? TP : 32) / 2; o > 0; o >>= 1) {
    Partial q;
    q.prod = shfl_xor(p.prod, o);
    q.e2 = __shfl_xor_sync(0xffffffffu, p.e2, o);
    q.args = __shfl_xor_sync(0xffffffffu, p.args, o);
    if (DISP) q.ex = shfl_xor(p.ex, o);
    join(p, q, DISP);
  }
  if constexpr (TP > 32) {
    __shared__ Partial s_p[TP / 32];
    if ((threadIdx.x & 31) == 0) s_p[threadIdx.x >> 5] = p;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int i = 1; i < TP / 32; ++i) join(p, s_p[i], DISP);
  }
  if (!live || r != 0) return;
  const double2 prod = p.prod;
  const int e2 = p.e2;
  const double2 ex = DISP ? ArF64::mul(p.ex, w) : ArF64::zero();   // gamma^T K^{-1} w X gamma
  // every factor's real part is 1 - Re(w) lambda_i: the smallest at an end of the spectrum
  const double mn = 1.0 - fmax(w.x * lam_min, w.x * lam_max);
  const bool ok = isfinite(prod.x) && isfinite(prod.y) && isfinite(ex.x) && isfinite(ex.y);
  const double LN2 = 0.693147180559945309417232121458;
  double* f = a.ldfin + 6 * e;                  // log q unfinished, as finish_logq takes it
  f[0] = prod.x;
  f[1] = prod.y;
  f[2] = (double)p.args;
  f[3] = fma(-0.5 * LN2, (double)e2, 0.5 * ex.x);
  f[4] = 0.5 * ex.y;
  f[5] = 0.0;
  a.minpiv[e] = ok ? mn : -1.0e300;
  if (!a.gout) return;
  // G = (p0 2^e0 / (prod 2^e2))^{1/2} exp((ex - ex(1)) / 2), the root on the sheet of the summed
  // arguments: the principal root times (-1)^m, m the winding of log prod
  const float a0 = atan2f((float)prod.y, (float)prod.x);
  const int m = (int)rintf((p.args - a0) * 0.159154943f);
  double2 g = inv_sqrt(prod);
  const int de = (int)e0 - e2, h = de >> 1;     // 2^(de / 2) = 2^h sqrt(2)^(de odd)
  double sc = rt0 * ((de & 1) ? 1.41421356237309504880 : 1.0);
  if (m & 1) sc = -sc;
  sc = ldexp(sc, h);
  g = make_double2(g.x * sc, g.y * sc);
  if (DISP) {
    double sn, cs;
    sincos(0.5 * (ex.y - ex0.y), &sn, &cs);
    const double m2 = exp(0.5 * (ex.x - ex0.x));
    g = ArF64::mul(g, make_double2(m2 * cs, m2 * sn));
  }
  a.gout[e] = g;
}

template <int TP, bool DISP>
__global__ void __launch_bounds__(kSpectralThreads) k_points_spectral(PointArgs a) {
  const long long e = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / TP;
  spectral_point<TP, DISP>(a, e, threadIdx.x % TP, e < a.grid.n_eval);
}

// A batch: block j takes the points e0 .. e0 + GBSBIN_SPECTRAL_BATCH_POINTS - 1 of its job's problem.
constexpr int kBatchTP = kSpectralThreads / GBSBIN_SPECTRAL_BATCH_POINTS;
__global__ void __launch_bounds__(kSpectralThreads) k_points_spectral_batch(PointBatch b) {
  const PointJob job = b.jobs[blockIdx.x];
  const PointArgs& a = b.probs[job.prob];
  const long long e = job.e0 + threadIdx.x / kBatchTP;
  const bool live = e < a.grid.n_eval;
  if (a.has_gamma) spectral_point<kBatchTP, true>(a, e, threadIdx.x % kBatchTP, live);
  else spectral_point<kBatchTP, false>(a, e, threadIdx.x % kBatchTP, live);
}

template <int TP>
cudaError_t launch_tp(const PointArgs& a, int threads, cudaStream_t s) {
  const long long per = threads / TP;
  const unsigned grid = (unsigned)((a.grid.n_eval + per - 1) / per);
  if (a.has_gamma) k_points_spectral<TP, true><<<grid, threads, 0, s>>>(a);
  else k_points_spectral<TP, false><<<grid, threads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_points_spectral(const PointArgs& a, int num_sms, cudaStream_t s) {
  // threads per point.  A CTA (four warps) each for long products on few points: a warp's chain of n / 32
  // factors, not the FP64 rate, is the time then (n = 512, 86 points: 21 us with a warp per point).  A
  // warp each, one to a CTA so that the points spread over the SMs, while every SM gets at most eight;
  // then eight lanes, then one.
  const long long pts = a.grid.n_eval;
  if (a.n >= 128 && pts <= 4LL * num_sms) return launch_tp<kSpectralThreads>(a, kSpectralThreads, s);
  if (pts <= 8LL * num_sms) return launch_tp<32>(a, 32, s);
  if (pts <= 64LL * num_sms) return launch_tp<8>(a, kSpectralThreads, s);
  return launch_tp<1>(a, kSpectralThreads, s);
}

cudaError_t launch_points_spectral_batch(const PointBatch& batch, cudaStream_t s) {
  k_points_spectral_batch<<<(unsigned)batch.njobs, kSpectralThreads, 0, s>>>(batch);
  return cudaGetLastError();
}

}  // namespace gbsbin
