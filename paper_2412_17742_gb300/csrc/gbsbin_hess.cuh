// The Householder reflector shared by the reductions to Hessenberg form of the large-matrix tree
// (gbsbin_points_btree.cu) and of the reverse pass along it (gbsbin_backward_tree.cu).
#pragma once

#include <cuda_runtime.h>

#include "gbsbin_df.cuh"

namespace gbsbin {

// The reflector of x (squared norm nrm2, first entry x0): alpha = -e^{i arg x0} ||x|| and
// beta = 2 / ||x - alpha e_1||^2 = 1 / (||x||^2 + ||x|| |x0|).
template <class Ar>
__device__ __forceinline__ void reflector(typename Ar::E nrm2, typename Ar::E x0, typename Ar::E& alpha,
                                          typename Ar::E& beta) {
  using E = typename Ar::E;
  const E nrm = Ar::rsqrt_real(nrm2);
  const E ax0 = Ar::rsqrt_real(Ar::norm2(x0));
  alpha = Ar::re(ax0) > 0.f ? Ar::neg(Ar::mul(x0, Ar::mul(nrm, Ar::rrecip(ax0)))) : Ar::neg(nrm);
  beta = Ar::rrecip(Ar::add(nrm2, Ar::mul(nrm, ax0)));
}
// In FP64 by Newton steps on FP32 seeds, ~30 FP64 instructions instead of ~120 of square roots and divisions: one
// warp runs this once per column, and each of its FP64 instructions takes 64 clocks.
template <>
__device__ __forceinline__ void reflector<ArF64>(double2 nrm2, double2 x0, double2& alpha, double2& beta) {
  const double a = ::fma(x0.x, x0.x, x0.y * x0.y), b = nrm2.x;
  if (!(a > 1e-30 && b < 1e30)) {                    // beyond the seeds' range
    const double nrm = ::sqrt(b), ax = ::sqrt(a);
    alpha = ax > 0.0 ? make_double2(-x0.x / ax * nrm, -x0.y / ax * nrm) : make_double2(-nrm, 0.0);
    beta = make_double2(1.0 / ::fma(nrm, ax, b), 0.0);
    return;
  }
  double ra = (double)rsqrtf((float)a), rb = (double)rsqrtf((float)b);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    ra *= ::fma(-0.5 * a * ra, ra, 1.5);
    rb *= ::fma(-0.5 * b * rb, rb, 1.5);
  }
  const double nrm = b * rb, ax = a * ra, f = -nrm * ra;
  alpha = make_double2(f * x0.x, f * x0.y);
  const double d = ::fma(nrm, ax, b);
  double y = (double)__frcp_rn((float)d);
  y = ::fma(y, ::fma(-d, y, 1.0), y);
  y = ::fma(y, ::fma(-d, y, 1.0), y);
  beta = make_double2(y, 0.0);
}

}  // namespace gbsbin
