// The Householder reflector shared by the reductions to Hessenberg form of the large-matrix tree
// (gbsbin_points_btree.cu) and of the reverse pass along it (gbsbin_backward_tree.cu).
#pragma once

#include <cuda_runtime.h>

#include "gbsbin_df.cuh"

namespace gbsbin {

// The reflector of x (first entry x0, squared norm of the others rest > 0): alpha = -e^{i arg x0} ||x||, v0 = x0 - alpha
// and beta = 2 / ||v||^2 with ||v||^2 = rest + |v0|^2 from the rounded v0.  I - beta v v^H is then unitary to beta's own
// rounding, whatever alpha's error: from ||x||^2 + ||x|| |x0| beta carried the errors of two square roots and a product, which
// a hundred reflectors add up in every leaf of a parent alike (reverse pass at n = 200 in pairs, 20 states: relative
// error of dL/dT 3.8e-13, by Gauss-Jordan leaves 2.9e-13).
template <class Ar>
__device__ __forceinline__ void reflector(typename Ar::E rest, typename Ar::E x0, typename Ar::E& alpha,
                                          typename Ar::E& v0, typename Ar::E& beta) {
  using E = typename Ar::E;
  const E a = Ar::norm2(x0), nrm = Ar::rsqrt_real(Ar::add(rest, a)), ax0 = Ar::rsqrt_real(a);
  alpha = Ar::re(ax0) > 0.f ? Ar::neg(Ar::mul(x0, Ar::mul(nrm, Ar::rrecip(ax0)))) : Ar::neg(nrm);
  v0 = Ar::add(x0, Ar::neg(alpha));
  // 1 / d to pair rounding: s0 (1 + r + r^2), r = 1 - d s0 below 2^-23
  const E d = Ar::add(rest, Ar::norm2(v0));
  const float s0 = __frcp_rn(d.x), r = __fsub_rn(fmaf(-d.x, s0, 1.0f), __fmul_rn(d.z, s0));
  float h, l;
  fast_two_sum(s0, __fmul_rn(s0, fmaf(r, r, r)), h, l);
  beta = make_float4(2.0f * h, 0.f, 2.0f * l, 0.f);
}
// In FP64 by Newton steps on FP32 seeds, ~30 FP64 instructions instead of ~120 of square roots and divisions: one
// warp runs this once per column, and each of its FP64 instructions takes 64 clocks.
template <>
__device__ __forceinline__ void reflector<ArF64>(double2 rest, double2 x0, double2& alpha, double2& v0, double2& beta) {
  const double a = ::fma(x0.x, x0.x, x0.y * x0.y), b = rest.x + a;
  if (!(a > 1e-30 && b < 1e30)) {                    // beyond the seeds' range
    const double nrm = ::sqrt(b), ax = ::sqrt(a);
    alpha = ax > 0.0 ? make_double2(-x0.x / ax * nrm, -x0.y / ax * nrm) : make_double2(-nrm, 0.0);
    v0 = make_double2(x0.x - alpha.x, x0.y - alpha.y);
    beta = make_double2(2.0 / (rest.x + ::fma(v0.x, v0.x, v0.y * v0.y)), 0.0);
    return;
  }
  double ra = (double)rsqrtf((float)a), rb = (double)rsqrtf((float)b);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    ra *= ::fma(-0.5 * a * ra, ra, 1.5);
    rb *= ::fma(-0.5 * b * rb, rb, 1.5);
  }
  const double f = -b * rb * ra;
  alpha = make_double2(f * x0.x, f * x0.y);
  v0 = make_double2(x0.x - alpha.x, x0.y - alpha.y);
  const double d = rest.x + ::fma(v0.x, v0.x, v0.y * v0.y);
  double y = (double)__frcp_rn((float)d);
  y = ::fma(y, ::fma(-d, y, 1.0), y);
  y = ::fma(y, ::fma(-d, y, 1.0), y);
  beta = make_double2(2.0 * y, 0.0);
}

}  // namespace gbsbin
