// Heralded (conditional) states of a Gaussian state (arXiv:2412.17742, Sec. VII, Eqs.
// heralded_state_internal and lhaf_heralded_offd_internal_1), from the generating function.
//
// The modes are heralding (group l), traced or kept.  With lhaf(A_p, gamma_p) the p-th
// derivative of exp(xi^T A xi / 2 + gamma^T xi) at 0, the sum over the heralding and traced
// photon patterns with weights w^n / n! is the complex-Gaussian expectation of that
// exponential with xi = sqrt(w) (alpha, conj alpha) on those modes, and the kept modes' Fock
// indices (u on the first half, v on the second) are Taylor coefficients of the rest:
//
//   sum_{n, t} lhaf(A_{(n,t,u)+(n,t,v)}, ...) w^n / (n! t!) = u! v! [x^u y^v] F(w; x, y),
//   F = exp(xi_F^T M xi_F / 2 + l^T xi_F + e) / sqrt(det(I - X D(w) A_DD)),
//
// D the heralding and traced indices (both halves; w = 1 on traced modes), F the kept ones, and
// <v|rho(b)|u> = Pr(0) sqrt(u! v!) [w^b][x^u y^v] F.  M, l and e are what block elimination of the D rows
// of I - D(w) XA leaves in the kept rows: with the augmented form of the tree (gbsbin_tree.cuh) the Schur
// complement is A'_F = X_F M, its row u' = l and its corner 2 e, and the pivots' product the determinant.  So the
// points share eliminations like those of the binned tables: the traced rows go on the host once per
// state (w = 1), the first group by its spectral form for all roots of its axis in one launch (k_tree_root), and a
// CTA per point sweeps the other groups, from the first group's result of its root (or, where the first axis is so long
// that its results would not fit the plan's memory, all groups).  Then the Taylor
// coefficients of exp(xi^T M xi / 2 + l^T xi) by (p_i + 1) c_{p + e_i} = l_i c_p + sum_j M_ij c_{p - e_j}
// (shells of equal total degree in parallel, in shared memory, seven warps), while the eighth warp continues
// the elimination into the kept block - its Schur complement is I - A'_F - for the heralding probability's
// generating function (every non-heralding mode traced, w = 1 on the kept ones), and forms both factors
// exp(e) / sqrt(det) from the pivots' products by inverse roots (no logarithms).  FP64 throughout.
//
// What bounds it is the FP64 pipe of the points' SMs (a warp's FP64 instruction takes its scheduler 64
// clocks): every entry of a sweep is one multiply-add with its row's multiplier, where the elimination it
// replaces recomputed the multiplier per entry, solved back and added e on one thread.  16 ports x 2 internal modes,
// two groups of twelve modes, 81 points, 2401 coefficients each: 460 us before (425 of them the point stage, one
// elimination of 60 rows per point), 117 with the three launches here.
//
// The inverse DFT over the heralding grid: rho(b) is Hermitian, so only the channels u <= v are transformed and
// each is written with its conjugate; the first two axes in one launch through shared memory, sums over k and
// R - k folded (x_k + x_{R-k} times the cosine, x_k - x_{R-k} times the sine: half the multiplications).
#include <cuda_runtime.h>

#include "gbsbin_herald.h"
#include "gbsbin_tree.cuh"

namespace gbsbin {
namespace {

constexpr int HT = 256;
constexpr int TAYLOR_THREADS = HT - 32;
constexpr long long SMEM_COEF = 6144;                // coefficients kept in shared memory (96 KB)

// exp(x) P^{-1/2} for a pivots' record (product p 2^e2 with the sum of its factors' arguments), the root on the
// sheet of that sum.
__device__ double2 record_value(double2 p, float e2, float args, double2 x) {
  e2 += (float)ArF64::normalise(p);
  const int e = (int)e2, h = e >> 1;                  // e = 2 h + (e & 1)
  const int wind = (int)rintf((args - atan2f((float)p.y, (float)p.x)) * 0.159154943f);
  double2 v = inv_sqrt(p);
  double s = ldexp(exp(x.x), -h) * ((e & 1) ? 0.70710678118654752440 : 1.0);
  if (wind & 1) s = -s;
  if (x.y == 0.0) return make_double2(v.x * s, v.y * s);
  double sn, cs;
  sincos(x.y, &sn, &cs);
  return ArF64::mul(v, make_double2(s * cs, s * sn));
}

__device__ __forceinline__ void taylor_sync() { asm volatile("bar.sync 1, %0;" ::"n"(TAYLOR_THREADS) : "memory"); }

// DEEP: the sweep starts at the first group (no depth 1 in memory).
template <bool DEEP>
__global__ void __launch_bounds__(HT) k_herald_points(HeraldArgs a, TreeArgs t) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ double2 blk[(GBSBIN_HERALD_MAX_F + 1) * (GBSBIN_HERALD_MAX_F + 1)];   // [[A'_F, c'], [u', .]]
  __shared__ double2 fin[(GBSBIN_HERALD_MAX_F + 1) * (GBSBIN_HERALD_MAX_F + 1)];
  __shared__ double2 Mq[GBSBIN_HERALD_MAX_F * GBSBIN_HERALD_MAX_F], lq[GBSBIN_HERALD_MAX_F];
  __shared__ double2 s_pref;
  __shared__ PathRec<double2> s_rec;
  __shared__ double s_min;                            // the smallest pivot real part so far
  const long long k = blockIdx.x;
  const int nf = a.nf, f1 = nf + 1, tid = threadIdx.x;
  if (!DEEP && a.L == 1) {                            // the only group: its spectral form gives the kept block
    double2* d = reinterpret_cast<double2*>(sm_raw);
    double2* dB = d + t.nb[0];
    const double2 w = root_at<ArF64>(t, 0, (int)k);
    root_factors<ArF64>(t, w, d, dB);
    for (int q = tid; q < f1 * f1; q += HT) {
      const int i = q / f1, j = q - q / f1 * f1;
      blk[q] = (i < nf && j < nf) || t.has_gamma ? root_entry<ArF64>(t, dB, i, j) : ArF64::zero();
    }
    if (tid < 32) {
      const PathRec<double2> pr = root_path<ArF64>(t, w);
      if (tid == 0) s_rec = pr;                       // with the traced rows' exponent
    }
    if (tid == 32) s_min = fmin(a.tmin, 1.0 - fmax(w.x * a.lam_min, w.x * a.lam_max));
    __syncthreads();
    if (tid == 0) s_rec.ex = ArF64::add(s_rec.ex, blk[f1 * f1 - 1]);
  } else {
    constexpr int l0 = DEEP ? 0 : 1;
    const Sweep<double2> w = level_sweep<ArF64, false, GBSBIN_MAX_L - l0>(t, l0, a.L - l0, k, sm_raw);
    for (int q = tid; q < f1 * f1; q += HT) {
      const int i = q / f1, j = q - q / f1 * f1;
      blk[q] = (i < nf && j < nf) || t.has_gamma ? w.G[(w.nb + i) * w.cols + w.nb + j] : ArF64::zero();
    }
    if (tid < 32) {
      const PathRec<double2> pr = sweep_path<ArF64, false>(t, l0, w);
      if (tid == 0) s_rec = pr;
    } else if (tid < 64) {                            // (the record's smallest pivot is FP32)
      double mn = a.tmin;
      if (!DEEP) {
        const double2 r = root_at<ArF64>(t, 0, (int)w.parent);
        mn = fmin(mn, 1.0 - fmax(r.x * a.lam_min, r.x * a.lam_max));
      }
      for (int q = tid - 32; q < w.nb; q += 32) {
        const double2 z = w.pivots[q];
        mn = z.x == z.x && z.y == z.y ? fmin(mn, z.x) : -1.0e300;
      }
      for (int o = 16; o > 0; o >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      if (tid == 32) s_min = mn;
    }
  }
  __syncthreads();
  const PathRec<double2> rec = s_rec;
  const int h = nf / 2;
  for (int q = tid; q < nf * nf; q += HT) {           // M = X_F A'_F, l = u'
    const int i = q / nf, j = q - q / nf * nf;
    Mq[q] = blk[(i < h ? i + h : i - h) * f1 + j];
  }
  if (tid < nf) lq[tid] = blk[nf * f1 + tid];
  // the coefficients in the sweep's memory (done with), or in the point's slot
  double2* slot = a.gcoef + (size_t)k * (a.ncoef + 1);
  double2* C = a.ncoef <= SMEM_COEF ? reinterpret_cast<double2*>(sm_raw) : slot;
  if (tid == 0) C[0] = ArF64::one();
  __syncthreads();
  if (tid >= TAYLOR_THREADS) {                        // the eighth warp: the scalar factors
    const int lane = tid & 31;
    for (int q = lane; q < f1 * f1; q += 32) {        // [[I - A'_F, c'], [-u', 2 e]]
      const int i = q / f1, j = q - q / f1 * f1;
      double2 v = blk[q];
      if (i < nf && j < nf) {
        v = ArF64::neg(v);
        if (i == j) v.x += 1.0;
      } else if (i == nf) {
        v = j == nf ? rec.ex : ArF64::neg(v);
      }
      fin[q] = v;
    }
    __syncwarp();
    double2 prod = rec.prod;
    float e2 = rec.meta.y, args = rec.meta.x;
    double mn = s_min;
    for (int c = 0; c < nf; ++c) {
      const double2 piv = fin[c * f1 + c], r = ArF64::recip(piv);
      prod = ArF64::mul(prod, piv);
      e2 += (float)ArF64::normalise(prod);
      args += atan2f((float)piv.y, (float)piv.x);
      mn = piv.x == piv.x && piv.y == piv.y ? fmin(mn, piv.x) : -1.0e300;
      const int n1 = nf - c;
      for (int q = lane; q < n1 * n1; q += 32) {
        const int i = c + 1 + q / n1, j = c + 1 + q - q / n1 * n1;
        fin[i * f1 + j] = ArF64::fms(fin[i * f1 + j], ArF64::mul(fin[i * f1 + c], r), fin[c * f1 + j]);
      }
      __syncwarp();
    }
    // lane 0: exp(e) / sqrt(det); lane 1: the heralding probability's value; one pass of the same code
    if (lane < 2) {
      const double2 x = lane ? fin[f1 * f1 - 1] : rec.ex;
      const double2 v = record_value(lane ? prod : rec.prod, lane ? e2 : rec.meta.y, lane ? args : rec.meta.x,
                                     make_double2(0.5 * x.x, 0.5 * x.y));
      if (lane) {
        slot[a.ncoef] = v;
        a.minpiv[k] = isfinite(v.x) && isfinite(v.y) ? mn : -1.0e300;
      } else {
        s_pref = v;
      }
    }
  } else {                                            // Taylor coefficients by shells, relative to the first
    for (int sh = 1; sh <= nf * a.cut; ++sh) {
      const int t1 = a.shell[sh + 1];
      for (int e = a.shell[sh] + tid; e < t1; e += TAYLOR_THREADS) {
        const int i0 = a.ti0[e];
        double2 val = ArF64::mul(lq[i0], C[a.tqm[e]]);
        const int* nb = a.tnb + (size_t)e * nf;
        for (int j = 0; j < nf; ++j)
          if (nb[j] >= 0) val = ArF64::fma(Mq[i0 * nf + j], C[nb[j]], val);
        const double p = (double)a.tp[e];
        double inv = (double)__frcp_rn((float)p);     // 1 / p: an exact small integer, two Newton steps
        inv = fma(inv, fma(-p, inv, 1.0), inv);
        inv = fma(inv, fma(-p, inv, 1.0), inv);
        C[a.tq[e]] = make_double2(val.x * inv, val.y * inv);
      }
      taylor_sync();
    }
  }
  __syncthreads();
  const double2 pref = s_pref;
  for (long long q = tid; q < a.ncoef; q += HT) slot[q] = ArF64::mul(pref, C[q]);
}

// ------------------------------------------------------------------------------ inverse DFT
// Sum over k < R of x_k exp(-2 pi i k b / R) from folded values at stride st: entry k holds x_k + x_{R-k} and entry
// R - k holds x_k - x_{R-k} (0 < k < R/2); entries 0 and R/2 as they are.
__device__ __forceinline__ double2 folded_sum(const double2* x, int st, int R, int b, const double2* __restrict__ tw) {
  double2 acc = x[0];
  if ((R & 1) == 0) {
    const double2 y = x[(R / 2) * st];
    acc = (b & 1) ? make_double2(acc.x - y.x, acc.y - y.y) : make_double2(acc.x + y.x, acc.y + y.y);
  }
  int idx = b;
  for (int k = 1; 2 * k < R; ++k) {
    const double2 s = x[k * st], d = x[(R - k) * st], w = tw[idx];   // w = (cos, -sin)
    acc.x = fma(w.x, s.x, fma(-w.y, d.y, acc.x));
    acc.y = fma(w.x, s.y, fma(w.y, d.x, acc.y));
    idx += b;
    if (idx >= R) idx -= R;
  }
  return acc;
}

// A finished entry of channel c (position in the list) at heralding outcome `cell`: rho and its mirror image, or
// Pr(b).
__device__ __forceinline__ void write_channel(const HeraldArgs& a, long long cell, int c, double2 v,
                                              double2* __restrict__ rho, double* __restrict__ prob) {
  const double s = a.pr0 / (double)a.npts;
  if (c == a.nchan - 1) {
    prob[cell] = v.x * s;
    a.prob_own[cell] = v.x * s;
    return;
  }
  const int ch = a.chan[c], u = ch / a.side, w = ch - u * a.side;
  const double f = s * a.chscale[ch];
  double2* r = rho + cell * a.ncoef;
  v = make_double2(v.x * f, u == w ? 0.0 : v.y * f);
  r[ch] = v;
  if (u != w) r[w * a.side + u] = make_double2(v.x, -v.y);
}

// Folds R entries at stride st in place, for each of n lines (base(line)), by the whole CTA.
template <class Base>
__device__ __forceinline__ void fold_lines(double2* X, int n, int R, int st, Base base) {
  const int half = (R - 1) / 2;
  for (int q = threadIdx.x; q < n * half; q += blockDim.x) {
    const int line = q / half, k = 1 + q - q / half * half;
    double2* x = X + base(line);
    const double2 p = x[k * st], m = x[(R - k) * st];
    x[k * st] = make_double2(p.x + m.x, p.y + m.y);
    x[(R - k) * st] = make_double2(p.x - m.x, p.y - m.y);
  }
}

// The first two axes: CTA = (index of the later axes, block of CB channels); in: the points' slots, out (when axes
// follow): [b_0][b_1][later][channel].
__global__ void __launch_bounds__(HT) k_herald_dft2(HeraldArgs a, int CB, long long later, double2* __restrict__ out,
                                                    double2* __restrict__ rho, double* __restrict__ prob) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int R0 = a.radix[0], R1 = a.radix[1], n0 = a.nout[0], n1 = a.nout[1];
  double2* X = reinterpret_cast<double2*>(sm_raw);    // [k0][k1][cb]
  double2* Y = X + (size_t)R0 * R1 * CB;              // [k0][b1][cb]
  const int blocks = (a.nchan + CB - 1) / CB;
  const long long p = blockIdx.x / blocks;
  const int c0 = (int)(blockIdx.x - p * blocks) * CB;
  for (int q = threadIdx.x; q < R0 * R1 * CB; q += HT) {
    const int cb = q % CB, kk = q / CB, c = c0 + cb;
    X[q] = c < a.nchan ? a.gcoef[((long long)kk * later + p) * (a.ncoef + 1) + (c == a.nchan - 1 ? a.ncoef : a.chan[c])]
                       : make_double2(0.0, 0.0);
  }
  __syncthreads();
  fold_lines(X, R0 * CB, R1, CB, [=](int line) { return line / CB * R1 * CB + line % CB; });
  __syncthreads();
  for (int q = threadIdx.x; q < R0 * n1 * CB; q += HT) {
    const int cb = q % CB, r = q / CB, b1 = r % n1, k0 = r / n1;
    Y[q] = folded_sum(X + (size_t)k0 * R1 * CB + cb, CB, R1, b1, a.tw + R0);
  }
  __syncthreads();
  fold_lines(Y, n1 * CB, R0, n1 * CB, [](int line) { return line; });
  __syncthreads();
  for (int q = threadIdx.x; q < n0 * n1 * CB; q += HT) {
    const int cb = q % CB, r = q / CB, b1 = r % n1, b0 = r / n1, c = c0 + cb;
    if (c >= a.nchan) continue;
    const double2 v = folded_sum(Y + (size_t)b1 * CB + cb, n1 * CB, R0, b0, a.tw);
    if (a.L == 2) write_channel(a, (long long)b0 * n1 + b1, c, v, rho, prob);
    else out[(((long long)b0 * n1 + b1) * later + p) * a.nchan + c] = v;
  }
}

// One axis: out[pre][b][post][c] = sum over k < R_l of in[pre][k][post][c] exp(-2 pi i k b / R_l), b < nout_l (pre
// runs over the axes already transformed, post over the later ones, c over the channels); slots: the input is the
// points' slots, every channel.  One thread per output element, consecutive threads on consecutive channels.
__global__ void k_herald_dft_axis(HeraldArgs a, int l, int slots, const double2* __restrict__ in,
                                  double2* __restrict__ out, double2* __restrict__ rho, double* __restrict__ prob) {
  long long pre = 1, post = 1;
  for (int q = 0; q < l; ++q) pre *= a.nout[q];
  for (int q = l + 1; q < a.L; ++q) post *= a.radix[q];
  const int R = a.radix[l], nb = a.nout[l];
  int off = 0;
  for (int q = 0; q < l; ++q) off += a.radix[q];
  const long long total = pre * nb * post * a.nchan, nch = slots ? a.ncoef + 1 : a.nchan;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    long long rest = t;
    const int c = (int)(rest % a.nchan);
    rest /= a.nchan;
    const long long pi = rest % post;
    rest /= post;
    const int b = (int)(rest % nb);
    const long long pr = rest / nb;
    const long long ch = !slots ? c : c == a.nchan - 1 ? a.ncoef : a.chan[c];
    const double2* src = in + ((pr * R) * post + pi) * nch + ch;
    const long long step = post * nch;
    double2 acc = make_double2(0.0, 0.0);
    int idx = 0;                                      // k b mod R, advanced by b per k
    for (int k = 0; k < R; ++k) {
      acc = ArF64::fma(src[(long long)k * step], a.tw[off + idx], acc);
      idx += b;
      if (idx >= R) idx -= R;
    }
    if (l + 1 < a.L) out[((pr * nb + b) * post + pi) * a.nchan + c] = acc;
    else write_channel(a, pr * nb + b, c, acc, rho, prob);   // post = 1 on the last axis
  }
}

}  // namespace

size_t herald_sweep_smem(int L, int nb0, int m1, bool deep) {
  if (deep) return tree_level_smem_bytes(nb0 + m1, nb0 + m1);
  if (L == 1) return sizeof(double2) * (size_t)nb0 * (m1 + 2);
  return tree_level_smem_bytes(m1, m1);
}

cudaError_t launch_herald(const HeraldArgs& a, const TreeArgs& t, int num_sms, double2* out, double* prob,
                          cudaStream_t s, int* launches) {
  cudaError_t err = cudaSuccess;
  *launches = 0;
  const bool deep = a.L > 1 && !t.A[1];
  if (a.L > 1 && !deep) {
    if ((err = launch_tree_root_fp64(t, num_sms, s)) != cudaSuccess) return err;
    ++*launches;
  }
  const size_t sweep = herald_sweep_smem(a.L, t.nb[0], t.m[1], deep);
  const size_t coef = a.ncoef <= SMEM_COEF ? sizeof(double2) * (size_t)a.ncoef : 0, smem = sweep > coef ? sweep : coef;
  auto points = deep ? k_herald_points<true> : k_herald_points<false>;
  if (smem > 32 * 1024 &&
      (err = cudaFuncSetAttribute(points, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return err;
  points<<<(unsigned)a.npts, HT, smem, s>>>(a, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  ++*launches;
  int l = 0;
  long long pre = 1;
  const double2* in = a.gcoef;
  if (a.L > 1) {                                      // two axes at once where a block of channels fits 96 KB
    const long long cell = (long long)a.radix[0] * (a.radix[1] + a.nout[1]);
    const int CB = (int)(cell < 6144 ? 6144 / cell : 0);
    if (CB >= 1) {
      const int cb = CB > 8 ? 8 : CB;
      long long later = 1;
      for (int q = 2; q < a.L; ++q) later *= a.radix[q];
      const size_t sm = sizeof(double2) * (size_t)cell * cb;
      if (sm > 48 * 1024 &&
          (err = cudaFuncSetAttribute(k_herald_dft2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)) != cudaSuccess)
        return err;
      const long long blocks = later * ((a.nchan + cb - 1) / cb);
      k_herald_dft2<<<(unsigned)blocks, HT, sm, s>>>(a, cb, later, a.scratch, out, prob);
      if ((err = cudaGetLastError()) != cudaSuccess) return err;
      ++*launches;
      in = a.scratch;
      pre = (long long)a.nout[0] * a.nout[1];
      l = 2;
    }
  }
  // the other axes one by one, ping-pong between the slots and the scratch buffer (each output is at most as
  // large as its input)
  for (; l < a.L; ++l) {
    long long post = 1;
    for (int q = l + 1; q < a.L; ++q) post *= a.radix[q];
    const long long work = pre * a.nout[l] * post * a.nchan;
    long long blocks = (work + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    double2* o = (in == a.gcoef) ? a.scratch : a.gcoef;
    k_herald_dft_axis<<<(unsigned)blocks, 256, 0, s>>>(a, l, l == 0 ? 1 : 0, in, o, out, prob);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    ++*launches;
    in = o;
    pre *= a.nout[l];
  }
  return cudaSuccess;
}

}  // namespace gbsbin
