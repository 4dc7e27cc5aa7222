// Device code of the tree of block eliminations shared by the small tree (gbsbin_points_tree.cu) and the heralded
// states (gbsbin_herald.cu): path records, the first level from the spectral form of the first group's block,
// and the elimination sweep of the later levels.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "gbsbin_device.cuh"
#include "gbsbin_df.cuh"
#include "gbsbin_internal.h"

namespace gbsbin {
namespace {

constexpr int LT_MAX = 512;      // threads of a level CTA (at most)
constexpr int SPAN_MAX = 4;      // groups one level launch may eliminate

// Path record of a node (48 bytes in both arithmetics): the pivot product scaled by a power
// of two; (FP32 argument sum, power of two, smallest pivot real part, -); the exponent sum.
template <class E>
struct PathRec {
  E prod;
  float4 meta;
  E ex;
};
static_assert(sizeof(PathRec<float4>) == 3 * sizeof(float4) && sizeof(PathRec<double2>) == 3 * sizeof(float4),
              "path records are three 16-byte slots");

template <class Ar>
__device__ __forceinline__ PathRec<typename Ar::E>* path_at(float4* base, long long node) {
  return reinterpret_cast<PathRec<typename Ar::E>*>(base + 3 * node);
}
template <class Ar>
__device__ __forceinline__ typename Ar::E* elem(float4* p) {
  return reinterpret_cast<typename Ar::E*>(p);
}

// w = exp(2 pi i k / R_l): from the pairs-of-FP32 table for ArDF (no FP64 conversion), else
// from the FP64 twiddles
template <class Ar>
__device__ __forceinline__ typename Ar::E root_at(const TreeArgs& a, int l, int k) {
  if constexpr (std::is_same<Ar, ArDF>::value) {
    int off = 0;
    for (int q = 0; q < l; ++q) off += a.grid.radix[q];
    return a.twdf[off + k];
  } else {
    return Ar::from(grid_root(a.tw, a.grid, l, k));
  }
}

// The path record after a set of pivots, by one full warp: lane t holds pivot t of the set
// (count <= span, a power of two <= 32; lanes beyond hold 1).  Product by a butterfly of
// pair products over aligned groups of span lanes (each level rescaled by a power of two),
// argument sum and smallest real part by butterflies too.  pr: the parent's record on
// input, the child's on output (every lane of the first group; all lanes when span = 32).
template <class Ar>
__device__ __forceinline__ void path_warp(PathRec<typename Ar::E>& pr, typename Ar::E piv, bool real, int span) {
  using E = typename Ar::E;
  E p = real ? piv : Ar::one();
  const float pre = Ar::re(piv), pim = Ar::im(piv);
  float arg = real ? atan2f(pim, pre) : 0.f;
  float mn = real ? pre : 3.0e38f;
  if (real && (!(pre == pre) || !(pim == pim))) mn = -3.0e38f;
  float e2 = 0.f;
  for (int o = span >> 1; o > 0; o >>= 1) {
    p = Ar::mul(p, shfl_xor(p, o));
    e2 += __shfl_xor_sync(0xffffffffu, e2, o);
    e2 += (float)Ar::normalise(p);
    arg = __fadd_rn(arg, __shfl_xor_sync(0xffffffffu, arg, o));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  // every lane now holds the same product, exponent, sum and minimum; fold in the parent
  E q = Ar::mul(pr.prod, p);
  const float e = pr.meta.y + e2 + (float)Ar::normalise(q);
  pr.prod = q;
  pr.meta = make_float4(__fadd_rn(pr.meta.x, arg), e, fminf(pr.meta.z, mn), 0.f);
}

// Level 0 from the spectral form of the first group's block.  XA is Hermitian, so A_00 = Q Lambda Q^H and
// W = w (I - w A_00)^-1 A_0r = Q diag(d) Q^H A_0r with d_k = w / (1 - w lambda_k): every entry of the child's
//   A' = A_rr + sum_k conj(B_ki) d_k B_kj,  c' = c_r + sum_k conj(B_ki) d_k b_k,
//   u' = u_r + sum_k q_k d_k B_kj,          exponent sum_k q_k d_k b_k
// (B = Q^H A_0r, b = Q^H c_0, q = u_0^T Q) is a sum of nb products of its own, where the elimination it
// replaces is nb steps with a barrier and a reciprocal each on as many SMs as the axis has roots.  The
// pivots' product is prod (1 - w lambda_k), each factor with Re > 0.  CTA (child, part): part of the child's
// rows, their left factors times d in shared memory.  n = 42, 14 rows per group, FP64: the levels took
// 53 us in one elimination of both, and take 11 (this launch) + 23.
// Where a level's CTAs are few and the sums cheap, the next level's launch forms its parents' entries itself
// (k_tree_level<Ar, true>).
constexpr int ROOT_THREADS = 256;

// d (nb) and d B (nb x X) of the root w in shared memory, by the whole CTA.
template <class Ar>
__device__ __forceinline__ void root_factors(const TreeArgs& a, typename Ar::E w, typename Ar::E* d, typename Ar::E* dB) {
  const int nb = a.nb[0], X = a.m[1] + 1;
  const typename Ar::E* lam = elem<Ar>(const_cast<float4*>(a.rlam));
  const typename Ar::E* B = elem<Ar>(const_cast<float4*>(a.rB));
  for (int k = threadIdx.x; k < nb; k += blockDim.x)
    d[k] = Ar::mul(w, Ar::recip(Ar::add(Ar::one(), Ar::neg(Ar::mul(w, lam[k])))));
  __syncthreads();
  for (int q = threadIdx.x; q < nb * X; q += blockDim.x) dB[q] = Ar::mul(d[q / X], B[q]);
  __syncthreads();
}

// Entry (i, j) of the child's augmented matrix: row mc is u', column mc is c', (mc, mc) the exponent.
template <class Ar>
__device__ __forceinline__ typename Ar::E root_entry(const TreeArgs& a, const typename Ar::E* dB, int i, int j) {
  using E = typename Ar::E;
  const int nb = a.nb[0], mc = a.m[1], X = mc + 1;
  const bool urow = i == mc, ccol = j == mc;
  E acc = urow ? (ccol ? Ar::zero() : elem<Ar>(a.u[0])[nb + j])
               : ccol ? elem<Ar>(a.c[0])[nb + i] : elem<Ar>(a.A[0])[(nb + i) * a.m[0] + nb + j];
  const E* left = urow ? elem<Ar>(const_cast<float4*>(a.ru)) : elem<Ar>(const_cast<float4*>(a.rB)) + i;
  const int step = urow ? 1 : X;
  E odd = Ar::zero();                                  // two chains
  int k = 0;
#pragma unroll 2
  for (; k + 2 <= nb; k += 2) {
    const E x = left[k * step], y = left[(k + 1) * step];
    acc = Ar::fma(urow ? x : Ar::conj(x), dB[k * X + j], acc);
    odd = Ar::fma(urow ? y : Ar::conj(y), dB[(k + 1) * X + j], odd);
  }
  if (k < nb) {
    const E x = left[k * step];
    acc = Ar::fma(urow ? x : Ar::conj(x), dB[k * X + j], acc);
  }
  return Ar::add(acc, odd);
}

// The first level's path record of the root w (its exponent apart), by one full warp.
template <class Ar>
__device__ __forceinline__ PathRec<typename Ar::E> root_path(const TreeArgs& a, typename Ar::E w) {
  using E = typename Ar::E;
  const int nb = a.nb[0], lane = threadIdx.x & 31;
  const E* lam = elem<Ar>(const_cast<float4*>(a.rlam));
  PathRec<E> pr = *path_at<Ar>(a.path[0], 0);
  int width = 1;
  while (width < nb && width < 32) width <<= 1;
  for (int t0 = 0; t0 < nb; t0 += 32) {
    const int t = t0 + lane;
    const E z = t < nb ? Ar::add(Ar::one(), Ar::neg(Ar::mul(w, lam[t]))) : Ar::zero();
    path_warp<Ar>(pr, z, t < nb, width);
  }
  return pr;
}

// Level l: one CTA per child (parent, k) of depth l.  Forward elimination of the nb pivot
// columns of the (m + 1) x (m + 1) augmented matrix
//
//   [ B      | w A_0r | w c_0 ]
//   [ -A_r0  | A_rr   | c_r   ]
//   [ -u_0^T | u_r^T  | 0     ]
//
// leaves the child's A' and c' in the middle rows and (u'^T | u_0^T y) in the last row:
// eliminating block 0 from a row [a_0 | a_r] gives a_r - a_0 B^-1 [w A_0r | w c_0].  Rows
// are never scaled (only the Schur complement is needed): step kk subtracts
// (G[i][kk] / G[kk][kk]) row kk from every row i > kk, each entry one fused multiply-subtract
// with its row's multiplier.  The multipliers run one step ahead: in step kk warp 0 updates
// column kk + 1 and then forms pivot kk + 1's reciprocal (every lane) and step kk + 1's
// multipliers, while warps 1.. update the columns right of it - one barrier per step, the
// hand-off off the critical path.  After the sweep warp 0 forms the child's path record
// while the other warps copy out the child's matrix and vectors.
//
// A launch may eliminate span consecutive groups l .. l + span - 1 at once (a node of depth
// l + span from its ancestor at depth l): the leading block is then those groups' rows, each
// pivot row scaled by its own group's root, and the Schur complement of that block is the
// same A'' as after span single-group sweeps (eliminating block 0 and then block 1 of the
// first Schur complement is eliminating [0 1] at once), with the same pivots.
// (48 registers: five 256-thread CTAs per SM, so a 729-CTA level runs in one wave)
// ROOT (l = 1): the parents are not read but formed from the first group's spectral form while the matrix is
// filled.  MS: the most groups (span) an instance takes.  The whole CTA calls it for one child; on return G holds the trailing block (row and column nb + i) and
// sweep.pivots the nb pivots, after a block barrier.
template <class E>
struct Sweep {
  E* G;                                              // rows x cols
  E* pivots;
  int nb, m, cols, rows;                             // m: rows before the sweep
  long long parent;
  void* root_path;                                   // ROOT: the root's record in shared memory
};
template <class Ar, bool ROOT, int MS>
__device__ __forceinline__ Sweep<typename Ar::E> level_sweep(const TreeArgs& a, int l, int span, long long child, void* smem) {
  using E = typename Ar::E;
  // the child's roots, last merged axis fastest in its index, and the pivot-row bounds
  E wg[MS];
  int bound[MS];
  long long rest = child;
  int nb = 0;
#pragma unroll
  for (int g = MS - 1; g >= 0; --g) {
    if (g < span) {
      const int R = a.grid.radix[l + g];
      const long long up = rest / R;
      wg[g] = root_at<Ar>(a, l + g, (int)(rest - up * R));
      rest = up;
    }
  }
#pragma unroll
  for (int g = 0; g < MS; ++g) {
    if (g < span) nb += a.nb[l + g];
    bound[g] = nb;
  }
  const long long parent = rest;
  const int m = a.m[l], mc = m - nb, cols = m + 1;
  const int rows = a.has_gamma ? m + 1 : m;
  E* G = reinterpret_cast<E*>(smem);                 // rows x cols
  E* pv = G + (size_t)rows * cols;                   // nb pivots
  E* Lm = pv + nb;                                   // 2 x rows: multipliers, this step and next
  const E* Ap = elem<Ar>(a.A[l]) + parent * (long long)m * m;
  const E* cp = elem<Ar>(a.c[l]) + parent * (long long)m;
  const E* up = elem<Ar>(a.u[l]) + parent * (long long)m;
  const int tid = threadIdx.x, LT = blockDim.x;
  const E zero = Ar::zero();
  E* dB = Lm + 2 * rows + (ROOT ? a.nb[0] : 0);      // ROOT: behind d
  E w0 = zero;
  if constexpr (ROOT) {
    w0 = root_at<Ar>(a, 0, (int)parent);
    root_factors<Ar>(a, w0, Lm + 2 * rows, dB);
  }
  // ROOT: the last warp forms the root's path record meanwhile
  PathRec<E>* rootp = reinterpret_cast<PathRec<E>*>(dB + (ROOT ? a.nb[0] * (m + 1) : 0));
  const int FT = ROOT ? LT - 32 : LT;                // threads that fill
  if (ROOT && tid >= FT) {
    const PathRec<E> pr = root_path<Ar>(a, w0);
    if (tid == FT) *rootp = pr;
  }
  for (int idx = tid; idx < (tid < FT ? rows * cols : 0); idx += FT) {
    const int i = idx / cols, s = idx - (idx / cols) * cols;
    E g, v;
    if constexpr (ROOT) v = s < m || a.has_gamma ? root_entry<Ar>(a, dB, i, s) : zero;
    if (i == m) {                                   // the u row; its corner is the parent's exponent
      if constexpr (!ROOT) v = s < m ? up[s] : zero;
      g = s < nb ? Ar::neg(v) : v;
    } else {
      if constexpr (!ROOT) v = s < m ? Ap[(long long)i * m + s] : (a.has_gamma ? cp[i] : zero);
      if (i < nb) {
        E w = wg[0];                                 // the root of row i's group
#pragma unroll
        for (int q = 1; q < MS; ++q)
          if (q < span && i >= bound[q - 1]) w = wg[q];
        g = Ar::mul(w, v);
        if (s < nb) {
          g = Ar::neg(g);
          if (s == i) g = Ar::add(g, Ar::one());
        }
      } else {
        g = s < nb ? Ar::neg(v) : v;
      }
    }
    G[idx] = g;
  }
  // one step of look-ahead: warp 0 updates column kk + 1 and at once forms pivot kk + 1's
  // reciprocal and the next multipliers (into the other buffer) while warps 1.. update the
  // columns right of it; one barrier per step
  __syncthreads();                                   // the matrix is filled
  if (tid < 32) {                                    // pivot 0 and its multipliers
    const E piv = G[0];
    if (tid == 0) pv[0] = piv;
    const E r = Ar::recip(piv);
    for (int i = 1 + tid; i < rows; i += 32) Lm[i] = Ar::mul(G[i * cols], r);
  }
  __syncthreads();
  for (int kk = 0; kk < nb; ++kk) {
    const E* Lc = Lm + (kk & 1) * rows;              // this step's multipliers
    if (tid < 32) {
      E* Ln = Lm + ((kk + 1) & 1) * rows;
      const int s1 = kk + 1;
      for (int i = kk + 1 + tid; i < rows; i += 32)
        G[i * cols + s1] = Ar::fms(G[i * cols + s1], Lc[i], G[kk * cols + s1]);
      if (kk + 1 < nb) {
        __syncwarp();
        const E piv = G[s1 * cols + s1];
        if (tid == 0) pv[s1] = piv;
        const E r = Ar::recip(piv);
        for (int i = s1 + 1 + tid; i < rows; i += 32) Ln[i] = Ar::mul(G[i * cols + s1], r);
      }
    } else {
      // entries (i, s), i in (kk, rows), s in (kk + 1, cols), over threads 32..; two
      // independent entries per pass.  floor(idx / w_) from a float reciprocal: idx < 2^14
      // and w_ <= 96 (heralded states), so (idx + 1/2) / w_ stays 1/(2 w_) from an integer, the product's error below 2^-16
      const int t = tid - 32, LO = LT - 32;
      const int w_ = cols - kk - 2, total = (rows - kk - 1) * w_;
      const float rw = 1.0f / (float)(w_ > 0 ? w_ : 1);
      for (int idx = t; idx < total; idx += 2 * LO) {
        const int idx2 = idx + LO;
        const int i = kk + 1 + (int)(((float)idx + 0.5f) * rw);
        const int sc = kk + 2 + (idx - (i - kk - 1) * w_);
        const E g1 = Ar::fms(G[i * cols + sc], Lc[i], G[kk * cols + sc]);
        if (idx2 < total) {
          const int i2 = kk + 1 + (int)(((float)idx2 + 0.5f) * rw);
          const int s2 = kk + 2 + (idx2 - (i2 - kk - 1) * w_);
          G[i2 * cols + s2] = Ar::fms(G[i2 * cols + s2], Lc[i2], G[kk * cols + s2]);
        }
        G[i * cols + sc] = g1;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  return Sweep<E>{G, pv, nb, m, cols, rows, parent, rootp};
}

// The child's path record after a sweep, by one full warp (every lane returns it).
template <class Ar, bool ROOT>
__device__ __forceinline__ PathRec<typename Ar::E> sweep_path(const TreeArgs& a, int l, const Sweep<typename Ar::E>& w) {
  using E = typename Ar::E;
  const int lane = threadIdx.x & 31;
  PathRec<E> pr;
  if constexpr (ROOT) pr = *static_cast<const PathRec<E>*>(w.root_path);   // exponent zero: the root's is in the corner
  else pr = *path_at<Ar>(a.path[l], w.parent);
  int width = 1;                                     // butterfly over the pivots' lanes only
  while (width < w.nb && width < 32) width <<= 1;
  for (int t0 = 0; t0 < w.nb; t0 += 32) {
    const int t = t0 + lane;
    path_warp<Ar>(pr, t < w.nb ? w.pivots[t] : Ar::zero(), t < w.nb, width);
  }
  if (a.has_gamma) pr.ex = Ar::add(pr.ex, w.G[w.m * w.cols + w.m]);
  return pr;
}

}  // namespace
}  // namespace gbsbin
