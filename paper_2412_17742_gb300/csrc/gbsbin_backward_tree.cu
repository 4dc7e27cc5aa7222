// The reverse pass along the tree of block eliminations (arXiv:2412.17742, Sec. III Eq. q_d on
// the product grid of Sec. VI; the adjoint follows from d log det A = tr(A^{-1} dA)).
//
// With rows ordered by group, E the rows of groups 0 .. L-2 and F the last group's, the
// per-point matrix M = conj(D) - XA of a grid point splits as [[M_EE, M_EF], [M_FE, M_FF]],
// and only M_FF = conj(w) I - XA_FF depends on the last axis's root w.  For a parent (a
// combination of the first L-1 axes' roots) let A = inv(M_EE), U = A M_EF, V = M_FE A; each
// leaf's Schur complement is S(w) = conj(w) I - C with C = XA_FF - XA_FE U, and
//   inv(M) = [[A + U inv(S) V, -U inv(S)], [-inv(S) V, inv(S)]],
//   x = inv(M) X gamma:  x_F = s = inv(S) c_F,  x_E = a_E - U s   (c_F = b_F - V b_E, a_E = A b_E),
//   y = inv(M)^T gamma:  y_F = t = inv(S)^T d_F,  y_E = e_E - V^T t (d_F = g_F - U^T g_E, e_E = A^T g_E).
// Summed over the parent's leaves with the weights beta, the adjoint 1/2 sum beta (y x^T + inv(M)^T)
// needs only R = sum beta inv(S), Q = sum beta t s^T, sigma_s = sum beta s, sigma_t = sum beta t and
// the beta sum b: with Z = Q + R^T,
//   EE = b (e_E a_E^T + A^T) - e_E (U sigma_s)^T - (V^T sigma_t) a_E^T + V^T Z U^T,
//   EF = e_E sigma_s^T - V^T Z,   FE = sigma_t a_E^T - Z U^T,   FF = Z,
// and 1/2 sum beta (x + X y) from sum beta x = (b a_E - U sigma_s, sigma_s), sum beta y =
// (b e_E - V^T sigma_t, sigma_t).  So a leaf inverts an mF x mF matrix instead of n x n, and the
// parent's O(n^3) products are shared by its leaves.  Launches per wave of parents: the parents'
// inverses, their products, the leaves (each CTA a contiguous run of leaves, its sums per parent in
// its own slots), the leaves' sums, the parents' assembly into partials (in the original row
// order, transposed as the per-point kernel keeps them), reduced once at the end in FP64.
#include <cuda_runtime.h>

#include "gbsbin_backward_tree.h"
#include "gbsbin_device.cuh"
#include "gbsbin_df.cuh"
#include "gbsbin_gj.cuh"
#include "gbsbin_hess.cuh"

namespace gbsbin {
namespace {

constexpr int kBtThreads = 256;
// The products of few parents are split by columns over several CTAs each, two to an SM: panels of eight.
constexpr int kBwdSplitNb = 8;

// The block-row buffer (nb x n) after the kernels' other shared arrays.
__host__ __device__ __forceinline__ size_t backward_tree_rn_offset(int n, int nb) {
  return (size_t)16 * ((size_t)2 * n * nb + (size_t)nb * nb + 4 * (size_t)n + 1) + sizeof(double2) * GBSBIN_MAX_L;
}

struct Parent {                    // the parent's slot in pbuf
  template <class E>
  __device__ static void map(E* P, int mE, int mF, E** A, E** U, E** V, E** C, E** aE, E** eE, E** cF, E** dF) {
    *A = P;
    *U = *A + mE * mE;
    *V = *U + mE * mF;
    *C = *V + mF * mE;
    *aE = *C + mF * mF;
    *eE = *aE + mE;
    *cF = *eE + mE;
    *dF = *cF + mF;
  }
};

__device__ __forceinline__ int group_of(const BwdTree& t, int a) {
  int l = 0;
  while (l + 1 < t.L && a >= t.goff[l + 1]) ++l;
  return l;
}

// Per parent: A = inv(M_EE) and the vectors.
template <class Ar>
__global__ void __launch_bounds__(kBtThreads) k_bwdt_parent(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = b.n, nb = b.nb, mE = t.mE, mF = t.mF, D = t.D, tid = threadIdx.x, NT = kBtThreads;
  E* Pc = reinterpret_cast<E*>(smem);
  E* Rx = Pc + (size_t)n * nb;
  E* Dg = Rx + (size_t)nb * n;
  double2* wr = reinterpret_cast<double2*>(Dg + nb * nb);
  const E* A0 = reinterpret_cast<const E*>(t.A0);
  for (long long p = t.p0 + blockIdx.x; p < t.p1; p += gridDim.x) {
    E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
    Parent::map(reinterpret_cast<E*>(t.pbuf) + (size_t)(p - t.p0) * t.pstride, mE, mF, &A, &U, &V, &C, &aE, &eE,
                &cF, &dF);
    if (tid < t.L - 1) wr[tid] = grid_root(b.tw, b.grid, tid, point_digit(p * t.half, b.grid, tid));
    __syncthreads();
    for (int q = tid; q < mE * mE; q += NT) {        // M_EE = conj(D_E) - XA_EE
      const int i = q / mE, j = q - (q / mE) * mE;
      E v = Ar::neg(A0[(size_t)i * D + j]);
      if (i == j) {
        const double2 w = wr[group_of(t, i)];
        v = Ar::add(v, Ar::from(make_double2(w.x, -w.y)));
      }
      A[q] = v;
    }
    __syncthreads();
    gj_invert<Ar>(A, mE, mE, nb, Pc, Rx, Dg, t.rn ? reinterpret_cast<E*>(smem + backward_tree_rn_offset(n, nb)) : nullptr);
    // a_E = A b_E, e_E = A^T g_E (b = X gamma: column n; g = gamma: row n)
    for (int i = tid; i < mE; i += NT) {
      E sa = Ar::zero(), se = Ar::zero();
      for (int k = 0; k < mE; ++k) {
        sa = Ar::fma(A[(size_t)i * mE + k], A0[(size_t)k * D + n], sa);
        se = Ar::fma(A[(size_t)k * mE + i], A0[(size_t)n * D + k], se);
      }
      aE[i] = sa;
      eE[i] = se;
    }
    __syncthreads();
    // c_F = b_F - V b_E = b_F + XA_FE a_E, d_F = g_F - U^T g_E = g_F + XA_EF^T e_E
    for (int f = tid; f < mF; f += NT) {
      E sc = A0[(size_t)(mE + f) * D + n], sd = A0[(size_t)n * D + mE + f];
      for (int k = 0; k < mE; ++k) {
        sc = Ar::fma(A0[(size_t)(mE + f) * D + k], aE[k], sc);
        sd = Ar::fma(A0[(size_t)k * D + mE + f], eE[k], sd);
      }
      cF[f] = sc;
      dF[f] = sd;
    }
    __syncthreads();
  }
}

// The columns [lo, hi) of m that split y of `splits` takes.
__device__ __forceinline__ void split_range(int m, int y, int splits, int& lo, int& hi) {
  lo = (int)((long long)m * y / splits);
  hi = (int)((long long)m * (y + 1) / splits);
}

// Per parent and split: U = -A XA_EF, C = XA_FF - XA_FE U and V = -XA_FE A on its columns.
template <class Ar>
__global__ void __launch_bounds__(kBtThreads, 2) k_bwdt_products(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int nb = kBwdSplitNb, mE = t.mE, mF = t.mF, D = t.D, tid = threadIdx.x, NT = kBtThreads;
  E* Pc = reinterpret_cast<E*>(smem);
  E* Rx = Pc + (size_t)b.n * nb;
  const E* A0 = reinterpret_cast<const E*>(t.A0);
  int f0, f1, e0, e1;
  split_range(mF, blockIdx.y, gridDim.y, f0, f1);
  split_range(mE, blockIdx.y, gridDim.y, e0, e1);
  const int nf = f1 - f0;
  for (long long pr = blockIdx.x; pr < t.p1 - t.p0; pr += gridDim.x) {
    E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
    Parent::map(reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride, mE, mF, &A, &U, &V, &C, &aE, &eE, &cF, &dF);
    for (int q = tid; q < mF * nf; q += NT) {
      const int i = q / nf, j = f0 + q - (q / nf) * nf;
      C[(size_t)i * mF + j] = A0[(size_t)(mE + i) * D + mE + j];
    }
    __syncthreads();
    const E* AF = A0 + (size_t)mE * D;
#pragma unroll 1
    for (int g = 0; g < 3; ++g)                        // U, V, C (one call: the compiler inlines each)
      gemm_staged<Ar>(g == 0 ? U + f0 : (g == 1 ? V + e0 : C + f0), g == 1 ? mE : mF, g == 0 ? A : AF, g == 0 ? mE : D, 1,
                      g == 0 ? A0 + mE + f0 : (g == 1 ? A + e0 : U + f0), g == 0 ? D : (g == 1 ? mE : mF), 1,
                      g == 0 ? mE : mF, g == 1 ? e1 - e0 : nf, mE, g == 2, true, nb, Pc, Rx);
  }
}

// Leaves: CTA c takes leaves [c per, (c + 1) per) of the wave (parent-major); per leaf
// inv(S(w)), s, t and the sums into the slot of (c, parent).
template <class Ar>
__global__ void __launch_bounds__(kBwdLeafThreads, 2) k_bwdt_leaf(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  // shared memory sized by mF (backward_leaf_smem_bytes): two CTAs of four warps per SM, so
  // that one leaf's barriers overlap another's arithmetic
  const int mE = t.mE, mF = t.mF, nb = kBwdLeafNb, tid = threadIdx.x, NT = kBwdLeafThreads;
  E* Pc = reinterpret_cast<E*>(smem);
  E* Rx = Pc + (size_t)mF * nb;
  E* Rnb = Rx + (size_t)nb * mF;
  E* Dg = Rnb + (size_t)nb * mF;
  E* cFs = Dg + nb * nb;
  E* dFs = cFs + mF;
  E* sv = dFs + mF;
  E* tv = sv + mF;
  const int per_slot = t.leaf_ctas > b.nparts ? 2 : 1;   // leaf CTAs sharing one n x n slot
  E* W = reinterpret_cast<E*>(reinterpret_cast<char*>(b.ws) + (size_t)(blockIdx.x / per_slot) * (size_t)b.ws_slot_bytes) +
         (size_t)(blockIdx.x % per_slot) * mF * mF;
  const long long nleaves = (t.p1 - t.p0) * t.half;
  const long long l0 = (long long)blockIdx.x * t.per, l1 = min(l0 + t.per, nleaves);
  const long long pfirst = l0 / t.half;
  long long cur = -1;
  E* Cp = nullptr;
  for (long long l = l0; l < l1; ++l) {
    const long long pr = l / t.half, kl = l - pr * t.half;
    E* part = reinterpret_cast<E*>(t.part) + ((size_t)blockIdx.x * t.maxspan + (size_t)(pr - pfirst)) * t.lstride;
    E* R = part;
    E* Q = R + mF * mF;
    E* ss = Q + mF * mF;
    E* st = ss + mF;
    E* bb = st + mF;
    if (pr != cur) {                                   // a new parent: zero its sums, load c_F, d_F
      E *A, *U, *V, *aE, *eE, *cF, *dF;
      Parent::map(reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride, mE, mF, &A, &U, &V, &Cp, &aE, &eE, &cF,
                  &dF);
      for (long long q = tid; q < t.lstride; q += NT) part[q] = Ar::zero();
      for (int f = tid; f < mF; f += NT) {
        cFs[f] = cF[f];
        dFs[f] = dF[f];
      }
      cur = pr;
      __syncthreads();
    }
    const long long e = (t.p0 + pr) * t.half + kl;
    const double2 beta = b.beta[e];
    if (beta.x == 0.0 && beta.y == 0.0) continue;
    const double2 w = grid_root(b.tw, b.grid, t.L - 1, (int)kl);
    for (int q = tid; q < mF * mF; q += NT) {        // S = conj(w) I - C
      const int i = q / mF, j = q - (q / mF) * mF;
      E v = Ar::neg(Cp[q]);
      if (i == j) v = Ar::add(v, Ar::from(make_double2(w.x, -w.y)));
      W[q] = v;
    }
    __syncthreads();
    gj_invert<Ar>(W, mF, mF, nb, Pc, Rx, Dg, Rnb);
    {                                                  // s = inv(S) c_F (warp per row), t = inv(S)^T d_F
      const int lane = tid & 31, warp = tid >> 5;
      for (int i = warp; i < mF; i += NT / 32) {
        E acc = Ar::zero();
        for (int j = lane; j < mF; j += 32) acc = Ar::fma(W[(size_t)i * mF + j], cFs[j], acc);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc = Ar::add(acc, shfl_xor(acc, o));
        if (lane == 0) sv[i] = acc;
      }
      for (int j = tid; j < mF; j += NT) {
        E acc = Ar::zero();
        for (int i = 0; i < mF; ++i) acc = Ar::fma(W[(size_t)i * mF + j], dFs[i], acc);
        tv[j] = acc;
      }
    }
    __syncthreads();
    const E be = Ar::from(beta);
    for (int q = tid; q < mF * mF; q += NT) {
      const int i = q / mF, j = q - (q / mF) * mF;
      R[q] = Ar::fma(be, W[q], R[q]);
      Q[q] = Ar::fma(be, Ar::mul(tv[i], sv[j]), Q[q]);
    }
    for (int f = tid; f < mF; f += NT) {
      ss[f] = Ar::fma(be, sv[f], ss[f]);
      st[f] = Ar::fma(be, tv[f], st[f]);
    }
    if (tid == 0) bb[0] = Ar::add(bb[0], be);
    __syncthreads();
  }
}

// ---------------------------------------------------------------- leaves in the Hessenberg basis
// The leaves of a parent differ by conj(w) I only, so one unitary reduction C = Q H Q^H serves them all:
// inv(S) = Q inv(N) Q^H with N = conj(w) I - H, and with c' = Q^H c_F, d' = Q^T d_F
//   s = Q s',  t = conj(Q) t',  Q + R^T = conj(Q) (Q' + R'^T) Q^T,
// the primed sums those of the leaves with N, c', d'.  N = L U by the forward's unpivoted Hessenberg elimination (L
// unit lower bidiagonal with multipliers l), so the inverse takes the m^3 / 6 multiply-adds of the triangular one
// and O(m^2) more, instead of m^3: inv(N) L = inv(U) gives row i of inv(N) from the right,
// x_ij = inv(U)_ij - l_j x_i,j+1.  At n = 200 (81 parents, 3321 leaves of 100 rows, pairs of FP32) the Gauss-Jordan
// leaves took 10.1 ms; the reduction takes 0.87, the leaves 2.91 and the way back 1.08.
constexpr int kBwdHessMax = GBSBIN_BT_MAX_HESS;
constexpr int kBwdHessThreads = 512;
constexpr int kRotThreads = 256;
constexpr int kRotSlots = (kBwdHessMax + 7) / 8;

template <class E>
struct Rotated {                                       // the rest of a parent's slot: its leaves' sums
  E *Z, *ss, *st, *v0, *beta;
  static __device__ Rotated map(E* P, int n, int mF) {
    Rotated r;
    r.Z = P + (size_t)n * n + 2 * n;
    r.ss = r.Z + mF * mF;
    r.st = r.ss + mF;
    r.v0 = r.st + mF;
    r.beta = r.v0 + mF;
    return r;
  }
};

// Sum over the g = 2^k lanes of a group.
template <class Ar>
__device__ __forceinline__ typename Ar::E group_sum(typename Ar::E v, int g) {
  for (int o = g >> 1; o > 0; o >>= 1) v = Ar::add(v, shfl_xor(v, o));
  return v;
}

// C -> H in place, a CTA per parent, [C, c_F, conj(d_F)] in shared memory (row stride odd).  The lanes of a column
// form its product with the reflector and update it, then the lanes of a row: three barriers per step.  Below the
// subdiagonal the reflectors' entries stay; their first entries and factors go to v0 and beta.
template <class Ar>
__global__ void __launch_bounds__(kBwdHessThreads) k_bwdt_hess(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int m = t.mF, ld = (m + 2) | 1, tid = threadIdx.x, T = kBwdHessThreads, lane = tid & 31;
  E* M = reinterpret_cast<E*>(smem);
  E* v = M + (size_t)m * ld;
  E* sc = v + m;
  E* const P = reinterpret_cast<E*>(t.pbuf) + (size_t)blockIdx.x * t.pstride;
  E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
  Parent::map(P, t.mE, m, &A, &U, &V, &C, &aE, &eE, &cF, &dF);
  const Rotated<E> rot = Rotated<E>::map(P, b.n, m);
  for (int q = tid; q < m * m; q += T) M[(size_t)(q / m) * ld + q % m] = C[q];
  for (int i = tid; i < m; i += T) {
    M[(size_t)i * ld + m] = cF[i];
    M[(size_t)i * ld + m + 1] = Ar::conj(dF[i]);
  }
  __syncthreads();
  const int extra = t.has_gamma ? 2 : 0;
  for (int k = 0; k + 2 < m; ++k) {
    if (tid < 32) {
      E rest = Ar::zero();
      for (int i = k + 2 + lane; i < m; i += 32) rest = Ar::add(rest, Ar::norm2(M[(size_t)i * ld + k]));
      rest = group_sum<Ar>(rest, 32);
      const E x0 = M[(size_t)(k + 1) * ld + k];
      E alpha = x0, v0 = Ar::zero(), beta = Ar::zero();
      if (Ar::re(rest) > 0.f) reflector<Ar>(rest, x0, alpha, v0, beta);
      for (int i = k + 1 + lane; i < m; i += 32) v[i] = i == k + 1 ? v0 : M[(size_t)i * ld + k];
      if (lane == 0) {
        sc[0] = beta;
        rot.v0[k] = v[k + 1];
        rot.beta[k] = beta;
      }
      __syncwarp();
      if (lane == 0) M[(size_t)(k + 1) * ld + k] = alpha;
    }
    __syncthreads();
    const E beta = sc[0];
    if (Ar::re(beta) > 0.f) {
      {                                                // columns k + 1 .. m + 1 from the left
        const int nc = m - 1 - k + extra, g = nc * 8 <= T ? 8 : 4, q = tid & (g - 1);
        const int groups = T / g, rounds = (nc + groups - 1) / groups;
        for (int r = 0; r < rounds; ++r) {
          const int c = r * groups + tid / g, j = k + 1 + c;
          E sum = Ar::zero();
          if (c < nc)
            for (int i = k + 1 + q; i < m; i += g) sum = Ar::fma(Ar::conj(v[i]), M[(size_t)i * ld + j], sum);
          sum = Ar::mul(beta, group_sum<Ar>(sum, g));
          if (c < nc)
            for (int i = k + 1 + q; i < m; i += g) M[(size_t)i * ld + j] = Ar::fms(M[(size_t)i * ld + j], v[i], sum);
        }
      }
      __syncthreads();
      {                                                // rows from the right
        const int g = m * 8 <= T ? 8 : 4, q = tid & (g - 1), i = tid / g;
        E sum = Ar::zero();
        if (i < m)
          for (int j = k + 1 + q; j < m; j += g) sum = Ar::fma(M[(size_t)i * ld + j], v[j], sum);
        sum = Ar::mul(beta, group_sum<Ar>(sum, g));
        if (i < m)
          for (int j = k + 1 + q; j < m; j += g) M[(size_t)i * ld + j] = Ar::fms(M[(size_t)i * ld + j], sum, Ar::conj(v[j]));
      }
    }
    __syncthreads();
  }
  for (int q = tid; q < m * m; q += T) C[q] = M[(size_t)(q / m) * ld + q % m];
  for (int i = tid; i < m; i += T) {
    cF[i] = M[(size_t)i * ld + m];
    dF[i] = Ar::conj(M[(size_t)i * ld + m + 1]);
  }
}

// Leaves: CTA c takes leaves [c per, (c + 1) per) of the wave.  Four phases: one warp eliminates the Hessenberg
// matrix (its row in registers, four columns a lane) and leaves U in shared memory (packed by rows, the diagonal
// inverted); U is inverted in place, the 8 x 8 diagonal blocks first, then block columns left to right,
// X_J = -X (U_J X_JJ) in 1 x 4 tiles; a thread per row then runs the recurrence of inv(N) and adds to the sums.
template <class Ar, bool DISP>
__global__ void __launch_bounds__(kBwdLeafThreads, 2) k_bwdt_hleaf(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int m = t.mF, tid = threadIdx.x, NT = kBwdLeafThreads, lane = tid & 31, warp = tid >> 5;
  E* Up = reinterpret_cast<E*>(smem);                  // U, then its inverse: row i at row(i) + j, j >= i
  E* Tb = Up + (size_t)m * (m + 1) / 2;                // m x 8
  E* lv = Tb + (size_t)8 * m;
  E* yv = lv + m;
  E* zv = yv + m;
  auto row = [&](int i) { return i * m - i * (i + 1) / 2; };
  const long long nleaves = (t.p1 - t.p0) * t.half;
  const long long l0 = (long long)blockIdx.x * t.per, l1 = min(l0 + t.per, nleaves);
  const long long pfirst = l0 / t.half;
  long long cur = -1;
  const E *H = nullptr, *cs = nullptr, *ds = nullptr;
  for (long long l = l0; l < l1; ++l) {
    const long long pr = l / t.half, kl = l - pr * t.half;
    E* Z = reinterpret_cast<E*>(t.part) + ((size_t)blockIdx.x * t.maxspan + (size_t)(pr - pfirst)) * t.lstride;
    E* ss = Z + m * m;
    E* st = ss + m;
    E* bb = st + m;
    if (pr != cur) {
      E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
      Parent::map(reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride, t.mE, m, &A, &U, &V, &C, &aE, &eE, &cF, &dF);
      H = C;
      cs = cF;
      ds = dF;
      for (long long q = tid; q < t.lstride; q += NT) Z[q] = Ar::zero();
      cur = pr;
      __syncthreads();
    }
    const long long e = (t.p0 + pr) * t.half + kl;
    const double2 beta = b.beta[e];
    if (beta.x == 0.0 && beta.y == 0.0) continue;
    const double2 w = grid_root(b.tw, b.grid, t.L - 1, (int)kl);
    const E wc = Ar::from(make_double2(w.x, -w.y)), be = Ar::from(beta);
    if (warp == 0) {
      E r[4], hn[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const int j = lane + 32 * s;
        r[s] = j < m ? Ar::neg(H[j]) : Ar::zero();
        hn[s] = j < m ? H[m + j] : Ar::zero();
      }
      if (lane == 0) r[0] = Ar::add(r[0], wc);
      E y = DISP ? cs[0] : Ar::zero();
#pragma unroll
      for (int sb = 0; sb < 4; ++sb) {
        const int iend = min(m, 32 * sb + 32);
        for (int i = 32 * sb; i < iend; ++i) {
          const int il = i & 31;
          const E rp = Ar::recip(shfl(r[sb], il));
#pragma unroll
          for (int s = 0; s < 4; ++s) {
            const int j = lane + 32 * s;
            if (s >= sb && j >= i && j < m) Up[row(i) + j] = j == i ? rp : r[s];
          }
          if (DISP && lane == 0) yv[i] = y;
          if (i + 1 < m) {
            const E lm = Ar::neg(Ar::mul(shfl(hn[sb], il), rp));
            if (lane == 0) lv[i] = lm;
            if (DISP) y = Ar::fms(cs[i + 1], lm, y);
            const E* hrow = H + (size_t)min(i + 2, m - 1) * m;
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              const int j = lane + 32 * s;
              if (s < sb) continue;
              E x = Ar::neg(hn[s]);
              if (j == i + 1) x = Ar::add(x, wc);
              hn[s] = j < m ? hrow[j] : Ar::zero();
              r[s] = Ar::fms(x, lm, r[s]);
            }
          } else if (lane == 0) {
            lv[i] = Ar::zero();
          }
        }
      }
    }
    __syncthreads();
    {                                                  // the diagonal blocks, a thread per column
      const int j = tid, K = j & ~7, jj = j & 7;
      E x[8];
#pragma unroll
      for (int ii = 7; ii >= 0; --ii) {
        x[ii] = Ar::zero();
        if (j < m && ii <= jj) {
          const E rp = Up[row(K + ii) + K + ii];
          if (ii == jj) {
            x[ii] = rp;
          } else {
            E acc = Ar::zero();
#pragma unroll
            for (int kk = ii + 1; kk < 8; ++kk)
              if (kk <= jj) acc = Ar::fms(acc, Up[row(K + ii) + K + kk], x[kk]);
            x[ii] = Ar::mul(acc, rp);
          }
        }
      }
      __syncthreads();
#pragma unroll
      for (int ii = 0; ii < 7; ++ii)
        if (j < m && ii < jj) Up[row(K + ii) + j] = x[ii];
    }
    __syncthreads();
    for (int K = 8; K < m; K += 8) {
      const int bs = min(8, m - K);
      for (int q = tid; q < 8 * K; q += NT) {          // T = U_J X_JJ
        const int k = q >> 3, c = q & 7;
        E acc = Ar::zero();
        if (c < bs)
          for (int cc = 0; cc <= c; ++cc) acc = Ar::fma(Up[row(k) + K + cc], Up[row(K + cc) + K + c], acc);
        Tb[q] = acc;
      }
      __syncthreads();
      const int nw = (2 * K + 31) / 32;                // warps' items of 16 rows, the longest with the shortest
      for (int rd = 0; rd * 4 < nw; ++rd) {
        const int wi = rd * 4 + ((rd & 1) ? 3 - warp : warp);
        if (wi >= nw) continue;
        const int i = wi * 16 + (lane >> 1), h = 4 * (lane & 1);
        E acc[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[c] = Ar::zero();
        const int base = i < K ? row(i) : 0;
        for (int k = wi * 16; k < K; ++k) {
          const E u = (i < K && k >= i) ? Up[base + k] : Ar::zero();
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[c] = Ar::fms(acc[c], u, Tb[8 * k + h + c]);
        }
        if (i < K)
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (h + c < bs) Up[base + K + h + c] = acc[c];
      }
      __syncthreads();
    }
    E bs_i = Ar::zero();                               // beta s_i
    if (DISP) {                                        // s = inv(U) y, z = inv(U)^T d: m + 1 terms a thread
      if (tid < m) {
        E sa = Ar::zero(), za = Ar::zero();
        for (int j = tid; j < m; ++j) sa = Ar::fma(Up[row(tid) + j], yv[j], sa);
        for (int i = 0; i <= tid; ++i) za = Ar::fma(Up[row(i) + tid], ds[i], za);
        zv[tid] = za;
        bs_i = Ar::mul(be, sa);
        ss[tid] = Ar::add(ss[tid], bs_i);
      }
      __syncthreads();
    }
    if (tid < m) {                                     // row tid of inv(N); Z[j][i] += beta (t_j s_i + x_ij)
      E x = Ar::zero(), tj = Ar::zero();
      const int base = row(tid);
      for (int jb = m - 1; jb >= 0; jb -= 4) {
        E zo[4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (jb - c >= 0) zo[c] = Z[(size_t)(jb - c) * m + tid];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int j = jb - c;
          if (j < 0) continue;
          const E lj = lv[j];
          x = Ar::fms(j >= tid ? Up[base + j] : Ar::zero(), lj, x);
          E z = Ar::fma(be, x, zo[c]);
          if (DISP) {
            tj = Ar::fms(zv[j], lj, tj);
            z = Ar::fma(tj, bs_i, z);
            if (j == tid) st[j] = Ar::fma(be, tj, st[j]);
          }
          Z[(size_t)j * m + tid] = z;
        }
      }
    }
    if (tid == 0) bb[0] = Ar::add(bb[0], be);
    __syncthreads();
  }
}

// Back from the Hessenberg basis: RIGHT 0: Z <- conj(Q) Z', sigma_t <- conj(Q) sigma_t' from the leaf CTAs' sums;
// RIGHT 1: Z <- Z Q^T, sigma_s <- Q sigma_s'.  The columns (then the rows) are independent: eight lanes each hold
// one in registers and apply the reflectors last to first, all of them in shared memory, without a barrier.
template <class Ar, bool RIGHT>
__global__ void __launch_bounds__(kRotThreads, 2) k_bwdt_unrot(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int m = t.mF, tid = threadIdx.x, NT = kRotThreads, g = tid & 7;
  const long long pr = blockIdx.x;
  E* Vs = reinterpret_cast<E*>(smem);                  // reflector k at off(k) + i, i = k + 1 .. m - 1
  E* bet = Vs + (size_t)m * (m - 1) / 2;
  auto off = [&](int k) { return k * (m - 1) - k * (k - 1) / 2 - (k + 1); };
  E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
  E* const P = reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride;
  Parent::map(P, t.mE, m, &A, &U, &V, &C, &aE, &eE, &cF, &dF);
  const Rotated<E> rot = Rotated<E>::map(P, b.n, m);
  for (int q = tid; q < m * m; q += NT) {
    const int i = q / m, k = q - (q / m) * m;
    if (k + 2 < m && i > k) Vs[off(k) + i] = i == k + 1 ? rot.v0[k] : C[q];
  }
  for (int k = tid; k + 2 < m; k += NT) bet[k] = rot.beta[k];
  __syncthreads();
  const int j = blockIdx.y * (NT / 8) + tid / 8;       // the column (or row); m: the vector
  const long long c0 = (pr * t.half) / t.per, c1 = (pr * t.half + t.half - 1) / t.per;
  E z[kRotSlots];
#pragma unroll
  for (int q = 0; q < kRotSlots; ++q) {
    const int i = g + 8 * q;
    z[q] = Ar::zero();
    if (i >= m || j > m) continue;
    if (RIGHT && j < m) {
      z[q] = rot.Z[(size_t)j * m + i];
      continue;
    }
    for (long long c = c0; c <= c1; ++c) {
      const E* part = reinterpret_cast<const E*>(t.part) +
                      ((size_t)c * t.maxspan + (size_t)(pr - (c * t.per) / t.half)) * t.lstride;
      z[q] = Ar::add(z[q], j < m ? part[(size_t)i * m + j] : part[m * m + (RIGHT ? 0 : m) + i]);
    }
  }
  for (int k = m - 3; k >= 0; --k) {
    const E* v = Vs + off(k);
    const int q0 = (k + 1) >> 3;
    E s0 = Ar::zero();
#pragma unroll
    for (int q = 0; q < kRotSlots; ++q) {
      const int i = g + 8 * q;
      if (q >= q0 && i > k && i < m) s0 = Ar::fma(RIGHT ? Ar::conj(v[i]) : v[i], z[q], s0);
    }
    s0 = Ar::mul(bet[k], group_sum<Ar>(s0, 8));
#pragma unroll
    for (int q = 0; q < kRotSlots; ++q) {
      const int i = g + 8 * q;
      if (q >= q0 && i > k && i < m) z[q] = Ar::fms(z[q], RIGHT ? v[i] : Ar::conj(v[i]), s0);
    }
  }
#pragma unroll
  for (int q = 0; q < kRotSlots; ++q) {
    const int i = g + 8 * q;
    if (i >= m || j > m) continue;
    if (j < m) rot.Z[RIGHT ? (size_t)j * m + i : (size_t)i * m + j] = z[q];
    else (RIGHT ? rot.ss : rot.st)[i] = z[q];
  }
}

template <class Ar>
cudaError_t launch_hess_leaves(const BackwardArgs& b, const BwdTree& t, long long parents, long long leaf_ctas,
                               cudaStream_t s) {
  const int m = t.mF;
  const size_t hsm = (size_t)16 * ((size_t)m * ((m + 2) | 1) + m + 1);
  const size_t lsm = (size_t)16 * ((size_t)m * (m + 1) / 2 + 11 * (size_t)m);
  const size_t rsm = (size_t)16 * ((size_t)m * (m - 1) / 2 + m);
  auto leaf = t.has_gamma ? k_bwdt_hleaf<Ar, true> : k_bwdt_hleaf<Ar, false>;
  cudaError_t err;
  if ((err = cudaFuncSetAttribute(k_bwdt_hess<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)hsm)) !=
          cudaSuccess ||
      (err = cudaFuncSetAttribute(leaf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lsm)) != cudaSuccess ||
      (err = cudaFuncSetAttribute(k_bwdt_unrot<Ar, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm)) !=
          cudaSuccess ||
      (err = cudaFuncSetAttribute(k_bwdt_unrot<Ar, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rsm)) !=
          cudaSuccess)
    return err;
  k_bwdt_hess<Ar><<<(unsigned)parents, kBwdHessThreads, hsm, s>>>(b, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  leaf<<<(unsigned)leaf_ctas, kBwdLeafThreads, lsm, s>>>(b, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  const dim3 rg((unsigned)parents, (unsigned)((m + 1 + kRotThreads / 8 - 1) / (kRotThreads / 8)));
  k_bwdt_unrot<Ar, false><<<rg, kRotThreads, rsm, s>>>(b, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  k_bwdt_unrot<Ar, true><<<rg, kRotThreads, rsm, s>>>(b, t);
  return cudaGetLastError();
}

// The sums of Gauss-Jordan leaves over their CTAs: Z = Q + R^T, sigma_s, sigma_t per parent.
template <class Ar>
__global__ void __launch_bounds__(kBtThreads) k_bwdt_sum(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  const int mF = t.mF, q = blockIdx.y * kBtThreads + threadIdx.x;
  const long long pr = blockIdx.x;
  const Rotated<E> rot = Rotated<E>::map(reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride, b.n, mF);
  const long long c0 = (pr * t.half) / t.per, c1 = (pr * t.half + t.half - 1) / t.per;
  if (q >= mF * mF + 2 * mF) return;
  E z = Ar::zero();
  for (long long c = c0; c <= c1; ++c) {
    const E* part = reinterpret_cast<const E*>(t.part) +
                    ((size_t)c * t.maxspan + (size_t)(pr - (c * t.per) / t.half)) * t.lstride;
    z = Ar::add(z, part[mF * mF + q]);
    if (q < mF * mF) z = Ar::add(z, part[(size_t)(q % mF) * mF + q / mF]);
  }
  rot.Z[q] = z;                                        // (sigma_s and sigma_t follow Z in both)
}

// Per parent and split: the three products on its columns of E and of F, and 1/2 (Phi + Psi^T) of them into the
// parent's partial in the original row order (ST[j][i] = S[i][j]); the splits of a partial write different rows
// of ST.  Bound by the issue of the products' multiply-adds (one warp's latency where the blocks are small).  81
// parents of 100 + 100 rows in pairs on 152 SMs: one CTA each 1.72 ms, three 1.05; with the parents' products, 1.60
// -> 0.56 + 0.84 ms.  13 parents of 24 + 24 rows in FP64: parents, leaves and assembly 617 us -> 250 (entry by entry
// instead of 36 tiles of 4 x 4, three splits).
template <class Ar>
__global__ void __launch_bounds__(kBtThreads, 2) k_bwdt_assemble(BackwardArgs b, BwdTree t) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = b.n, nb = kBwdSplitNb, mE = t.mE, mF = t.mF, tid = threadIdx.x, NT = kBtThreads;
  const int lane = tid & 31, warp = tid >> 5;
  E* Pc = reinterpret_cast<E*>(smem);
  E* Rx = Pc + (size_t)n * nb;
  E* uS = Rx + (size_t)nb * n;
  E* vT = uS + mE;
  E* bbs = vT + mE;
  E* ST = reinterpret_cast<E*>(b.partS) + (size_t)blockIdx.x * n * n;
  E* sg = reinterpret_cast<E*>(b.partg) + (size_t)blockIdx.x * n;
  E* W = reinterpret_cast<E*>(reinterpret_cast<char*>(b.ws) + (size_t)blockIdx.x * (size_t)b.ws_slot_bytes);
  E* X1 = W;                                           // Z U^T (mF x mE)
  E* X2 = X1 + mF * mE;                                // V^T Z U^T (mE x mE)
  E* X3 = X2 + mE * mE;                                // V^T Z (mE x mF)
  int f0, f1, e0, e1;
  split_range(mF, blockIdx.y, gridDim.y, f0, f1);
  split_range(mE, blockIdx.y, gridDim.y, e0, e1);
  auto mine = [&](int c) { return c < mE ? c >= e0 && c < e1 : c - mE >= f0 && c - mE < f1; };
  if (t.zero_partials) {
    for (int jo = warp; jo < n; jo += NT / 32)
      if (mine(t.pinv[jo]))
        for (int io = lane; io < n; io += 32) ST[(size_t)jo * n + io] = Ar::zero();
    if (blockIdx.y == 0)
      for (int q = tid; q < n; q += NT) sg[q] = Ar::zero();
    __syncthreads();
  }
  for (long long p = t.p0 + blockIdx.x; p < t.p1; p += gridDim.x) {
    const long long pr = p - t.p0;
    E *A, *U, *V, *C, *aE, *eE, *cF, *dF;
    E* const P = reinterpret_cast<E*>(t.pbuf) + (size_t)pr * t.pstride;
    Parent::map(P, mE, mF, &A, &U, &V, &C, &aE, &eE, &cF, &dF);
    const Rotated<E> rot = Rotated<E>::map(P, n, mF);
    const E *Z = rot.Z, *ss = rot.ss, *st = rot.st;
    if (tid == 0) {
      const long long c0 = (pr * t.half) / t.per, c1 = (pr * t.half + t.half - 1) / t.per;
      E v = Ar::zero();
      for (long long c = c0; c <= c1; ++c)
        v = Ar::add(v, reinterpret_cast<const E*>(t.part)[((size_t)c * t.maxspan +
                                                           (size_t)(pr - (c * t.per) / t.half) + 1) * t.lstride - 1]);
      bbs[0] = v;
    }
#pragma unroll 1
    for (int g = 0; g < 3; ++g)                        // X1, X2, X3
      gemm_staged<Ar>(g == 0 ? X1 + e0 : (g == 1 ? X2 + e0 : X3 + f0), g == 2 ? mF : mE, g == 0 ? Z : V,
                      g == 0 ? mF : 1, g == 0 ? 1 : mE,
                      g == 0 ? U + (size_t)e0 * mF : (g == 1 ? X1 + e0 : Z + f0), g == 0 ? 1 : (g == 1 ? mE : mF),
                      g == 0 ? mF : 1, g == 0 ? mF : mE, g == 2 ? f1 - f0 : e1 - e0, mF, false, false, nb, Pc, Rx);
    for (int i = tid; i < mE; i += NT) {             // U sigma_s, V^T sigma_t
      E su = Ar::zero(), sv = Ar::zero();
      for (int k = 0; k < mF; ++k) {
        su = Ar::fma(U[(size_t)i * mF + k], ss[k], su);
        sv = Ar::fma(V[(size_t)k * mE + i], st[k], sv);
      }
      uS[i] = su;
      vT[i] = sv;
    }
    __syncthreads();
    const E bsum = bbs[0];
    const E half = Ar::from(make_double2(0.5, 0.0));
    for (int jo = warp; jo < n; jo += NT / 32) {
      const int c = t.pinv[jo];
      if (!mine(c)) continue;
      for (int io = lane; io < n; io += 32) {        // ST[jo][io] = S[io][jo]
        const int a = t.pinv[io];
        E v;
        if (a < mE && c < mE)
          v = Ar::add(Ar::fma(bsum, Ar::add(Ar::mul(eE[a], aE[c]), A[(size_t)c * mE + a]),
                              Ar::neg(Ar::add(Ar::mul(eE[a], uS[c]), Ar::mul(vT[a], aE[c])))),
                      X2[(size_t)a * mE + c]);
        else if (a < mE)
          v = Ar::fms(Ar::mul(eE[a], ss[c - mE]), Ar::one(), X3[(size_t)a * mF + (c - mE)]);
        else if (c < mE)
          v = Ar::fms(Ar::mul(st[a - mE], aE[c]), Ar::one(), X1[(size_t)(a - mE) * mE + c]);
        else
          v = Z[(size_t)(a - mE) * mF + (c - mE)];
        const size_t q = (size_t)jo * n + io;
        ST[q] = Ar::fma(half, v, ST[q]);
      }
    }
    for (int io = tid; blockIdx.y == 0 && io < n; io += NT) {   // 1/2 (sum beta x + X sum beta y)
      const int h = n / 2, po = io < h ? io + h : io - h;
      const int a = t.pinv[io], ap = t.pinv[po];
      const E xs = a < mE ? Ar::fms(Ar::mul(bsum, aE[a]), Ar::one(), uS[a]) : ss[a - mE];
      const E ys = ap < mE ? Ar::fms(Ar::mul(bsum, eE[ap]), Ar::one(), vT[ap]) : st[ap - mE];
      sg[io] = Ar::fma(half, Ar::add(xs, ys), sg[io]);
    }
    __syncthreads();
  }
}

template <class Ar>
cudaError_t tree_wave(const BackwardArgs& b, const BwdTree& t0, cudaStream_t s) {
  BwdTree t = t0;
  const size_t base = backward_tree_smem_bytes(b.n, b.nb), with = base + (size_t)16 * b.nb * b.n;
  t.rn = with <= 226 * 1024 ? 1 : 0;
  const size_t smem = t.rn ? with : base, ssmem = backward_tree_smem_bytes(b.n, kBwdSplitNb);
  cudaError_t err;
  if ((err = cudaFuncSetAttribute(k_bwdt_parent<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) !=
          cudaSuccess ||
      (err = cudaFuncSetAttribute(k_bwdt_products<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem)) !=
          cudaSuccess ||
      (err = cudaFuncSetAttribute(k_bwdt_assemble<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssmem)) !=
          cudaSuccess)
    return err;
  const long long parents = t.p1 - t.p0;
  const long long gp = parents < b.nparts ? parents : b.nparts;
  // splits: two CTAs an SM in one wave, at least eight columns each (one CTA a parent: 81 parents 0.7 ms more, 13
  // parents of 24 + 24 rows 0.3 ms more of 2.0)
  const int cols = (t.mE < t.mF ? t.mE : t.mF) / 8, fill = (int)(2 * b.nparts / t.nparts);
  const int splits = cols < 1 || fill < 1 ? 1 : (cols < fill ? cols : fill);
  k_bwdt_parent<Ar><<<(unsigned)gp, kBtThreads, smem, s>>>(b, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  k_bwdt_products<Ar><<<dim3((unsigned)gp, (unsigned)splits), kBtThreads, ssmem, s>>>(b, t);
  if ((err = cudaGetLastError()) != cudaSuccess) return err;
  const long long nleaves = parents * t.half;
  const long long gl = (nleaves + t.per - 1) / t.per;
  if (t.hess) {
    if ((err = launch_hess_leaves<Ar>(b, t, parents, gl, s)) != cudaSuccess) return err;
  } else {
    const size_t lsmem = backward_leaf_smem_bytes(t.mF);
    if ((err = cudaFuncSetAttribute(k_bwdt_leaf<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)lsmem)) !=
        cudaSuccess)
      return err;
    k_bwdt_leaf<Ar><<<(unsigned)gl, kBwdLeafThreads, lsmem, s>>>(b, t);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
    const int words = t.mF * t.mF + 2 * t.mF;
    k_bwdt_sum<Ar><<<dim3((unsigned)parents, (unsigned)((words + kBtThreads - 1) / kBtThreads)), kBtThreads, 0, s>>>(b, t);
    if ((err = cudaGetLastError()) != cudaSuccess) return err;
  }
  k_bwdt_assemble<Ar><<<dim3((unsigned)t.nparts, (unsigned)splits), kBtThreads, ssmem, s>>>(b, t);
  return cudaGetLastError();
}

}  // namespace

size_t backward_leaf_smem_bytes(int mF) {
  return (size_t)16 * ((size_t)3 * mF * kBwdLeafNb + (size_t)kBwdLeafNb * kBwdLeafNb + 4 * (size_t)mF);
}

// The reduction and the way back are launches of one or a few CTAs per parent, O(mF^3) each, as long for one parent
// as for an SM each, and the way back grows with the parents; the saving grows with the leaves per SM and faster with
// mF, the less in FP64 whose leaves are bound by their products. Reverse-pass kernels, Hessenberg over Gauss-Jordan
// leaves, at 8 / 16 / 24 leaves per SM (61 parents; 140 parents):
//   rows  pairs                                  FP64
//   32    1.14 / 0.97 / 0.88; 1.15 / 1.02 / 0.92   1.48 / 1.22 / 1.10; 1.85 / 1.57 / 1.36
//   40    1.04 / 0.87 / 0.78; 1.08 / 0.93 / 0.82   1.20 / 0.95 / 0.83; 1.52 / 1.23 / 1.04
//   48    0.91 / 0.74 / 0.67; 0.95 / 0.81 / 0.71   1.18 / 0.92 / 0.81; 1.48 / 1.20 / 1.00
//   60    0.88 / 0.72 / 0.65; 0.94 / 0.80 / 0.71   0.94 / 0.73 / 0.64; 1.18 / 0.94 / 0.78
//   80    0.74 / 0.56 / 0.49; 0.82 / 0.65 / 0.55   0.90 / 0.65 / 0.55; 1.06 / 0.81 / 0.66
//   100   0.55 / 0.40 / 0.34; 0.65 / 0.45 / 0.37   0.71 / 0.49 / 0.41; 0.94 / 0.64 / 0.51
// The line: leaves per SM by the rows and the arithmetic, times 1 + parents / SMs, and eight in any case.
bool backward_hess_suits(int mF, long long parents, long long half, int num_sms, bool df) {
  if (mF < (df ? 32 : 40) || mF > kBwdHessMax) return false;
  const double least = df ? (mF < 40 ? 14.5 : mF < 48 ? 9.2 : 4.0) : (mF < 60 ? 14.0 : mF < 80 ? 7.5 : mF < 100 ? 5.3 : 4.0);
  const long long rounds = (parents + num_sms - 1) / num_sms;
  const double leaves = (double)(parents * half) / num_sms;
  return leaves >= 8.0 * rounds && leaves >= least * (1.0 + (double)parents / num_sms);
}

size_t backward_tree_smem_bytes(int n, int nb) {
  return (size_t)16 * ((size_t)2 * n * nb + (size_t)nb * nb + 4 * (size_t)n + 1) + sizeof(double2) * GBSBIN_MAX_L;
}

cudaError_t launch_backward_tree_wave(const BackwardArgs& b, const BwdTree& t, cudaStream_t s) {
  return b.df ? tree_wave<ArDF>(b, t, s) : tree_wave<ArF64>(b, t, s);
}

}  // namespace gbsbin
