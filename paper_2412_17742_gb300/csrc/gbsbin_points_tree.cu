// Grid points by a tree of block eliminations (arXiv:2412.17742, Sec. III Eq. q_d on the
// roots-of-unity grid of Sec. VI), in pairs of FP32 or in FP64.
//
// Order the rows and columns of K(w) = I - D(w) A (A = XA) by detector group, group 0
// first (a symmetric permutation: det and the bilinear form below are unchanged, and
// every unpivoted pivot keeps Re > 0, so the branch of log det is the one of the
// per-point LU).  The leading block of group 0 is B = I - w_0 A_00, and eliminating it
// leaves the Schur complement
//
//   K_rr - K_r0 B^-1 K_0r = I - D_r (A_rr + A_r0 W),   W = w_0 B^-1 A_0r,
//
// again of the form I - D' A' with A' depending on w_0 only.  So every point with the same
// phases w_0..w_l shares the first l + 1 eliminations: depth l of the tree holds one
// reduced matrix per combination of the first l axes' roots, and a grid point is a leaf
// (the last group's block, last axis halved by conjugate symmetry).  The displacement term
// u^T K^-1 v, u = gamma, v = D X gamma, splits the same way: each elimination adds
// u_0^T y with y = w_0 B^-1 c_0 (v = D c), and leaves c' = c_r + A_r0 y, u' = u_r + W^T u_0.
//
// A level CTA runs one Gauss-Jordan sweep over the first nb columns of
//
//   [ B      | w A_0r | w c_0 ]        ->   [ I | W  | y  ]
//   [ -A_r0  | A_rr   | c_r   ]             [ . | A' | c' ],
//
// whose pivots are those of B's unpivoted LU.  log q = 1/2 sum(u_0^T y) - 1/2 sum Log(pivots).
// Each node carries a path record - the pivot product (scaled by a power of two), the FP32
// sum of the pivots' arguments, the exponent sum and the smallest pivot real part - and
// leaves write the unfinished form from which the inverse DFT takes G (undisplaced plans' leaves write G themselves)
// and log q is finished in FP64 when asked for.
//
// Arithmetic: every kernel is written once over an arithmetic (gbsbin_df.cuh): pairs of
// FP32 (about 46 bits) on the FMA pipe, or FP64.  The chains here are short and dependent;
// the FP64 pipe of this GPU issues one 32-lane instruction per ~64 cycles per scheduler,
// the FMA pipe one per cycle, so the pairs are the fast form and FP64 the exact-type one.
// Both store 16-byte elements (float4 hi/lo pairs or double2), so the tree's buffers and
// its launch shapes are the same.
#include <cuda_runtime.h>

#include <algorithm>

#include <type_traits>

#include "gbsbin_device.cuh"
#include "gbsbin_tree.cuh"

namespace gbsbin {
namespace {

template <class Ar>
__global__ void __launch_bounds__(ROOT_THREADS) k_tree_root(TreeArgs a, int parts) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char gsm_raw[];
  const int child = blockIdx.x / parts, part = blockIdx.x - child * parts;
  const int mc = a.m[1], tid = threadIdx.x;
  const int cols = a.has_gamma ? mc + 1 : mc, rows = cols;   // row mc: u', column mc: c'
  const E w = root_at<Ar>(a, 0, child);
  const int nb = a.nb[0], r0 = rows * part / parts, r1 = rows * (part + 1) / parts;
  // d, then the left factors of this part's rows times d
  E* d = reinterpret_cast<E*>(gsm_raw);                // nb
  E* ld = d + nb;                                      // (r1 - r0) x nb
  const E* lam = elem<Ar>(const_cast<float4*>(a.rlam));
  const E* B = elem<Ar>(const_cast<float4*>(a.rB));
  const E* ru = elem<Ar>(const_cast<float4*>(a.ru));
  for (int k = tid; k < nb; k += ROOT_THREADS)
    d[k] = Ar::mul(w, Ar::recip(Ar::add(Ar::one(), Ar::neg(Ar::mul(w, lam[k])))));
  __syncthreads();
  for (int q = tid; q < (r1 - r0) * nb; q += ROOT_THREADS) {
    const int i = r0 + q / nb, k = q - q / nb * nb;
    ld[q] = Ar::mul(d[k], i == mc ? ru[k] : Ar::conj(B[k * (mc + 1) + i]));
  }
  __syncthreads();
  for (int q = tid; q < (r1 - r0) * cols; q += ROOT_THREADS) {
    const int i = r0 + q / cols, j = q - q / cols * cols;
    E v = i == mc ? (j == mc ? Ar::zero() : elem<Ar>(a.u[0])[nb + j])
                  : j == mc ? elem<Ar>(a.c[0])[nb + i] : elem<Ar>(a.A[0])[(nb + i) * a.m[0] + nb + j];
    const E* li = ld + (i - r0) * nb;
    for (int k = 0; k < nb; ++k) v = Ar::fma(li[k], B[k * (mc + 1) + j], v);
    if (i == mc && j == mc) path_at<Ar>(a.path[1], child)->ex = Ar::add(v, path_at<Ar>(a.path[0], 0)->ex);
    else if (i == mc) elem<Ar>(a.u[1])[(long long)child * mc + j] = v;
    else if (j == mc) elem<Ar>(a.c[1])[(long long)child * mc + i] = v;
    else elem<Ar>(a.A[1])[(long long)child * mc * mc + i * mc + j] = v;
  }
  if (part == 0 && tid < 32) {                         // the child's path record, its exponent apart
    const PathRec<E> pr = root_path<Ar>(a, w);
    if (tid == 0) {
      PathRec<E>* out = path_at<Ar>(a.path[1], child);
      out->prod = pr.prod;
      out->meta = pr.meta;
      if (!a.has_gamma) out->ex = Ar::zero();
    }
  }
}

// Level l: one CTA per child; after the sweep warp 0 forms the child's path record while the others copy out its
// matrix and vectors.  (48 registers: five 256-thread CTAs per SM, so a 729-CTA level runs in one wave)
template <class Ar, bool ROOT>
__global__ void __maxnreg__(48) k_tree_level(TreeArgs a, int l, int span) {
  using E = typename Ar::E;
  extern __shared__ __align__(16) unsigned char gsm_raw[];
  const long long child = blockIdx.x;
  const Sweep<E> w = level_sweep<Ar, ROOT, SPAN_MAX>(a, l, span, child, gsm_raw);
  const int tid = threadIdx.x, nb = w.nb, m = w.m, mc = m - nb, cols = w.cols;
  if (tid >= 32) {                                   // the child's A', c', u' (warps 1..)
    const int t = tid - 32, LO = blockDim.x - 32;
    E* Ac = elem<Ar>(a.A[l + span]) + child * (long long)mc * mc;
    for (int idx = t; idx < mc * mc; idx += LO) {
      const int i = idx / mc, j = idx - (idx / mc) * mc;
      Ac[idx] = w.G[(nb + i) * cols + nb + j];
    }
    if (a.has_gamma) {
      E* cc = elem<Ar>(a.c[l + span]) + child * (long long)mc;
      E* uc = elem<Ar>(a.u[l + span]) + child * (long long)mc;
      for (int j = t; j < mc; j += LO) {
        cc[j] = w.G[(nb + j) * cols + m];
        uc[j] = w.G[m * cols + nb + j];
      }
    }
  } else {                                           // the child's path record (warp 0)
    const PathRec<E> pr = sweep_path<Ar, ROOT>(a, l, w);
    if (tid == 0) *path_at<Ar>(a.path[l + span], child) = pr;
  }
}


// Leaves: a team of NL lanes per evaluated point (32 / NL teams per warp), lane r holding
// row r of B = I - w A_leaf and of the right-hand side w c in registers.  Step kk
// broadcasts row kk from its lane; the rows below subtract their multiple of it (the
// right-hand side with them), so U and L^-1 (w c) come out together; the back substitution
// then broadcasts one solution entry per step.  Lane r keeps pivot r; the team reduces the
// path record into its first lane, which writes the point.
template <class Ar, int NL>
__global__ void __launch_bounds__(128) k_tree_leaf(TreeArgs a) {
  using E = typename Ar::E;
  constexpr int TEAMS = 32 / NL;
  const int lane = threadIdx.x & 31;
  const int team = lane / NL, r = lane - team * NL;
  const int base = team * NL;
  const long long leaf = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * TEAMS + team;
  const bool live = team < TEAMS && leaf < a.grid.n_eval;
  const int l = a.grid.L - 1;
  const int H = a.grid.half;
  const long long parent = live ? leaf / H : 0;
  const int k = live ? (int)(leaf - parent * H) : 0;
  const E w = root_at<Ar>(a, l, k);
  const E* Ap = elem<Ar>(a.A[l]) + parent * (long long)NL * NL + (long long)(live ? r : 0) * NL;
  const E one = Ar::one(), zero = Ar::zero();
  E b[NL];
#pragma unroll
  for (int j = 0; j < NL; ++j) {
    b[j] = Ar::neg(Ar::mul(w, Ap[j]));
    if (j == r) b[j] = Ar::add(b[j], one);
  }
  E y = zero, u = zero;
  if (a.has_gamma) {
    y = Ar::mul(w, elem<Ar>(a.c[l])[parent * NL + (live ? r : 0)]);
    u = elem<Ar>(a.u[l])[parent * NL + (live ? r : 0)];
  }
  E myinv = one, mypiv = one;
  // the step loop stays rolled (an unrolled copy per step overflows the instruction
  // cache); the row stays in registers, entries left of the step skipped by a uniform test
#pragma unroll 1
  for (int kk = 0; kk < NL; ++kk) {
    const int src = base + kk;
    E bk = b[0];
#pragma unroll
    for (int j = 1; j < NL; ++j)
      if (j == kk) bk = b[j];
    const E piv = shfl(bk, src);
    const E ykk = shfl(y, src);
    const E inv = Ar::recip(piv);
    if (r == kk) {
      myinv = inv;
      mypiv = piv;
    }
    const bool below = r > kk;
    const E li = Ar::mul(bk, inv);                   // used by the rows below only
#pragma unroll
    for (int j = 1; j < NL; ++j) {
      if (j <= kk) continue;
      const E rj = shfl(b[j], src);
      if (below) b[j] = Ar::fms(b[j], li, rj);
    }
    if (below) y = Ar::fms(y, li, ykk);
  }
  // the path record: lane r holds pivot r; a tree over the team (partner r + o, o = 8, 4,
  // 2, 1) leaves the product (rescaled by powers of two), the argument sum and the smallest
  // real part in lane 0, which folds in the parent's record
  PathRec<E> pr = *path_at<Ar>(a.path[l], parent);
  {
    E p = mypiv;
    const float pre = Ar::re(p), pim = Ar::im(p);
    float arg = atan2f(pim, pre), mn = pre, e2 = 0.f;
    if (!(pre == pre) || !(pim == pim)) mn = -3.0e38f;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      if (o >= NL) continue;
      const int partner = (lane + o) & 31;
      const E q = shfl(p, partner);
      const float qa = __shfl_sync(0xffffffffu, arg, partner), qm = __shfl_sync(0xffffffffu, mn, partner);
      const float qe = __shfl_sync(0xffffffffu, e2, partner);
      if (r + o < NL) {
        p = Ar::mul(p, q);
        e2 += qe + (float)Ar::normalise(p);
        arg = __fadd_rn(arg, qa);
        mn = fminf(mn, qm);
      }
    }
    E prod = Ar::mul(pr.prod, p);
    const float e = pr.meta.y + e2 + (float)Ar::normalise(prod);
    pr.prod = prod;
    pr.meta = make_float4(__fadd_rn(pr.meta.x, arg), e, fminf(pr.meta.z, mn), 0.f);
  }
  E ex = pr.ex;
  if (a.has_gamma) {                                  // x = U^-1 y, ex += u^T x
    E acc = y, x = zero;
#pragma unroll
    for (int t = NL - 1; t >= 0; --t) {
      if (r == t) x = Ar::mul(acc, myinv);
      const E xt = shfl(x, base + t);
      if (r < t) acc = Ar::fms(acc, b[t], xt);
    }
    E part = Ar::mul(u, x);
#pragma unroll
    for (int t = 0; t < NL; ++t) ex = Ar::add(ex, shfl(part, base + t));
  }
  if (!live || r != 0) return;
  const double LN2 = 0.693147180559945309417232121458;
  const double2 P = Ar::to(pr.prod), X = Ar::to(ex);
  double* f = a.ldfin + 6 * leaf;
  f[0] = P.x;
  f[1] = P.y;
  f[2] = (double)pr.meta.x;
  f[3] = -0.5 * (double)pr.meta.y * LN2 + 0.5 * X.x;
  f[4] = 0.5 * X.y;
  f[5] = 0.0;
  a.minpiv[leaf] = (double)pr.meta.z;
  if (a.gout) {                                      // G = q / q(1) = (P0 / P)^(1/2) 2^((e0 - e)/2) (-1)^w
    const float TWO_PI = 6.28318530717958647692f;
    const float argP = atan2f(Ar::im(pr.prod), Ar::re(pr.prod));
    const float m = rintf((pr.meta.x - argP) / TWO_PI);         // winding of log det at this point
    E p0;
    if constexpr (std::is_same<Ar, ArDF>::value) p0 = a.p0df;
    else p0 = Ar::from(make_double2(a.p0re, a.p0im));
    const E Z = Ar::mul(p0, Ar::recip(pr.prod));
    const float kz = rintf((atan2f(Ar::im(Z), Ar::re(Z)) - (a.p0arg - argP)) / TWO_PI);
    const int wind = (int)(kz + m - a.m0);
    const int d = (int)(a.e0 - pr.meta.y);
    const int hexp = (d - (d & 1)) / 2;
    if constexpr (std::is_same<Ar, ArDF>::value) {
      // sqrt(2) and 2^hexp applied to the pair (exact power-of-two scaling), one conversion
      E g = Ar::csqrt(Z);
      if (d & 1) {
        constexpr double SQ2 = 1.41421356237309504880;
        constexpr float SQ2_HI = (float)SQ2;
        constexpr float SQ2_LO = (float)(SQ2 - (double)SQ2_HI);
        g = Ar::mul(g, make_float4(SQ2_HI, 0.f, SQ2_LO, 0.f));
      }
      if (hexp >= -126 && hexp <= 127) {
        const float sc = __uint_as_float((unsigned)(127 + hexp) << 23) * ((wind & 1) ? -1.f : 1.f);
        g = make_float4(g.x * sc, g.y * sc, g.z * sc, g.w * sc);
        if (a.gout_df) reinterpret_cast<float4*>(a.gout)[leaf] = g;   // the DFT reads pairs
        else a.gout[leaf] = Ar::to(g);
      } else {
        const double2 gd = Ar::to(g);
        const double sg = (wind & 1) ? -1.0 : 1.0;
        const double2 gv = make_double2(sg * ldexp(gd.x, hexp), sg * ldexp(gd.y, hexp));
        if (a.gout_df) reinterpret_cast<float4*>(a.gout)[leaf] = Ar::from(gv);
        else a.gout[leaf] = gv;
      }
    } else {
      double2 g = Ar::to(Ar::csqrt(Z));
      if (d & 1) {
        g.x *= 1.41421356237309504880;
        g.y *= 1.41421356237309504880;
      }
      const double sg = (wind & 1) ? -1.0 : 1.0;
      a.gout[leaf] = make_double2(sg * ldexp(g.x, hexp), sg * ldexp(g.y, hexp));
    }
  }
}

template <class Ar, int NL>
cudaError_t launch_leaf(const TreeArgs& a, cudaStream_t s) {
  constexpr int TEAMS = 32 / NL;
  const long long warps = (a.grid.n_eval + TEAMS - 1) / TEAMS;
  const long long blocks = (warps + 1) / 2;           // two warps per CTA: spread evenly over SMs
  k_tree_leaf<Ar, NL><<<(unsigned)blocks, 64, 0, s>>>(a);
  return cudaGetLastError();
}

// The first level on its own: its rows split so that the CTAs fill the SMs.
template <class Ar>
cudaError_t launch_root(const TreeArgs& a, int num_sms, cudaStream_t s) {
  const long long nodes = a.grid.radix[0];
  const int rows = a.m[1] + (a.has_gamma ? 1 : 0);
  const int parts = (int)std::max<long long>(1, std::min<long long>(rows, num_sms / nodes));
  const size_t smem = sizeof(float4) * (size_t)a.nb[0] * ((rows + parts - 1) / parts + 1);
  if (smem > 48 * 1024) {
    const cudaError_t err = cudaFuncSetAttribute(k_tree_root<Ar>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
  }
  k_tree_root<Ar><<<(unsigned)(nodes * parts), ROOT_THREADS, smem, s>>>(a, parts);
  return cudaGetLastError();
}

// Children of the launch that starts at level l (nodes of them above it): levels whose children would fill fewer than
// half the SMs take the next level into the same launch (a level's fixed costs - launch, fill from the parent, copy-out,
// path record - are then paid once), up to SPAN_MAX groups and while a level remains before the leaves.
long long level_children(const GridDesc& g, int l, long long nodes, int num_sms, int* span) {
  long long children = nodes * g.radix[l];
  for (*span = 1; *span < SPAN_MAX && l + *span + 1 < g.L && 2 * children < num_sms; ++*span) children *= g.radix[l + *span];
  return children;
}

// The first level on its own, or formed by every child of the second's launch, which saves a launch and the way
// through memory and repeats the sums per child.  In clocks, per turn of the SMs: m^2 entries of nb products and
// ~10 more, 1 each in FP64 and 0.35 in pairs, at least a CTA's turn; against ~11000 saved in FP64, 7600 in pairs.  Whole
// tables, apart / fused: three groups of 8 rows, FP64, 81 children 54.5 / 48.1 us, 256 59.4 / 59.4, 729 81.9 / 111,
// 1600 145 / 204; of 12 rows 69.6 / 73.7, 80 / 94, 141 / 203, 291 / 422; in pairs 8 rows 38.0 / 34.8, 44.0 / 42.5, 53 / 64, 64 / 89;
// 12 rows 49.2 / 47.0, 55.3 / 55.4, 74 / 93, 112 / 159; four of 8 rows, pairs 53.2 / 49.8, FP64 87.8 / 88.1.
bool first_level_fused(const TreeArgs& a, const GridDesc& g, int num_sms, bool fp64) {
  if (g.L <= 2) return false;
  int span = 1;
  const long long turns = (level_children(g, 1, g.radix[0], num_sms, &span) + num_sms - 1) / num_sms;
  const double sums = (a.nb[0] + 10.0) * a.m[1] * a.m[1] * (fp64 ? 1.0 : 0.35);
  return (double)turns * std::max(fp64 ? 5400.0 : 3000.0, sums) < (fp64 ? 11000.0 : 7600.0);
}

// Level 0 from the spectral form or, where the plan does without it, by elimination like the other levels.
template <class Ar>
cudaError_t launch_tree(const TreeArgs& a, int num_sms, cudaStream_t s, int* launches) {
  cudaError_t err = cudaSuccess;
  *launches = 1;                                      // the leaves
  constexpr bool fp64 = !std::is_same<Ar, ArDF>::value;
  long long nodes = a.spectral ? a.grid.radix[0] : 1;
  bool fused = a.spectral && first_level_fused(a, a.grid, num_sms, fp64);
  if (a.spectral && !fused) {
    if ((err = launch_root<Ar>(a, num_sms, s)) != cudaSuccess) return err;
    ++*launches;
  }
  for (int l = a.spectral ? 1 : 0; l + 1 < a.grid.L;) {
    int span = 1, nb = a.nb[l];
    const long long children = level_children(a.grid, l, nodes, num_sms, &span);
    for (int g = 1; g < span; ++g) nb += a.nb[l + g];
    const size_t smem = tree_level_smem_bytes(nb, a.m[l]) + (fused ? sizeof(float4) * ((size_t)a.nb[0] * (a.m[1] + 2) + 3) : 0);
    auto kernel = fused ? k_tree_level<Ar, true> : k_tree_level<Ar, false>;
    if (smem > 48 * 1024) {
      err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (err != cudaSuccess) return err;
    }
    const int m = a.m[l], width = m * m;              // entries of the first elimination step
    const int threads = width >= 1024 || fused ? 512 : width >= 256 ? 256 : 128;
    kernel<<<(unsigned)children, threads, smem, s>>>(a, l, span);
    ++*launches;
    err = cudaGetLastError();
    if (err != cudaSuccess) return err;
    nodes = children;
    l += span;
    fused = false;
  }
  switch (a.m[a.grid.L - 1]) {
    case 2: return launch_leaf<Ar, 2>(a, s);
    case 4: return launch_leaf<Ar, 4>(a, s);
    case 6: return launch_leaf<Ar, 6>(a, s);
    case 8: return launch_leaf<Ar, 8>(a, s);
    case 10: return launch_leaf<Ar, 10>(a, s);
    case 12: return launch_leaf<Ar, 12>(a, s);
    case 14: return launch_leaf<Ar, 14>(a, s);
    case 16: return launch_leaf<Ar, 16>(a, s);
    default: return cudaErrorInvalidConfiguration;
  }
}

}  // namespace

// The spectral form saves the first level's pivots in every child of the launch that would hold them, and costs the
// host an eigendecomposition per state, so it is taken where a state with one table gains or loses no more than 3 us (then
// further tables of the state decide).  Both in us, fitted to measured calls: the host 1.5 + 1e-3 nb^3 + 1.9e-3 nb^2 x
// (columns) (8 rows and 26 columns 5, 14 and 30 16, 32 and 18 64, 48 and 18 187); a pivot saved, per turn of the
// SMs, grows with the matrix, 0.04 m - 0.35 in FP64 and 0.0105 m in pairs (first groups of 14 of 42 rows 18 and 6 us, 32 of
// 48 49 and 18, 48 of 64 107 and 41).  set_state and one table at 48 of 64 rows in pairs: 332 us by elimination, 442
// from the spectral form; at 14 of 42 rows in FP64 194 and 184.
bool tree_spectral_suits(const TreeArgs& a, const GridDesc& g, int num_sms, bool fp64) {
  int span = 1;
  const double turns = (double)((level_children(g, 0, 1, num_sms, &span) + num_sms - 1) / num_sms);
  const double nb = a.nb[0], m = a.m[0], cols = m - nb + 2.0;
  const double host = 1.5 + 1e-3 * nb * nb * nb + 1.9e-3 * nb * nb * cols;
  const double gain = nb * turns * std::max(0.0, fp64 ? 0.04 * m - 0.35 : 0.0105 * m);
  // (apart from the second level's launch it is one launch more, ~4 us: groups of 4 rows, 729 children, pairs 43 us
  // apart, 39 by elimination)
  return host <= gain + 3.0 && (gain >= 4.0 || g.L == 2 || first_level_fused(a, g, num_sms, fp64));
}

size_t tree_level_smem_bytes(int nb, int m) { return sizeof(float4) * ((size_t)(m + 1) * (m + 1) + nb + 2 * (m + 1)); }

// Leaf blocks of 2, 4, ..., 16 rows have a kernel instance (0: not supported).
int tree_leaf_threads(int n) { return (n >= 2 && n <= 16 && n % 2 == 0) ? n : 0; }

cudaError_t launch_tree_root_fp64(const TreeArgs& a, int num_sms, cudaStream_t s) { return launch_root<ArF64>(a, num_sms, s); }

cudaError_t launch_points_tree(const TreeArgs& a, bool fp64, int num_sms, cudaStream_t s, int* launches) {
  return fp64 ? launch_tree<ArF64>(a, num_sms, s, launches) : launch_tree<ArDF>(a, num_sms, s, launches);
}

}  // namespace gbsbin
