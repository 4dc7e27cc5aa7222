// Fock inputs through a lossy linear circuit (arXiv:2412.17742, App. C) by a convolution over
// sub-multisets of the input photons.
//
// The generating function G(z) = perm(B(z)[p, p]) / p! is the coefficient of x^p in the product of N
// linear forms (B(z) x)_row, each input j giving p_j equal rows, and B(z) = B_0 + sum_l z_l B_l is linear in
// z.  The product of the first r rows is sum_m F_r[m](z) x^m over sub-multisets |m| = r, F_r[m] a
// polynomial of degree <= r in z, with
//   F_r[m] = sum_{k, m_k > 0} F_{r-1}[m - e_k] (B_0 + sum_l z_l B_l)[row_r, k],
// and splitting the rows in two halves, G = sum_m F1[m] F2[p - m], whose coefficients are the table
// itself (folded where a group's radix is smaller than its degree): no grid points, no transform.
// N = 16 single photons in three groups take 3.2e8 complex multiply-adds for the two halves (12870
// states of 165 monomials each) and 3.5e8 for the sum over states, against 1.4e9 complex products and
// 4e9 additions of the walk over 2^15 nodes x 2601 grid points (gbsbin_fock.cu), which shards keep.
//
// Arithmetic: 64-bit integer sums of products of digits (mad.wide.s32).  A state's monomials are 56-bit
// integers with one exponent per state, in two 28-bit digits; a complex product is three real ones (Karatsuba),
// each three digit products (the lo x lo term lies below the rounding), summed exactly over (k, t) and
// rounded once per layer.  On the unit circle sum_m |F_r[m](z)|^2 <= 1 for a contraction T (the amplitudes of
// r photons), so nothing cancels against larger intermediate terms.  The sum over states takes each
// monomial at its column's exponent, in 2 x 28 bits for plans of FP32 pairs of up to 2^14 states (the sums' upper parts
// moved out every 16 states) and 3 x 20 bits for the others, where products of two small entries must not be lost.
// (With states of 52 bits and the pairs' sum in 2 x 25 bits, pairs plans of 14 photons through a circuit of 2 to 5%
// transmission, whose small entries' products are all lo x lo, had 50 times the walk's error.)
// Relative error of whole tables against 80-bit arithmetic, 6 / 8 / 10 / 11 photons in two groups: transmissions of 40 to 90%
// 4.0 / 4.3 / 4.6 / 4.6e-16 (the walk: FP64 6.3 / 8.7 / 12 / 13e-16, pairs 4.0e-14 / 2.9e-14 / 1.5e-14 / 1.1e-14), of 2 to 5% 1.3 / 1.7 / 2.1 / 2.5e-16
// (pairs 1.1 / 1.7 / 3.4 / 3.3e-16; the walk 5.1 / 7.4 / 9.9 / 11e-16 and 4.7e-14 to 1.1e-14).
// Measured in a register-tiled loop, a complex multiply-add takes a scheduler 47 clocks with two digits, 68 in pairs of FP32
// and 424 in FP64.
//
// k_conv_layer: a warp per state (of either half); lane k finds the predecessor m - e_k; the factor's digits,
// shifted to the largest predecessor exponent, go to shared memory; lanes then hold a monomial each (six
// 64-bit sums) and run over (k, t).  Eight CTAs of four warps per SM, one monomial a lane: bound by the
// multiply-adds' issue like the variants of two and three monomials a lane, which hold fewer warps (whole
// tables at N = 16, three groups: 1340 us, 1380 and 1400).
// k_conv_scale: the last layers at their columns' scale, once per entry.
// k_conv_sum: a CTA of three warps per 24 x 16 tile of monomial pairs and chunk of states, 2 x 2 outputs a
// thread, the states copied asynchronously two stages ahead; the chunk is set so that the CTAs fill the SMs
// once.  (24 x 24 with 2 x 3 outputs: 646 us for the launch against 600, with fewer warps to hide the chains.)
// k_conv_table: a warp per table entry adds its monomial pairs over all chunks in a fixed order.
// N = 16, three groups, whole table: 6807 us by the walk in pairs of FP32 (31000 in FP64), 1350 us here.
#include "gbsbin_fock_conv.h"

namespace gbsbin {
namespace {

constexpr int kLayerWarps = 4;
constexpr int kSumThreads = 96;
constexpr int kStage = 16;                 // states staged at a time by k_conv_sum
constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ void mad(long long& c, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
}
// v >> s rounded to nearest (s > 0), v << -s otherwise; 0 from s = 63 on
__device__ __forceinline__ long long shift_round(long long v, int s) {
  if (s <= 0) return v << -s;
  if (s >= 63) return 0;
  return (v + (1ll << (s - 1))) >> s;
}
__device__ __forceinline__ int bit_length(long long v) {                  // of |v|
  return 64 - __clzll(v < 0 ? -v : v);
}

// CT1 = L + 1 at compile time (the predecessors' offsets then stay in registers), 0: any L.
template <int CT1>
__global__ void __launch_bounds__(kLayerWarps * 32, 8) k_conv_layer(FockConvArgs a, FockConvLayer y) {
  extern __shared__ int sm[];
  const int T1 = CT1 ? CT1 : a.L + 1, nd = T1 * y.nc;
  int* s_down = sm;                                          // [t][e] of this layer, as offsets into a predecessor
  int* s_max = s_down + nd;                                  // column exponents of the two halves
  int* s_b = sm + ((nd + 2 * y.nc + 1) & ~1) + threadIdx.x / 32 * (a.nin * T1 * 6);   // this warp's factor digits,
                                                             // 6 per (k, t), 8-byte aligned
  for (int i = threadIdx.x; i < nd; i += blockDim.x) {
    const int t = i / y.nc, e = i - t * y.nc, d = a.down[t * a.ndown + e];
    s_down[i] = d >= 0 && d < y.nc0 ? d : y.nc0;   // a row's entry past its last is zero
  }
  for (int i = threadIdx.x; i < 2 * y.nc; i += blockDim.x) s_max[i] = GBSBIN_FC_NONE;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long items = (long long)y.states * y.halves;
  for (long long it = blockIdx.x * kLayerWarps + threadIdx.x / 32; it < items; it += (long long)gridDim.x * kLayerWarps) {
    const int half = it >= y.states ? 1 : y.half0, i = (int)(it >= y.states ? it - y.states : it);
    const int in = (y.r - 1) & 1, out = y.r & 1;
    const int code = a.order[y.first + i];
    int pred = -1, ep = GBSBIN_FC_NONE;
    if (lane < a.nin && (code / a.stride[lane]) % a.radix[lane] > 0) {
      pred = a.rank[code - a.stride[lane]];
      ep = y.r == 1 ? a.E0[0] : a.E[half][in][pred];
    }
    const unsigned mask = __ballot_sync(kAll, pred >= 0);
    const int emax = __reduce_max_sync(kAll, ep);
    __syncwarp();
    for (int q0 = 0; q0 < a.nin * T1; q0 += 32) {            // the factor's digits at the common exponent
      const int q = q0 + lane;
      const int ek = __shfl_sync(kAll, ep, min(q / T1, 31));
      if (q >= a.nin * T1) continue;
      const longlong2 b = a.B[((size_t)y.row[half] * a.nin) * T1 + q];
      const int s = min(63, emax - ek);
      const long long br = shift_round(b.x, s), bi = shift_round(b.y, s);
      int* o = s_b + 6 * q;
      digits<kConvDigit>(br, o[0], o[1]);
      digits<kConvDigit>(bi, o[2], o[3]);
      o[4] = o[0] + o[2];
      o[5] = o[1] + o[3];
    }
    __syncwarp();
    const int4* Fin = y.r == 1 ? a.F0 : a.F[half][in];
    int4* Fout = a.F[half][out] + (size_t)i * (y.nc + 1);
    longlong2* raw = reinterpret_cast<longlong2*>(Fout);     // a lane's own entries, until the state's exponent is known
    long long big = 0;
    for (int c0 = 0; c0 < y.nc; c0 += 32) {                  // a monomial a lane
      const int e = c0 + lane;
      long long m1h = 0, m1l = 0, m2h = 0, m2l = 0, m3h = 0, m3l = 0;
      auto offset = [&](int t) { return e < y.nc ? s_down[t * y.nc + e] : y.nc0; };
      int dn[CT1 ? CT1 : 1];
      if (CT1) {
#pragma unroll
        for (int t = 0; t < CT1; ++t) dn[t] = offset(t);
      }
      auto term = [&](const int4* src, int k, int t, int d) {
        const int2* bp = reinterpret_cast<const int2*>(s_b + 6 * (k * T1 + t));
        const int2 br = bp[0], bi = bp[1], bs = bp[2];
        const int4 f = src[d];
        mad(m1h, f.x, br.x);
        mad(m1l, f.x, br.y);
        mad(m1l, f.y, br.x);
        mad(m2h, f.z, bi.x);
        mad(m2l, f.z, bi.y);
        mad(m2l, f.w, bi.x);
        const int sh = f.x + f.z, sl = f.y + f.w;
        mad(m3h, sh, bs.x);
        mad(m3l, sh, bs.y);
        mad(m3l, sl, bs.x);
      };
      for (unsigned left = mask; left; left &= left - 1) {
        const int k = __ffs(left) - 1;
        const int4* src = Fin + (size_t)__shfl_sync(kAll, pred, k) * (y.nc0 + 1);
        if (CT1) {
#pragma unroll
          for (int t = 0; t < CT1; ++t) term(src, k, t, dn[t]);
        } else {
          for (int t = 0; t < T1; ++t) term(src, k, t, offset(t));
        }
      }
      if (e < y.nc) {
        const long long rh = m1h - m2h, rl = m1l - m2l;
        const long long ih = m3h - m1h - m2h, il = m3l - m1l - m2l;
        const longlong2 v = make_longlong2(rh + shift_round(rl, kConvDigit), ih + shift_round(il, kConvDigit));
        raw[e] = v;
        big |= (v.x < 0 ? -v.x : v.x) | (v.y < 0 ? -v.y : v.y);
      }
    }
    // the state's exponent: its largest component in [2^55, 2^56)
    const unsigned bh = __reduce_or_sync(kAll, (unsigned)(big >> 32)), bl = __reduce_or_sync(kAll, (unsigned)big);
    const int len = bit_length((long long)bh << 32 | bl), s = len - kConvBits;
    const int eo = len == 0 || emax == GBSBIN_FC_NONE ? GBSBIN_FC_NONE : emax + s - (kConvRowBits - kConvBits);
    if (lane == 0) {
      a.E[half][out][i] = eo;
      Fout[y.nc] = make_int4(0, 0, 0, 0);
    }
    for (int e = lane; e < y.nc; e += 32) {
      const longlong2 v = raw[e];
      long long x = eo == GBSBIN_FC_NONE ? 0 : shift_round(v.x, s), z = eo == GBSBIN_FC_NONE ? 0 : shift_round(v.y, s);
      int4 f;
      digits<kConvDigit>(x, f.x, f.y);
      digits<kConvDigit>(z, f.z, f.w);
      Fout[e] = f;
      if (y.last[half]) {
        const int lx = max(bit_length(x), bit_length(z));
        if (lx > 0) atomicMax(s_max + half * y.nc + e, eo + lx - kConvBits);
      }
    }
  }
  if (y.last[0] || y.last[1]) {
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * y.nc; i += blockDim.x) {
      const int half = i / y.nc;
      if (y.last[half] && s_max[i] != GBSBIN_FC_NONE) atomicMax(a.colexp[half] + i - half * y.nc, s_max[i]);
    }
  }
}

// The last layers' entries at their columns' scale, in place: ND digits of BITS bits of
// round(F 2^(ND BITS - column exponent)), the third digits apart.  Once per entry here, where the contraction's
// tiles would repeat the 64-bit shifts seven times over.
template <int ND>
__global__ void __launch_bounds__(256) k_conv_scale(FockConvArgs a) {
  const int half = blockIdx.y, n = half ? a.n2 : a.n1, par = a.h[half] & 1;
  const unsigned total = (unsigned)a.states * (unsigned)(n + 1);
  for (unsigned q = blockIdx.x * 256u + threadIdx.x; q < total; q += gridDim.x * 256u) {
    const unsigned m = q / (unsigned)(n + 1), e = q - m * (unsigned)(n + 1);
    if ((int)e == n) continue;                 // the row's zero entry
    const int4 f = a.F[half][par][q];
    const int col = a.colexp[half][e], ex = a.E[half][par][m];
    int4 d = make_int4(0, 0, 0, 0);
    int2 d2 = make_int2(0, 0);
    if (col > GBSBIN_FC_NONE && ex != GBSBIN_FC_NONE) {
      constexpr int B = ND == 3 ? 20 : 28;
      const int s = min(63, kConvBits - ND * B + col - ex);
      long long x = shift_round(((long long)f.x << kConvDigit) + f.y, s), z = shift_round(((long long)f.z << kConvDigit) + f.w, s);
      if (ND == 3) {
        int lo;
        lo = ((int)((unsigned)x << (32 - B))) >> (32 - B);
        x = (x - lo) >> B;
        d2.x = lo;
        lo = ((int)((unsigned)z << (32 - B))) >> (32 - B);
        z = (z - lo) >> B;
        d2.y = lo;
      }
      digits<B>(x, d.x, d.y);
      digits<B>(z, d.z, d.w);
    }
    a.F[half][par][q] = d;
    if (ND == 3) a.F3[half][q] = d2;
  }
}

template <int BYTES>
__device__ __forceinline__ void copy_async(void* smem, const void* gmem, bool valid) {   // zeros when not valid
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  const int bytes = valid ? BYTES : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(s), "l"(gmem), "n"(BYTES), "r"(bytes) : "memory");
}

// One component product's ND (ND + 1) / 2 digit products, by weight.
template <int ND>
__device__ __forceinline__ void mad_digits(long long (&m)[ND], const int (&x)[ND], const int (&y)[ND]) {
#pragma unroll
  for (int w = 0; w < ND; ++w)
#pragma unroll
    for (int i = 0; i <= w; ++i) mad(m[w], x[i], y[w - i]);
}

// Sums over a chunk of states of F1[m][a] F2[p - m][b] for a 24 x 16 tile of (a, b); two stages of
// kStage states in flight.  With two digits of 28 bits a stage's sums reach 16 x 2^29 x 2^29 = 2^62, so after each their
// parts from bit kUpper on move to 32-bit sums (at most 2^22 a stage, 2^28 in all); three digits of 20 bits stay below
// 2^54 over all states.
constexpr int kUpper = 40;
template <int ND>
__global__ void __launch_bounds__(kSumThreads, ND == 3 ? 4 : 5) k_conv_sum(FockConvArgs a) {
  __shared__ int4 sx[2][kStage][kConvRows], sy[2][kStage][kConvCols];
  __shared__ int2 sx3[2][ND == 3 ? kStage : 1][kConvRows], sy3[2][ND == 3 ? kStage : 1][kConvCols];
  const int a0 = blockIdx.x * kConvRows, b0 = blockIdx.y * kConvCols;
  const int m0 = blockIdx.z * a.chunk, m1 = min(a.states, m0 + a.chunk);
  const int4* F1 = a.F[0][a.h[0] & 1];
  const int4* F2 = a.F[1][a.h[1] & 1];
  // warp w and lane / 8 give two rows, lane % 8 two columns
  const int r = (threadIdx.x >> 5) * 8 + ((threadIdx.x & 31) >> 3) * 2, q = (threadIdx.x & 7) * 2;
  long long m1s[2][2][ND] = {}, m2s[2][2][ND] = {}, m3s[2][2][ND] = {};
  constexpr int NU = ND == 2 ? 2 : 1;
  int u1s[2][2][NU] = {}, u2s[2][2][NU] = {}, u3s[2][2][NU] = {};
  auto move_up = [](long long& m, int& u) {
    u += (int)(m >> kUpper);
    m &= (1ll << kUpper) - 1;
  };
  // 24 threads per row of the first half (in order), 16 per row of the second (the complement's)
  const int xc = threadIdx.x % kConvRows, xs = threadIdx.x / kConvRows;
  const int yc = threadIdx.x % kConvCols, ys = threadIdx.x / kConvCols;
  auto stage = [&](int ms, int buf) {
    const bool vx = a0 + xc < a.n1, vy = b0 + yc < a.n2;
    for (int st = xs; st < kStage; st += kSumThreads / kConvRows) {
      const bool v = vx && ms + st < m1;
      const size_t o = v ? (size_t)(ms + st) * (a.n1 + 1) + a0 + xc : 0;
      copy_async<16>(&sx[buf][st][xc], F1 + o, v);
      if (ND == 3) copy_async<8>(&sx3[buf][st][xc], a.F3[0] + o, v);
    }
    for (int st = ys; st < kStage; st += kSumThreads / kConvCols) {
      const bool v = vy && ms + st < m1;
      const size_t o = v ? (size_t)a.rank[a.full - a.order[a.first + ms + st]] * (a.n2 + 1) + b0 + yc : 0;
      copy_async<16>(&sy[buf][st][yc], F2 + o, v);
      if (ND == 3) copy_async<8>(&sy3[buf][st][yc], a.F3[1] + o, v);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // an entry's digits: real, imaginary and their sum
  auto entry = [](int4 f, int2 f3, int (&re)[ND], int (&im)[ND], int (&su)[ND]) {
    re[0] = f.x;
    re[1] = f.y;
    im[0] = f.z;
    im[1] = f.w;
    if constexpr (ND == 3) {
      re[2] = f3.x;
      im[2] = f3.y;
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) su[d] = re[d] + im[d];
  };
  stage(m0, 0);
  int buf = 0;
  for (int ms = m0; ms < m1; ms += kStage, buf ^= 1) {
    if (ms + kStage < m1) {
      stage(ms + kStage, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
#pragma unroll 4
    for (int st = 0; st < kStage; ++st) {
      const int st3 = ND == 3 ? st : 0;
      int xr[2][ND], xi[2][ND], xu[2][ND];
#pragma unroll
      for (int i = 0; i < 2; ++i) entry(sx[buf][st][r + i], sx3[buf][st3][r + i], xr[i], xi[i], xu[i]);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        int yr[ND], yi[ND], yu[ND];
        entry(sy[buf][st][q + j], sy3[buf][st3][q + j], yr, yi, yu);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          mad_digits<ND>(m1s[i][j], xr[i], yr);
          mad_digits<ND>(m2s[i][j], xi[i], yi);
          mad_digits<ND>(m3s[i][j], xu[i], yu);
        }
      }
    }
    if constexpr (ND == 2) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            move_up(m1s[i][j][w], u1s[i][j][w]);
            move_up(m2s[i][j][w], u2s[i][j][w]);
            move_up(m3s[i][j][w], u3s[i][j][w]);
          }
    }
    __syncthreads();                             // the buffer is refilled by the next iteration's stage
  }
  double2* out = a.parts + (size_t)blockIdx.z * a.n1 * a.n2;
  const int exponent = *a.exponent;
  constexpr int B = ND == 3 ? 20 : 28;
  const double k = 1.0 / (double)(1 << B);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int ea = a0 + r + i, eb = b0 + q + j;
      if (ea >= a.n1 || eb >= a.n2) continue;
      const int ca = a.colexp[0][ea], cb = a.colexp[1][eb];
      double2 v = make_double2(0.0, 0.0);
      if (ca > GBSBIN_FC_NONE && cb > GBSBIN_FC_NONE) {
        double re = 0.0, im = 0.0;               // from the lowest weight up
#pragma unroll
        for (int w = ND - 1; w >= 0; --w) {
          double r = (double)(m1s[i][j][w] - m2s[i][j][w]), q = (double)(m3s[i][j][w] - m1s[i][j][w] - m2s[i][j][w]);
          if constexpr (ND == 2) {
            constexpr double up = (double)(1ll << kUpper);
            r = fma((double)(u1s[i][j][w] - u2s[i][j][w]), up, r);
            q = fma((double)(u3s[i][j][w] - u1s[i][j][w] - u2s[i][j][w]), up, q);
          }
          re = fma(re, k, r);
          im = fma(im, k, q);
        }
        const int s = ca + cb + exponent - 2 * B;
        v = make_double2(ldexp(re, s), ldexp(im, s));
      }
      out[(size_t)ea * a.n2 + eb] = v;
    }
}

constexpr int kTableWarps = 8;
__global__ void __launch_bounds__(kTableWarps * 32) k_conv_table(FockConvArgs a) {
  __shared__ double s_sum[kTableWarps], s_im[kTableWarps];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t np = (size_t)a.n1 * a.n2;
  double sum = 0.0, im = 0.0;
  for (long long t = (long long)blockIdx.x * kTableWarps + w; t < a.table_size; t += (long long)gridDim.x * kTableWarps) {
    double2 v = make_double2(0.0, 0.0);
    for (int i = a.pair_first[t] + lane; i < a.pair_first[t + 1]; i += 32) {
      const double2* src = a.parts + a.pair_list[i];
      for (int c = 0; c < a.nchunks; ++c) {
        const double2 x = src[(size_t)c * np];
        v.x += x.x;
        v.y += x.y;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(kAll, v.x, o);
      v.y += __shfl_xor_sync(kAll, v.y, o);
    }
    if (lane == 0) a.P[t] = v.x;
    sum += v.x;
    im = fmax(im, fabs(v.y));
  }
  if (!a.diag) return;
  if (lane == 0) {
    s_sum[w] = sum;
    s_im[w] = im;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < kTableWarps; ++i) {
      sum += s_sum[i];
      im = fmax(im, s_im[i]);
    }
    double* d = a.diag + 4 * blockIdx.x;
    d[0] = sum;
    d[1] = im;
    d[2] = 1.0;
    d[3] = 0.0;
    if (blockIdx.x == 0) {
      a.diag[4 * GBSBIN_DIAG_SLOTS] = 0.0;
      a.diag[4 * GBSBIN_DIAG_SLOTS + 1] = 0.0;
      a.diag[4 * GBSBIN_DIAG_SLOTS + 2] = (double)gridDim.x;
    }
  }
}

}  // namespace

int fock_conv_slots_per_sm(int nd) {
  int n = 0;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, nd == 3 ? k_conv_sum<3> : k_conv_sum<2>, kSumThreads, 0) == cudaSuccess ? n : 0;
}

size_t fock_conv_layer_smem(int nin, int L, int nc) {
  return ((size_t)(L + 3) * nc + 1 + (size_t)kLayerWarps * nin * (L + 1) * 6) * sizeof(int);
}

cudaError_t launch_fock_conv(const FockConvArgs& a, const FockConvLayer* layers, int nlayers, int num_sms,
                             cudaStream_t s, int* launches) {
  // 0x80808080 lies below every exponent; the two halves' columns are adjacent
  const cudaError_t e = cudaMemsetAsync(a.colexp[0], 0x80, ((size_t)a.n1 + a.n2) * sizeof(int), s);
  if (e != cudaSuccess) return e;
  for (int l = 0; l < nlayers; ++l) {
    const FockConvLayer& y = layers[l];
    const size_t smem = fock_conv_layer_smem(a.nin, a.L, y.nc);
    const long long items = (long long)y.states * y.halves;
    long long grid = (items + kLayerWarps - 1) / kLayerWarps;
    if (grid > 8LL * num_sms) grid = 8LL * num_sms;
    switch (a.L) {
      case 1: k_conv_layer<2><<<(unsigned)grid, kLayerWarps * 32, smem, s>>>(a, y); break;
      case 2: k_conv_layer<3><<<(unsigned)grid, kLayerWarps * 32, smem, s>>>(a, y); break;
      case 3: k_conv_layer<4><<<(unsigned)grid, kLayerWarps * 32, smem, s>>>(a, y); break;
      default: k_conv_layer<0><<<(unsigned)grid, kLayerWarps * 32, smem, s>>>(a, y);
    }
  }
  const long long entries = (long long)a.states * (a.n2 + 1);
  const dim3 gs((unsigned)(entries < 256LL * 8 * num_sms ? (entries + 255) / 256 : 8LL * num_sms), 2);
  const dim3 g((a.n1 + kConvRows - 1) / kConvRows, (a.n2 + kConvCols - 1) / kConvCols, a.nchunks);
  if (a.nd == 3) {
    k_conv_scale<3><<<gs, 256, 0, s>>>(a);
    k_conv_sum<3><<<g, kSumThreads, 0, s>>>(a);
  } else {
    k_conv_scale<2><<<gs, 256, 0, s>>>(a);
    k_conv_sum<2><<<g, kSumThreads, 0, s>>>(a);
  }
  long long tb = (a.table_size + kTableWarps - 1) / kTableWarps;
  if (tb > GBSBIN_DIAG_SLOTS) tb = GBSBIN_DIAG_SLOTS;
  k_conv_table<<<(unsigned)tb, kTableWarps * 32, 0, s>>>(a);
  *launches = nlayers + 3;
  return cudaGetLastError();
}

}  // namespace gbsbin
