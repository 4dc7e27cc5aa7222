// Fock inputs by a convolution over sub-multisets of the photons: the interface between the host plan
// (gbsbin_fock_host.cpp) and the kernels (gbsbin_fock_conv.cu).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "gbsbin_internal.h"

namespace gbsbin {

#define GBSBIN_FC_NONE (-(1 << 28))       // exponent of an all-zero state or column

// A state's monomials are integers of kConvBits bits, value x 2^(exponent - kConvBits), in two digits of kConvDigit.
// Coefficients in fixed point, round(b 2^kConvRowBits / 2^e) with e the row's exponent: components up to 2^55, high
// digits up to 2^27 and the sum of two (the third factor of a complex product by three real ones) up to 2^28, and a
// row's sum of component magnitudes below 2^59. A layer's 64-bit sums then stay below 2^63 for up to kConvMaxTerms
// terms (the largest: sums of 2^29 x 2^28 per term and 2^28 x 2^31), and its results are three bits finer than a state's.
constexpr int kConvDigit = 28, kConvBits = 2 * kConvDigit;
constexpr int kConvMaxTerms = 56;         // photons of a layer, or occupied inputs, times L + 1
constexpr int kConvRowBits = 55;
// e of a row whose largest component is `big` and whose component magnitudes add to `all`: big < 2^e, all < 16 x 2^e
inline int conv_row_exponent(double big, double all) {
  int e = 0, ea = 0;
  std::frexp(big, &e);
  std::frexp(all * 1.0001, &ea);
  return std::max(e, ea - 4);
}
inline long long conv_fixed(double v, int e) { return std::llrint(std::ldexp(v, kConvRowBits - e)); }
template <int BITS>
__host__ __device__ __forceinline__ void digits(long long v, int& hi, int& lo) {   // v = hi 2^BITS + lo, |lo| <= 2^(BITS-1)
  lo = ((int)((unsigned)v << (32 - BITS))) >> (32 - BITS);
  hi = (int)((v - lo) >> BITS);
}
struct FockConvArgs {
  int nin, L, N, h[2];                    // occupied inputs, groups, photons, factors of each half
  int stride[GBSBIN_FOCK_MAX_IN];         // code of a state m: sum m_k stride[k]
  int radix[GBSBIN_FOCK_MAX_IN];          // p_k + 1
  int full;                               // code of p
  const int* rank;                        // code -> index within its layer
  const int* order;                       // layer after layer: index -> code
  const int* down;                        // [t][e]: monomial e without z_{t-1} (t = 0: e itself), -1: none
  int ndown;                              // monomials of degree <= h[1] (the stride of `down`)
  const longlong2* B;                     // [row][k][t], fixed point
  const int4* F0;                         // the empty product: digits of 2^(kConvBits - 1), and its exponent 1
  const int* E0;
  int4* F[2][2];                          // [half][parity]: state x monomial, digits (re hi, lo, im hi, lo)
  int* E[2][2];                           // [half][parity]: the state's exponent
  int nd;                                 // digits of the sum over states: 2 (28 bits; pairs, up to 2^14 states) or 3 (20 bits)
  int2* F3[2];                            // with three: the last layers' third digits (re, im)
  int* colexp[2];                         // per monomial of the last layer: exponent of its largest entry
  int states, first, n1, n2;              // last layer of the first half: states, its codes in order; monomials
                                          // of each half
  int chunk, nchunks;                     // states per contraction CTA
  const int* exponent;                    // sum of the rows' exponents (of the circuit, so in device memory: a captured
                                          // launch then serves later circuits)
  double2* parts;                         // nchunks x n1 x n2
  const int* pair_first;                  // table entry -> its pairs (a n2 + b) in pair_list
  const int* pair_list;
  long long table_size;
  double* P;
  double* diag;
};
// One layer r >= 1 of both halves (those that reach it): states of r photons, nc monomials of degree
// <= r, nc0 of degree <= r - 1; order[first ..] are its codes.  `last[half]` asks for the column maxima.
struct FockConvLayer {
  int r, states, first, nc, nc0, row[2];  // row[half]: row of B of this layer's factor
  int halves, half0;                      // number of halves that reach this layer, and the first of them
  int last[2];
};
constexpr int kConvRows = 24, kConvCols = 16;   // monomials of either half per contraction CTA
constexpr int kConvMaxChunk = 1024;       // states per CTA: the sums' range (k_conv_sum)
int fock_conv_slots_per_sm(int nd);           // resident contraction CTAs of an SM
size_t fock_conv_layer_smem(int nin, int L, int nc);
cudaError_t launch_fock_conv(const FockConvArgs& a, const FockConvLayer* layers, int nlayers, int num_sms,
                             cudaStream_t s, int* launches);

}  // namespace gbsbin
