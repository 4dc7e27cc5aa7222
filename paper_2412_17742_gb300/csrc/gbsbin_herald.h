// Heralded states (gbsbin_herald.cu, gbsbin_herald_host.cpp).  Not part of the public ABI.
#pragma once

#include "gbsbin_internal.h"

namespace gbsbin {

// The traced modes are eliminated on the host (w = 1 at every point); the rest are ordered by heralding group,
// the kept modes (nf rows, both halves) last, and the groups run as the levels of a tree of block eliminations
// (TreeArgs, gbsbin_tree.cuh; A[1] = nullptr: without depth 1 in memory, each point from the first group).  The Taylor coefficients are visited in order of total degree from a table
// built with the plan: entry t of shell s (s = 1 .. nf cut, entries shell[s] .. shell[s + 1] - 1) is
// coefficient q = tq[t], computed from p - e_i0 (index tqm[t], i0 = ti0[t] the first non-zero digit,
// p_i0 = tp[t]) and its neighbours p - e_i0 - e_j (tnb[t nf + j], -1 where that digit is zero).  A channel is
// a pair (u, v); rho is Hermitian, so the inverse DFT runs over those with u <= v (chan[]) and the heralding
// probability's value.
#define GBSBIN_HERALD_MAX_F (2 * GBSBIN_HERALD_MAX_KEPT)
struct HeraldArgs {
  int L, nf, cut;
  int radix[GBSBIN_MAX_L];           // oversample (cutoff + 1) per heralding group
  int nout[GBSBIN_MAX_L];            // cutoff + 1
  long long npts;                    // prod radix
  long long ncoef;                   // (cut + 1)^nf
  int side;                          // (cut + 1)^(nf / 2): channel = u side + v
  int nchan;                         // channels with u <= v, then one for the heralding probability
  long long table;                   // prod nout
  double pr0;                        // Pr(0) of the whole state
  double tmin;                       // the traced rows' smallest pivot (1e300: none)
  double lam_min, lam_max;           // the ends of the first group's spectrum
  const double2* tw;                 // exp(-2 pi i d / radix[l]), d < radix[l], group after group
  const double* chscale;             // [ncoef] prod_i sqrt(p_i!)
  const int* chan;                   // [nchan - 1] the channels with u <= v
  const int* shell;                  // [nf cut + 2] first table entry of each shell
  const int* tq;                     // [ncoef - 1] coefficient of each entry
  const int* tqm;
  const int* ti0;
  const int* tp;
  const int* tnb;                    // [(ncoef - 1) nf]
  double2* gcoef;                    // npts x (ncoef + 1): Taylor coefficients at each point, then
                                     // the heralding probability's generating function
  double2* scratch;                  // npts x (ncoef + 1): the inverse DFT's other buffer
  double* minpiv;                    // npts: smallest pivot real part of both eliminations
  double* prob_own;                  // table: the plan's copy of Pr(b) (diagnostics)
};
size_t herald_sweep_smem(int L, int nb0, int m1, bool deep);   // shared memory of a point's elimination
cudaError_t launch_herald(const HeraldArgs& a, const TreeArgs& t, int num_sms, double2* out, double* prob,
                          cudaStream_t s, int* launches);

}  // namespace gbsbin
