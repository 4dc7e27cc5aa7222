// Host side of heralded states (arXiv:2412.17742, Sec. VII): validation, XA ordered by mode role with its traced
// rows eliminated, the first heralding group's spectral form, the grid's twiddles, Pr(0), device buffers and the
// launches (the first group's roots, the points, the inverse DFT over the heralding grid).
#include <algorithm>
#include <cmath>
#include <complex>
#include <new>
#include <vector>

#include "gbsbin_herald.h"
#include "gbsbin_host_state.h"

using cd = std::complex<double>;
using namespace gbsbin;

struct gbsbin_herald_plan {
  gbsbin_options opt{};
  HeraldArgs args{};
  int n2 = 0;
  long long table_size = 0;              // complex elements of rho
  bool executed = false;
  int last_launches = 0, num_sms = 0;
  TreeArgs tree{};                       // the heralding groups' levels
  double2* d_depth1 = nullptr;           // depth 1: matrices, vectors, path records
  double logq1_re = 0.0;
  size_t upload_bytes = 0;
  // device
  unsigned char* d_const = nullptr;      // tree inputs, tw, chscale, channel and Taylor tables
  double2* d_gcoef = nullptr;
  double2* d_scratch = nullptr;
  double* d_minpiv = nullptr;
  double* d_prob = nullptr;              // the plan's copy of Pr(b)
  double2* d_rho_tmp = nullptr;          // execute_host's device result
  double* d_prob_tmp = nullptr;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

namespace {

template <typename T>
int dalloc(T** p, size_t count) {
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return e == cudaErrorMemoryAllocation ? GBSBIN_ERR_NOMEM : GBSBIN_ERR_CUDA;
  }
  return GBSBIN_OK;
}

void free_all(gbsbin_herald_plan* P) {
  void* ptrs[] = {P->d_const, P->d_gcoef, P->d_scratch, P->d_minpiv, P->d_prob, P->d_rho_tmp, P->d_prob_tmp, P->d_depth1};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  if (P->ev0) cudaEventDestroy(P->ev0);
  if (P->ev1) cudaEventDestroy(P->ev1);
}

// Byte image of the constant inputs, each piece 16-byte aligned.
struct Blob {
  std::vector<unsigned char> bytes;
  size_t put(const void* src, size_t n) {
    const size_t off = (bytes.size() + 15) & ~(size_t)15;
    bytes.resize(off + n);
    if (n) std::copy((const unsigned char*)src, (const unsigned char*)src + n, bytes.begin() + off);
    return off;
  }
};

std::vector<double2> to_d2(const std::vector<cd>& v) {
  std::vector<double2> o(v.size());
  for (size_t q = 0; q < v.size(); ++q) o[q] = make_double2(v[q].real(), v[q].imag());
  return o;
}

}  // namespace

extern "C" {

int gbsbin_herald_plan_create(const gbsbin_herald_problem* p, const gbsbin_options* o, gbsbin_herald_plan** out) {
  if (!out) return GBSBIN_ERR_ARG;
  *out = nullptr;
  if (!p || !p->role || !p->cutoff) return GBSBIN_ERR_ARG;
  const gbsbin_problem* s = &p->state;
  if (s->M <= 0 || s->K <= 0 || (!s->sigma1 && (!s->r || !s->T))) return GBSBIN_ERR_ARG;
  gbsbin_options opt;
  gbsbin_default_options(&opt);
  if (o) opt = *o;
  if (opt.precision != GBSBIN_FP64 || opt.oversample < 1 || opt.want_backward || opt.shard_end != 0 ||
      opt.shard_begin != 0 || (opt.tile_override != 0 && opt.tile_override != GBSBIN_KERNEL_HERALD_FP64))
    return GBSBIN_ERR_ARG;
  const int L = p->L, nm = s->M * s->K, n2 = 2 * nm;
  if (L < 1 || L > GBSBIN_MAX_L || p->fock_cutoff < 0) return GBSBIN_ERR_ARG;
  if (n2 > GBSBIN_HERALD_MAX_MODES2) return GBSBIN_ERR_UNSUPPORTED;
  std::vector<int> cnt(L, 0), Dm, kept;
  for (int m = 0; m < nm; ++m) {
    const int r = p->role[m];
    if (r < GBSBIN_HERALD_KEPT || r >= L) return GBSBIN_ERR_ARG;
    if (r >= 0) cnt[r]++;
    if (r == GBSBIN_HERALD_KEPT) kept.push_back(m);
    else Dm.push_back(m);
  }
  for (int l = 0; l < L; ++l)
    if (cnt[l] == 0) return GBSBIN_ERR_PARTITION;
  const int nk = (int)kept.size();
  if (nk < 1 || nk > GBSBIN_HERALD_MAX_KEPT) return GBSBIN_ERR_UNSUPPORTED;
  const int nf = 2 * nk, cut = p->fock_cutoff;
  long long ncoef = 1;
  for (int i = 0; i < nf; ++i) {
    ncoef *= cut + 1;
    if (ncoef > GBSBIN_HERALD_MAX_COEF) return GBSBIN_ERR_UNSUPPORTED;
  }
  HeraldArgs a{};
  a.L = L;
  a.nf = nf;
  a.cut = cut;
  a.ncoef = ncoef;
  a.npts = 1;
  a.table = 1;
  int rsum = 0;
  for (int l = 0; l < L; ++l) {
    if (p->cutoff[l] < 0) return GBSBIN_ERR_CUTOFF;
    const long long R = (long long)opt.oversample * (p->cutoff[l] + 1LL);
    if (R > (1LL << 26)) return GBSBIN_ERR_CUTOFF;
    a.radix[l] = (int)R;
    a.nout[l] = p->cutoff[l] + 1;
    a.npts *= R;
    a.table *= a.nout[l];
    rsum += (int)R;
    if (a.npts > GBSBIN_MAX_POINTS || rsum > (1 << 26)) return GBSBIN_ERR_CUTOFF;
  }
  // the per-point coefficient tensors and the DFT's scratch (16 bytes an entry) stay within 8 GiB
  if ((double)a.npts * (double)(ncoef + 1) > (double)(1LL << 28)) return GBSBIN_ERR_UNSUPPORTED;
  std::vector<cd> XA, gamma, Xgamma;
  int st = host_state(s, n2, XA, gamma, Xgamma);
  if (st) return st;
  // row order: traced modes, the heralding groups, the kept modes; each set's annihilation rows, then its
  // creation rows.  The traced rows are eliminated here (w = 1): the same augmented form as the tree's levels,
  // [[I - A_TT, A_T., c_T], [-A_.T, A_.., c_.], [-u_T, u_., 0]], whose trailing block is the traced-out state's
  std::vector<int> order;
  TreeArgs t{};
  auto add_role = [&](int role) {
    const size_t before = order.size();
    for (int half = 0; half < 2; ++half)
      for (int m = 0; m < nm; ++m)
        if (p->role[m] == role) order.push_back(m + half * nm);
    return (int)(order.size() - before);
  };
  const int nt = add_role(GBSBIN_HERALD_TRACED), nr = n2 - nt, W = n2 + 1;
  for (int l = 0; l < L; ++l) t.nb[l] = add_role(l);
  add_role(GBSBIN_HERALD_KEPT);
  int rem = nr;
  for (int l = 0; l < L; ++l) {
    t.m[l] = rem;
    rem -= t.nb[l];
  }
  if (L == 1) t.m[1] = nf;
  std::vector<cd> Z((size_t)W * W, cd(0.0));
  for (int i = 0; i < n2; ++i) {
    for (int j = 0; j < n2; ++j) {
      const cd v = XA[(size_t)order[i] * n2 + order[j]];
      Z[(size_t)i * W + j] = j < nt ? (i == j ? 1.0 : 0.0) - v : v;
      if (i < nt && j >= nt) Z[(size_t)i * W + j] = v;
      if (i >= nt && j < nt) Z[(size_t)i * W + j] = -v;
    }
    Z[(size_t)i * W + n2] = Xgamma[order[i]];
    Z[(size_t)n2 * W + i] = i < nt ? -gamma[order[i]] : gamma[order[i]];
  }
  cd tprod = 1.0;
  double targ = 0.0, tmin = 1.0e300;
  int te2 = 0;
  for (int k = 0; k < nt; ++k) {
    const cd piv = Z[(size_t)k * W + k];
    tprod *= piv;
    int ex;
    std::frexp(std::max(std::fabs(tprod.real()), std::fabs(tprod.imag())), &ex);
    tprod = cd(std::ldexp(tprod.real(), -ex), std::ldexp(tprod.imag(), -ex));
    te2 += ex;
    targ += std::atan2(piv.imag(), piv.real());
    tmin = std::min(tmin, piv.real());
    for (int i = k + 1; i < W; ++i) {
      const cd f = Z[(size_t)i * W + k] / piv;
      if (f == cd(0.0)) continue;
      for (int j = k + 1; j < W; ++j) Z[(size_t)i * W + j] -= f * Z[(size_t)k * W + j];
    }
  }
  std::vector<cd> A0((size_t)nr * nr), c0(nr), u0(nr);
  for (int i = 0; i < nr; ++i) {                     // Hermitian up to rounding: made exactly so
    for (int j = 0; j < nr; ++j)
      A0[(size_t)i * nr + j] = 0.5 * (Z[(size_t)(nt + i) * W + nt + j] + std::conj(Z[(size_t)(nt + j) * W + nt + i]));
    c0[i] = Z[(size_t)(nt + i) * W + n2];
    u0[i] = Z[(size_t)n2 * W + nt + i];
  }
  for (int i = 0; i < n2; ++i)
    if (gamma[i] != cd(0.0)) t.has_gamma = 1;
  // the first group's spectral form
  const int nb0 = t.nb[0], rest = nr - nb0;
  std::vector<cd> A00((size_t)nb0 * nb0), rlam(nb0), rB((size_t)nb0 * (rest + 1)), ru(nb0);
  {
    const int X = rest + 2;                          // columns: A_0r, c_0, conj(u_0)
    std::vector<double> xr((size_t)nb0 * X), xi((size_t)nb0 * X), ev;
    for (int i = 0; i < nb0; ++i) {
      for (int j = 0; j < nb0; ++j) A00[(size_t)i * nb0 + j] = A0[(size_t)i * nr + j];
      for (int j = 0; j < X; ++j) {
        const cd v = j < rest ? A0[(size_t)i * nr + nb0 + j] : j == rest ? c0[i] : std::conj(u0[i]);
        xr[(size_t)i * X + j] = v.real();
        xi[(size_t)i * X + j] = v.imag();
      }
    }
    if (!hermitian_spectrum(A00, nb0, ev, xr.data(), xi.data(), X)) return GBSBIN_ERR_NUMERIC;
    a.tmin = tmin;
    a.lam_min = *std::min_element(ev.begin(), ev.end());
    a.lam_max = *std::max_element(ev.begin(), ev.end());
    for (int k = 0; k < nb0; ++k) {
      const double *yr = &xr[(size_t)k * X], *yi = &xi[(size_t)k * X];
      rlam[k] = ev[k];
      for (int j = 0; j <= rest; ++j) rB[(size_t)k * (rest + 1) + j] = cd(yr[j], yi[j]);
      ru[k] = cd(yr[rest + 1], -yi[rest + 1]);
    }
  }
  struct {
    double2 prod;
    float4 meta;
    double2 ex;
  } path0 = {make_double2(tprod.real(), tprod.imag()), make_float4((float)targ, (float)te2, (float)std::min(tmin, 3.0e38), 0.f),
             make_double2(Z[(size_t)n2 * W + n2].real(), Z[(size_t)n2 * W + n2].imag())};
  // the Taylor coefficients in order of total degree, each with its predecessor p - e_i0 (i0
  // its first non-zero digit) and that predecessor's neighbours p - e_i0 - e_j
  const int cp1 = cut + 1, nsh = nf * cut;
  std::vector<std::vector<int>> by_shell((size_t)nsh + 1);
  for (long long q = 1; q < ncoef; ++q) {
    long long r = q;
    int tot = 0;
    for (int i = 0; i < nf; ++i) {
      tot += (int)(r % cp1);
      r /= cp1;
    }
    by_shell[tot].push_back((int)q);
  }
  std::vector<int> shell((size_t)nsh + 2, 0), tq, tqm, ti0, tp, tnb;
  std::vector<long long> stride(nf);
  stride[nf - 1] = 1;
  for (int i = nf - 2; i >= 0; --i) stride[i] = stride[i + 1] * cp1;
  for (int sh = 1; sh <= nsh; ++sh) {
    shell[sh] = (int)tq.size();
    for (int q : by_shell[sh]) {
      int dig[GBSBIN_HERALD_MAX_F];
      for (int i = 0; i < nf; ++i) dig[i] = (int)((q / stride[i]) % cp1);
      int i0 = 0;
      while (dig[i0] == 0) ++i0;
      const long long qm = q - stride[i0];
      tq.push_back(q);
      tqm.push_back((int)qm);
      ti0.push_back(i0);
      tp.push_back(dig[i0]);
      for (int j = 0; j < nf; ++j) {
        const int dj = dig[j] - (j == i0 ? 1 : 0);
        tnb.push_back(dj > 0 ? (int)(qm - stride[j]) : -1);
      }
    }
  }
  shell[nsh + 1] = (int)tq.size();
  const double TWO_PI = 6.283185307179586476925286766559;
  std::vector<double2> tw((size_t)rsum);
  for (int l = 0, off = 0; l < L; off += a.radix[l], ++l)
    for (int d = 0; d < a.radix[l]; ++d) {
      const cd v = std::polar(1.0, -TWO_PI * (double)d / (double)a.radix[l]);
      tw[off + d] = make_double2(v.real(), v.imag());
    }
  // the channels (u, v) with u <= v
  a.side = 1;
  for (int i = 0; i < nk; ++i) a.side *= cp1;
  std::vector<int> chan;
  for (int u = 0; u < a.side; ++u)
    for (int v = u; v < a.side; ++v) chan.push_back(u * a.side + v);
  a.nchan = (int)chan.size() + 1;
  std::vector<double> fs(cut + 1), chs((size_t)ncoef);
  fs[0] = 1.0;
  for (int i = 1; i <= cut; ++i) fs[i] = fs[i - 1] * std::sqrt((double)i);   // sqrt(i!)
  for (long long q = 0; q < ncoef; ++q) {
    long long r = q;
    double v = 1.0;
    for (int i = 0; i < nf; ++i) {
      v *= fs[r % (cut + 1)];
      r /= cut + 1;
    }
    chs[q] = v;
  }
  double mp = 0.0;
  const cd lq1 = host_logq1(XA, gamma, Xgamma, n2, &mp);
  if (!(mp > 0.0) || !std::isfinite(lq1.real())) return GBSBIN_ERR_NONPHYSICAL;
  a.pr0 = std::exp(-lq1.real());

  Blob b;
  const size_t o_tw = b.put(tw.data(), tw.size() * sizeof(double2));
  auto put_d2 = [&b](const std::vector<cd>& v) {
    const std::vector<double2> d = to_d2(v);
    return b.put(d.data(), d.size() * sizeof(double2));
  };
  const size_t o_A0 = put_d2(A0), o_c0 = put_d2(c0), o_u0 = put_d2(u0), o_rlam = put_d2(rlam), o_rB = put_d2(rB),
               o_ru = put_d2(ru), o_path = b.put(&path0, sizeof(path0));
  const size_t o_chan = b.put(chan.data(), chan.size() * sizeof(int));
  const size_t o_chs = b.put(chs.data(), chs.size() * sizeof(double));
  const size_t o_shell = b.put(shell.data(), shell.size() * sizeof(int));
  const size_t o_tq = b.put(tq.data(), tq.size() * sizeof(int));
  const size_t o_tqm = b.put(tqm.data(), tqm.size() * sizeof(int));
  const size_t o_ti0 = b.put(ti0.data(), ti0.size() * sizeof(int));
  const size_t o_tp = b.put(tp.data(), tp.size() * sizeof(int));
  const size_t o_tnb = b.put(tnb.data(), tnb.size() * sizeof(int));

  gbsbin_herald_plan* P = new (std::nothrow) gbsbin_herald_plan();
  if (!P) return GBSBIN_ERR_NOMEM;
  P->opt = opt;
  P->n2 = n2;
  P->table_size = a.table * ncoef;
  P->logq1_re = lq1.real();
  P->upload_bytes = b.bytes.size();
  if ((st = dalloc(&P->d_const, b.bytes.size())) || (st = dalloc(&P->d_gcoef, (size_t)(a.npts * (ncoef + 1)))) ||
      (st = dalloc(&P->d_scratch, (size_t)(a.npts * (ncoef + 1)))) || (st = dalloc(&P->d_minpiv, (size_t)a.npts)) ||
      (st = dalloc(&P->d_prob, (size_t)a.table))) {
    free_all(P);
    delete P;
    return st;
  }
  // depth 1 of the tree, within the same 8 GiB and where there is room for it; without it every point sweeps all groups
  const double depth1 = L > 1 ? (double)a.radix[0] * ((double)t.m[1] * (t.m[1] + 2) + 3) : 0.0;
  const bool kept_roots = L > 1 && 2.0 * (double)a.npts * (double)(ncoef + 1) + depth1 <= (double)(1LL << 29) &&
                          dalloc(&P->d_depth1, (size_t)depth1) == GBSBIN_OK;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess ||
      cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
      cudaMemcpy(P->d_const, b.bytes.data(), b.bytes.size(), cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(P->d_prob, 0, (size_t)a.table * sizeof(double)) != cudaSuccess ||
      (opt.want_timing && (cudaEventCreate(&P->ev0) != cudaSuccess || cudaEventCreate(&P->ev1) != cudaSuccess))) {
    cudaGetLastError();
    free_all(P);
    delete P;
    return GBSBIN_ERR_CUDA;
  }
  unsigned char* c = P->d_const;
  a.tw = reinterpret_cast<const double2*>(c + o_tw);
  a.chan = reinterpret_cast<const int*>(c + o_chan);
  t.A[0] = reinterpret_cast<float4*>(c + o_A0);
  t.c[0] = reinterpret_cast<float4*>(c + o_c0);
  t.u[0] = reinterpret_cast<float4*>(c + o_u0);
  t.path[0] = reinterpret_cast<float4*>(c + o_path);
  t.rlam = reinterpret_cast<const float4*>(c + o_rlam);
  t.rB = reinterpret_cast<const float4*>(c + o_rB);
  t.ru = reinterpret_cast<const float4*>(c + o_ru);
  t.tw = a.tw;
  t.grid.L = L;
  for (int l = 0; l < L; ++l) t.grid.radix[l] = a.radix[l];
  if (kept_roots) {
    float4* q = reinterpret_cast<float4*>(P->d_depth1);
    const size_t R0 = (size_t)a.radix[0], m1 = (size_t)t.m[1];
    t.A[1] = q;
    t.c[1] = t.A[1] + R0 * m1 * m1;
    t.u[1] = t.c[1] + R0 * m1;
    t.path[1] = t.u[1] + R0 * m1;
  }
  P->tree = t;
  a.chscale = reinterpret_cast<const double*>(c + o_chs);
  a.shell = reinterpret_cast<const int*>(c + o_shell);
  a.tq = reinterpret_cast<const int*>(c + o_tq);
  a.tqm = reinterpret_cast<const int*>(c + o_tqm);
  a.ti0 = reinterpret_cast<const int*>(c + o_ti0);
  a.tp = reinterpret_cast<const int*>(c + o_tp);
  a.tnb = reinterpret_cast<const int*>(c + o_tnb);
  a.gcoef = P->d_gcoef;
  a.scratch = P->d_scratch;
  a.minpiv = P->d_minpiv;
  a.prob_own = P->d_prob;
  P->args = a;
  *out = P;
  return GBSBIN_OK;
}

long long gbsbin_herald_table_size(const gbsbin_herald_plan* P) { return P ? P->table_size : -1; }

long long gbsbin_herald_prob_size(const gbsbin_herald_plan* P) { return P ? P->args.table : -1; }

int gbsbin_herald_execute(gbsbin_herald_plan* P, gbsbin_complex* rho_out, double* prob_out, void* stream) {
  if (!P || !rho_out || !prob_out) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (P->ev0 && cudaEventRecord(P->ev0, s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  if (launch_herald(P->args, P->tree, P->num_sms, reinterpret_cast<double2*>(rho_out), prob_out, s, &P->last_launches) != cudaSuccess) {
    cudaGetLastError();
    return GBSBIN_ERR_CUDA;
  }
  P->executed = true;
  if (P->ev1 && cudaEventRecord(P->ev1, s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  return GBSBIN_OK;
}

int gbsbin_herald_execute_host(gbsbin_herald_plan* P, gbsbin_complex* rho_host, double* prob_host, void* stream) {
  if (!P || !rho_host || !prob_host) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int st = GBSBIN_OK;
  if (!P->d_rho_tmp && ((st = dalloc(&P->d_rho_tmp, (size_t)P->table_size)) ||
                        (st = dalloc(&P->d_prob_tmp, (size_t)P->args.table))))
    return st;
  st = gbsbin_herald_execute(P, reinterpret_cast<gbsbin_complex*>(P->d_rho_tmp), P->d_prob_tmp, stream);
  if (!st && (cudaMemcpyAsync(rho_host, P->d_rho_tmp, (size_t)P->table_size * sizeof(double2),
                              cudaMemcpyDeviceToHost, s) != cudaSuccess ||
              cudaMemcpyAsync(prob_host, P->d_prob_tmp, (size_t)P->args.table * sizeof(double),
                              cudaMemcpyDeviceToHost, s) != cudaSuccess))
    st = GBSBIN_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess && !st) st = GBSBIN_ERR_CUDA;
  return st;
}

int gbsbin_herald_diagnostics(gbsbin_herald_plan* P, gbsbin_diag* out, void* stream) {
  if (!P || !out) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const HeraldArgs& a = P->args;
  std::vector<double> mp((size_t)a.npts, 1.0), pr((size_t)a.table, 0.0);
  if (P->executed &&
      (cudaMemcpyAsync(mp.data(), P->d_minpiv, mp.size() * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
       cudaMemcpyAsync(pr.data(), P->d_prob, pr.size() * sizeof(double), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
       cudaStreamSynchronize(s) != cudaSuccess)) {
    cudaGetLastError();
    return GBSBIN_ERR_CUDA;
  }
  double sum = 0.0, mn = 1e300;
  long long bad = 0;
  for (double v : pr) sum += v;
  for (double v : mp) {
    if (!(v > 0.0)) ++bad;
    mn = std::fmin(mn, v);
  }
  *out = gbsbin_diag{};
  out->sum_P = sum;
  out->max_imag = 0.0;
  out->min_pivot_re = P->executed ? mn : 1.0;
  out->n_bad_points = bad;
  out->n_points = a.npts;
  out->n_evaluated = a.npts;
  out->table_size = P->table_size;
  out->n = P->n2;
  out->kernel = GBSBIN_KERNEL_HERALD_FP64;
  out->log_q1_re = P->logq1_re;
  out->point_kernel_ms = 0.0;
  out->state_upload_bytes = (long long)P->upload_bytes;
  out->launches = P->last_launches;
  if (P->ev1 && P->executed) {
    float ms = 0.f;
    if (cudaEventSynchronize(P->ev1) != cudaSuccess || cudaEventElapsedTime(&ms, P->ev0, P->ev1) != cudaSuccess) {
      cudaGetLastError();
      return GBSBIN_ERR_CUDA;
    }
    out->point_kernel_ms = ms;
  }
  if (bad > 0 || !std::isfinite(sum)) return GBSBIN_ERR_NUMERIC;
  return GBSBIN_OK;
}

int gbsbin_herald_plan_destroy(gbsbin_herald_plan* P) {
  if (!P) return GBSBIN_OK;
  cudaDeviceSynchronize();
  free_all(P);
  delete P;
  return GBSBIN_OK;
}

}  // extern "C"
