// Host side of the Fock-input path (arXiv:2412.17742, App. C): validation, the FP64
// coefficient matrices I - T^dag T and T_l^dag T_l restricted to the occupied inputs, the
// node and output-group roots, device workspaces and the launches: the convolution over
// sub-multisets of the photons (gbsbin_fock_conv.cu) where it costs less, else nodes x points
// and the inverse DFT of the output groups.
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <new>
#include <vector>

#include "gbsbin_fock_conv.h"
#include "gbsbin_internal.h"

using cd = std::complex<double>;
using namespace gbsbin;

struct gbsbin_fock_plan {
  int M = 0, L = 0;
  gbsbin_options opt{};
  std::vector<int> photons, bin_of_mode, cutoff;
  std::vector<int> pos_input;            // input port of each position (position 0: held)
  bool df = false;
  int zt = 1;                            // output-group points per thread
  int kernel = 0;
  int num_sms = 0;
  long long table_size = 0;
  FockArgs args{};
  size_t coef_count = 0;                 // (L + 1) nin^2
  bool executed = false;                 // an execute has been enqueued
  // device
  unsigned char* d_state = nullptr;      // coef (double2) then coef_df (float4)
  double2* d_xtw = nullptr;
  float4* d_xtw_df = nullptr;
  double2* d_zr = nullptr;
  float4* d_zr_df = nullptr;
  double2* d_tw = nullptr;               // inverse-DFT twiddles exp(-2 pi i m / R)
  double2* d_parts = nullptr;
  double2* d_bufA = nullptr;
  double2* d_bufB = nullptr;
  double* d_diag = nullptr;
  unsigned* d_bar = nullptr;
  double* d_table = nullptr;
  unsigned char* h_stage = nullptr;      // pinned copy of the state block
  size_t state_bytes = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  // the convolution (whole plans where it costs less than the node walk)
  bool conv = false;
  FockConvArgs cv{};
  std::vector<FockConvLayer> layers;
  unsigned char* d_conv = nullptr;       // its tables, states and partial sums
  int last_launches = 0;
};

namespace {

float4 split_df(cd v) {
  const float hr = (float)v.real(), hi = (float)v.imag();
  return make_float4(hr, hi, (float)(v.real() - (double)hr), (float)(v.imag() - (double)hi));
}

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

void free_all(gbsbin_fock_plan* P) {
  if (P->d_conv) {                       // one block holds everything
    P->d_state = nullptr;
    P->d_diag = nullptr;
    P->d_table = nullptr;
  }
  void* ptrs[] = {P->d_state, P->d_xtw, P->d_xtw_df, P->d_zr, P->d_zr_df, P->d_tw, P->d_parts,
                  P->d_bufA, P->d_bufB, P->d_diag, P->d_bar, P->d_table, P->d_conv};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  if (P->h_stage) cudaFreeHost(P->h_stage);
  if (P->ev0) cudaEventDestroy(P->ev0);
  if (P->ev1) cudaEventDestroy(P->ev1);
}

// ||T||_2 <= 1: (1 + 1e-10) I - T^dag T must admit a Cholesky factor.
bool contraction(const std::vector<cd>& T, int M) {
  std::vector<cd> A((size_t)M * M);
  for (int j = 0; j < M; ++j)
    for (int k = 0; k < M; ++k) {
      cd s = 0.0;
      for (int i = 0; i < M; ++i) s += std::conj(T[(size_t)i * M + j]) * T[(size_t)i * M + k];
      A[(size_t)j * M + k] = (j == k ? 1.0 + 1e-10 : 0.0) - s;
    }
  for (int j = 0; j < M; ++j) {
    double d = A[(size_t)j * M + j].real();
    for (int k = 0; k < j; ++k) d -= std::norm(A[(size_t)j * M + k]);
    if (!(d > 0.0)) return false;
    d = std::sqrt(d);
    A[(size_t)j * M + j] = d;
    for (int i = j + 1; i < M; ++i) {
      cd s = A[(size_t)i * M + j];
      for (int k = 0; k < j; ++k) s -= A[(size_t)i * M + k] * std::conj(A[(size_t)j * M + k]);
      A[(size_t)i * M + j] = s / d;
    }
  }
  return true;
}

// Coefficient matrices into the pinned staging block: m = 0: I - T^dag T, m = 1 + l:
// T_l^dag T_l, over the occupied inputs in position order, stored [m][k][j]; then the same
// as FP32 pairs.
int stage_transfer(gbsbin_fock_plan* P, const gbsbin_complex* Tin) {
  const int M = P->M, L = P->L, nin = P->args.nin;
  std::vector<cd> T((size_t)M * M);
  for (size_t q = 0; q < T.size(); ++q) {
    T[q] = cd(Tin[q].re, Tin[q].im);
    if (!std::isfinite(Tin[q].re) || !std::isfinite(Tin[q].im)) return GBSBIN_ERR_ARG;
  }
  if (!contraction(T, M)) return GBSBIN_ERR_NONPHYSICAL;
  double2* coef = reinterpret_cast<double2*>(P->h_stage);
  float4* coef_df = reinterpret_cast<float4*>(P->h_stage + P->coef_count * sizeof(double2));
  for (int m = 0; m <= L; ++m)
    for (int k = 0; k < nin; ++k)
      for (int j = 0; j < nin; ++j) {
        const int jj = P->pos_input[j], kk = P->pos_input[k];
        cd s = 0.0;
        for (int i = 0; i < M; ++i)
          if (m == 0 || P->bin_of_mode[i] == m - 1) s += std::conj(T[(size_t)i * M + jj]) * T[(size_t)i * M + kk];
        if (m == 0) s = (j == k ? 1.0 : 0.0) - s;
        const size_t q = ((size_t)m * nin + k) * nin + j;
        coef[q] = make_double2(s.real(), s.imag());
        coef_df[q] = split_df(s);
      }
  if (P->conv) {   // the same by rows in fixed point, each row scaled by a power of two
    longlong2* B = reinterpret_cast<longlong2*>(P->h_stage + P->coef_count * (sizeof(double2) + sizeof(float4)));
    int exponent = 0;
    for (int j = 0; j < nin; ++j) {
      auto at = [&](int k, int m) { return coef[((size_t)m * nin + k) * nin + j]; };
      double big = 0.0, all = 0.0;
      for (int k = 0; k < nin; ++k)
        for (int m = 0; m <= L; ++m) {
          big = std::fmax(big, std::fmax(std::fabs(at(k, m).x), std::fabs(at(k, m).y)));
          all += std::fabs(at(k, m).x) + std::fabs(at(k, m).y);
        }
      const int e = conv_row_exponent(big, all);
      for (int k = 0; k < nin; ++k)
        for (int m = 0; m <= L; ++m)
          B[((size_t)j * nin + k) * (L + 1) + m] = make_longlong2(conv_fixed(at(k, m).x, e), conv_fixed(at(k, m).y, e));
      exponent += e * P->args.pw[j];
    }
    std::memcpy(B + P->coef_count, &exponent, sizeof(exponent));
  }
  return GBSBIN_OK;
}

// Whether the convolution serves the plan, with its layers and sizes: its estimated time (60 clocks
// of a scheduler per warp's multiply-add, as measured, and ~3 us per launch) against the node walk's at its measured rates (1.25e13 FP32 operations a second, 63 per
// factor, in pairs of FP32; 4.5e11 FP64 operations, 10 per factor).  Bounded: 2^22 states in all, 2^20 monomial
// pairs and 2^22 table entries, 1 GB of states, 48 KB of shared memory per layer CTA.
bool conv_layout(gbsbin_fock_plan* P) {
  const FockArgs& a = P->args;
  FockConvArgs& c = P->cv;
  int N = 0;
  double codes = 1.0;
  for (int j = 0; j < a.nin; ++j) {
    codes *= a.pw[j] + 1.0;
    if (codes > (double)(1 << 22)) return false;
    N += a.pw[j];
  }
  if (N < 4 || P->table_size > (1 << 22)) return false;
  // The walk of few nodes is shorter than the convolution's launches (N / 2 layers and three more, ~6 us each): one or
  // two occupied inputs (2 + 2 photons, one group, pairs 20 us against 29, 6 + 6 32 against 49, three groups FP64 10 + 10 123
  // against 127), three of up to five photons in one group (27 to 36 us against 29 to 37).
  if (a.nin <= 2 || (a.nin == 3 && N <= 5 && a.L == 1)) return false;
  c.nin = a.nin;
  c.L = a.L;
  c.N = N;
  c.h[0] = N / 2;
  c.h[1] = N - N / 2;
  std::vector<double> mono(c.h[1] + 1, 1.0);            // monomials of degree <= r in L variables
  for (int r = 1; r <= c.h[1]; ++r) {
    mono[r] = mono[r - 1] * (r + a.L) / r;
    if (mono[r] > 4096.0) return false;
  }
  if (std::min(c.h[1], a.nin) * (a.L + 1) > kConvMaxTerms) return false;
  c.n1 = (int)std::lround(mono[c.h[0]]);
  c.n2 = (int)std::lround(mono[c.h[1]]);
  if ((double)c.n1 * c.n2 > (double)(1 << 20) || fock_conv_layer_smem(a.nin, a.L, c.n2) > 48 * 1024) return false;
  // states per layer: coefficients of prod (1 + x + .. + x^p_j)
  std::vector<double> cnt(1, 1.0);
  for (int j = 0; j < a.nin; ++j) {
    std::vector<double> nx(cnt.size() + a.pw[j], 0.0);
    for (size_t u = 0; u < cnt.size(); ++u)
      for (int v = 0; v <= a.pw[j]; ++v) nx[u + v] += cnt[u];
    cnt.swap(nx);
  }
  // two digits leave out lo x lo, up to 2^-57 a product: of many states' small entries that adds up (pairs, 2 to 5%
  // transmission, 16 photons in two groups 9e-15 of the table, the walk 3e-15)
  c.nd = P->df && cnt[c.h[0]] < (double)(1 << 14) ? 2 : 3;
  std::vector<int> row;
  for (int j = 0; j < a.nin; ++j)
    for (int v = 0; v < a.pw[j]; ++v) row.push_back(j);
  P->layers.clear();
  double clocks = 0.0, bytes = 0.0;
  int first = 1;
  for (int r = 1; r <= c.h[1]; ++r) {
    FockConvLayer y{};
    y.r = r;
    y.states = (int)cnt[r];
    y.first = first;
    first += y.states;
    y.nc = (int)std::lround(mono[r]);
    y.nc0 = (int)std::lround(mono[r - 1]);
    y.halves = r <= c.h[0] ? 2 : 1;
    y.half0 = y.halves == 2 ? 0 : 1;
    for (int h = 0; h < 2; ++h) {
      if (h == 0 && r > c.h[0]) continue;
      y.row[h] = row[(h ? c.h[0] : 0) + r - 1];
      y.last[h] = r == c.h[h];
    }
    clocks += y.halves * (double)y.states * std::min(r, a.nin) * ((y.nc + 31) / 32) * (a.L + 1);
    bytes = std::fmax(bytes, 16.0 * y.states * (y.nc + 1.0));
    P->layers.push_back(y);
  }
  c.states = (int)cnt[c.h[0]];
  c.first = P->layers[c.h[0] - 1].first;
  clocks += (c.nd - 1) * (double)c.states * ((c.n1 + 23) / 24 * 24.0) * ((c.n2 + 15) / 16 * 16.0) / 32.0;
  if (4.0 * bytes > (double)(1 << 30)) return false;
  const double t_conv = 60.0 * clocks / (4.0 * P->num_sms * 1.9e9) + 3e-6 * (P->layers.size() + 3);
  const double pairs = (double)(a.x_hi - a.x_lo) * a.grid.n_full * N;
  const double t_walk = (P->df ? pairs * 63.0 / 1.25e13 : pairs * 10.0 / 4.5e11) + 25e-6;
  return t_conv < t_walk;
}

// Tables and workspaces of the convolution and the plan's state, diagnostics and table in one device block (a block of
// its own for each small array is one of 2 MB more to allocate and give back, ~65 us).
int conv_setup(gbsbin_fock_plan* P) {
  FockConvArgs& c = P->cv;
  const FockArgs& a = P->args;
  const int L = c.L, nin = c.nin, hi = c.h[1];
  int codes = 1;
  for (int j = 0; j < nin; ++j) {
    c.stride[j] = codes;
    c.radix[j] = a.pw[j] + 1;
    codes *= c.radix[j];
  }
  c.full = codes - 1;
  // codes by layer: the sum of digits, digit after digit over all lower codes, then a counting sort
  std::vector<int> rank(codes, 0), order(P->layers.back().first + P->layers.back().states);
  {
    std::vector<int> sum(codes, 0), next(hi + 1, 0);
    for (int j = 0; j < nin; ++j)
      for (int v = 1; v < c.radix[j]; ++v)
        for (int q = 0; q < c.stride[j]; ++q) sum[(size_t)v * c.stride[j] + q] = sum[q] + v;
    for (int r = 1; r <= hi; ++r) next[r] = P->layers[r - 1].first;
    const std::vector<int> begin(next);
    for (int q = 0; q < codes; ++q) {
      const int r = sum[q];
      if (r > hi) continue;
      rank[q] = next[r] - begin[r];
      order[next[r]++] = q;
    }
  }
  // monomials by degree (a layer's are a prefix), L exponents each, and each without one of its variables
  std::vector<int> mono((size_t)c.n2 * L);
  int nm = 0;
  for (int d = 0; d <= hi; ++d) {
    std::vector<int> e(L, 0);
    e[L - 1] = d;
    for (;; ++nm) {                             // compositions of d, the last variable running down
      if (nm == c.n2) return GBSBIN_ERR_UNSUPPORTED;
      std::copy(e.begin(), e.end(), mono.begin() + (size_t)nm * L);
      int l = L - 1;
      while (l > 0 && e[l] == 0) --l;
      if (l == 0) break;
      const int v = e[l];
      e[l] = 0;
      e[l - 1] += 1;
      e[L - 1] = v - 1;
    }
    ++nm;
  }
  if (nm != c.n2) return GBSBIN_ERR_UNSUPPORTED;
  c.ndown = c.n2;
  std::vector<int> down((size_t)(L + 1) * c.n2, -1);
  {
    std::vector<long long> unit(L, 1);          // a monomial's key: its exponents as digits of base hi + 1
    for (int l = L - 2; l >= 0; --l) unit[l] = unit[l + 1] * (hi + 1);
    std::vector<std::pair<long long, int>> idx(c.n2);
    for (int e = 0; e < c.n2; ++e) {
      long long key = 0;
      for (int l = 0; l < L; ++l) key += unit[l] * mono[(size_t)e * L + l];
      idx[e] = std::make_pair(key, e);
    }
    std::sort(idx.begin(), idx.end());
    for (const std::pair<long long, int>& k : idx) {
      down[k.second] = k.second;
      for (int l = 0; l < L; ++l)
        if (mono[(size_t)k.second * L + l] > 0)
          down[(size_t)(l + 1) * c.n2 + k.second] =
              std::lower_bound(idx.begin(), idx.end(), std::make_pair(k.first - unit[l], -1))->second;
    }
  }
  // the pairs (a, b) of each table entry: exponents add, folded modulo the radices
  const GridDesc& g = a.grid;
  c.table_size = P->table_size;
  std::vector<int> to((size_t)c.n1 * c.n2), first(P->table_size + 1, 0), list;
  {
    std::vector<long long> part((size_t)L * (c.N + 1));   // an exponent's share of the entry, below any sum if cut off
    long long stride = 1;
    for (int l = L - 1; l >= 0; --l) {
      for (int b = 0; b <= c.N; ++b)
        part[(size_t)l * (c.N + 1) + b] = b % g.radix[l] < g.nout[l] ? stride * (b % g.radix[l]) : -(1LL << 40);
      stride *= g.nout[l];
    }
    for (int x = 0; x < c.n1; ++x)
      for (int y = 0; y < c.n2; ++y) {
        const int *ex = &mono[(size_t)x * L], *ey = &mono[(size_t)y * L];
        long long t = 0;
        for (int l = 0; l < L; ++l) t += part[(size_t)l * (c.N + 1) + ex[l] + ey[l]];
        to[(size_t)x * c.n2 + y] = t >= 0 ? (int)t : -1;
        if (t >= 0) ++first[t + 1];
      }
  }
  for (long long t = 0; t < P->table_size; ++t) first[t + 1] += first[t];
  list.resize(std::max(1, first[P->table_size]));
  {
    std::vector<int> next(first);
    for (size_t q = 0; q < to.size(); ++q)
      if (to[q] >= 0) list[next[to[q]]++] = (int)q;
  }
  // chunks of states: one wave of resident CTAs, at most kConvMaxChunk states each
  const long long tiles = (long long)((c.n1 + kConvRows - 1) / kConvRows) * ((c.n2 + kConvCols - 1) / kConvCols);
  const long long slots = (long long)std::max(1, fock_conv_slots_per_sm(c.nd)) * P->num_sms;
  long long nch = std::max<long long>(1, slots / tiles);
  nch = std::min<long long>(nch, (c.states + 31) / 32);
  c.chunk = (int)std::min<long long>((c.states + nch - 1) / nch, kConvMaxChunk);
  c.nchunks = (c.states + c.chunk - 1) / c.chunk;
  // one block: offsets in 16-byte units
  size_t at = 0;
  auto take = [&at](size_t bytes) {
    const size_t o = at;
    at += (bytes + 15) / 16 * 16;
    return o;
  };
  size_t fmax[2] = {0, 0}, emax = 0;
  for (const FockConvLayer& y : P->layers) {
    for (int h = y.half0; h < 2; ++h) fmax[h] = std::max(fmax[h], (size_t)y.states * (y.nc + 1));
    emax = std::max(emax, (size_t)y.states);
  }
  const size_t o_rank = take(rank.size() * 4), o_order = take(order.size() * 4), o_down = take(down.size() * 4),
               o_first = take(first.size() * 4), o_list = take(list.size() * 4), o_f0 = take(32), o_e0 = take(4),
               o_c0 = take(((size_t)c.n1 + c.n2) * 4);
  size_t o_F[2][2], o_E[2][2];
  for (int h = 0; h < 2; ++h)
    for (int p = 0; p < 2; ++p) {
      o_F[h][p] = take(fmax[h] * 16);
      o_E[h][p] = take(emax * 4);
    }
  size_t o_F3[2] = {0, 0};
  for (int h = 0; h < 2 && c.nd == 3; ++h) o_F3[h] = take((size_t)c.states * ((h ? c.n2 : c.n1) + 1) * 8);
  const size_t o_parts = take((size_t)c.nchunks * c.n1 * c.n2 * 16), o_state = take(P->state_bytes),
               o_diag = take(GBSBIN_DIAG_DOUBLES * sizeof(double)), o_table = take((size_t)P->table_size * sizeof(double));
  const int st = dalloc(&P->d_conv, at);
  if (st) return st;
  unsigned char* d = P->d_conv;
  const int f0[8] = {1 << (kConvDigit - 1), 0, 0, 0, 0, 0, 0, 0}, e0 = 1;   // 1 = 2^55 2^-56 2^1, then the row's zero entry
  std::vector<unsigned char> tables(o_c0);               // the tables come first: one copy
  auto put = [&tables](size_t o, const void* src, size_t bytes) { std::memcpy(tables.data() + o, src, bytes); };
  put(o_rank, rank.data(), rank.size() * 4);
  put(o_order, order.data(), order.size() * 4);
  put(o_down, down.data(), down.size() * 4);
  put(o_first, first.data(), first.size() * 4);
  put(o_list, list.data(), list.size() * 4);
  put(o_f0, f0, 32);
  put(o_e0, &e0, 4);
  if (cudaMemcpy(d, tables.data(), tables.size(), cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    return GBSBIN_ERR_CUDA;
  }
  c.rank = (const int*)(d + o_rank);
  c.order = (const int*)(d + o_order);
  c.down = (const int*)(d + o_down);
  c.pair_first = (const int*)(d + o_first);
  c.pair_list = (const int*)(d + o_list);
  c.F0 = (const int4*)(d + o_f0);
  c.E0 = (const int*)(d + o_e0);
  c.colexp[0] = (int*)(d + o_c0);
  c.colexp[1] = c.colexp[0] + c.n1;
  for (int h = 0; h < 2; ++h)
    for (int p = 0; p < 2; ++p) {
      c.F[h][p] = (int4*)(d + o_F[h][p]);
      c.E[h][p] = (int*)(d + o_E[h][p]);
    }
  for (int h = 0; h < 2; ++h) c.F3[h] = c.nd == 3 ? (int2*)(d + o_F3[h]) : nullptr;
  c.parts = (double2*)(d + o_parts);
  P->d_state = d + o_state;
  P->d_diag = (double*)(d + o_diag);
  P->d_table = (double*)(d + o_table);
  c.B = (const longlong2*)(P->d_state + P->coef_count * (sizeof(double2) + sizeof(float4)));
  c.exponent = (const int*)(c.B + P->coef_count);
  return GBSBIN_OK;
}

}  // namespace

extern "C" {

int gbsbin_fock_plan_create(const gbsbin_fock_problem* p, const gbsbin_options* o, gbsbin_fock_plan** out) {
  if (!out) return GBSBIN_ERR_ARG;
  *out = nullptr;
  if (!p || p->M <= 0 || !p->T || !p->photons || !p->bin_of_mode || !p->cutoff) return GBSBIN_ERR_ARG;
  gbsbin_options opt;
  gbsbin_default_options(&opt);
  if (o) opt = *o;
  if (opt.oversample < 1 || (opt.precision != GBSBIN_FP64 && opt.precision != GBSBIN_FP32_REFINE))
    return GBSBIN_ERR_ARG;
  if (opt.tile_override != 0 && opt.tile_override != GBSBIN_KERNEL_FOCK_FP64 &&
      opt.tile_override != GBSBIN_KERNEL_FOCK_DF32)
    return GBSBIN_ERR_ARG;
  if (opt.want_backward) return GBSBIN_ERR_UNSUPPORTED;
  const int M = p->M, L = p->L;
  if (L < 1 || L > M) return GBSBIN_ERR_ARG;
  if (L > GBSBIN_FOCK_MAX_GROUPS) return GBSBIN_ERR_UNSUPPORTED;
  std::vector<int> seen(L, 0);
  for (int i = 0; i < M; ++i) {
    if (p->bin_of_mode[i] < 0 || p->bin_of_mode[i] >= L) return GBSBIN_ERR_PARTITION;
    seen[p->bin_of_mode[i]] = 1;
  }
  for (int l = 0; l < L; ++l)
    if (!seen[l]) return GBSBIN_ERR_PARTITION;
  long long npts = 1;
  for (int l = 0; l < L; ++l) {
    if (p->cutoff[l] < 0) return GBSBIN_ERR_CUTOFF;
    npts *= (long long)opt.oversample * (p->cutoff[l] + 1);
    if (npts > GBSBIN_MAX_POINTS) return GBSBIN_ERR_CUTOFF;
  }
  // occupied inputs; position 0 holds the one with the fewest photons (lowest port on ties)
  std::vector<int> occ;
  for (int j = 0; j < M; ++j) {
    if (p->photons[j] < 0) return GBSBIN_ERR_ARG;
    if (p->photons[j] > GBSBIN_FOCK_MAX_PER_INPUT) return GBSBIN_ERR_UNSUPPORTED;
    if (p->photons[j] > 0) occ.push_back(j);
  }
  if ((int)occ.size() > GBSBIN_FOCK_MAX_INPUTS) return GBSBIN_ERR_UNSUPPORTED;
  {
    std::vector<cd> T((size_t)M * M);
    for (size_t q = 0; q < T.size(); ++q) {
      if (!std::isfinite(p->T[q].re) || !std::isfinite(p->T[q].im)) return GBSBIN_ERR_ARG;
      T[q] = cd(p->T[q].re, p->T[q].im);
    }
    if (!contraction(T, M)) return GBSBIN_ERR_NONPHYSICAL;
  }
  gbsbin_fock_plan* P = new (std::nothrow) gbsbin_fock_plan();
  if (!P) return GBSBIN_ERR_NOMEM;
  P->M = M;
  P->L = L;
  P->opt = opt;
  P->photons.assign(p->photons, p->photons + M);
  P->bin_of_mode.assign(p->bin_of_mode, p->bin_of_mode + M);
  P->cutoff.assign(p->cutoff, p->cutoff + L);
  if (!occ.empty()) {
    int h = 0;
    for (int t = 1; t < (int)occ.size(); ++t)
      if (p->photons[occ[t]] < p->photons[occ[h]]) h = t;
    P->pos_input.push_back(occ[h]);
    for (int t = 0; t < (int)occ.size(); ++t)
      if (t != h) P->pos_input.push_back(occ[t]);
  }
  FockArgs& a = P->args;
  a.nin = (int)P->pos_input.size();
  a.L = L;
  a.nd = a.nin > 0 ? a.nin - 1 : 0;
  for (int j = 0; j < a.nin; ++j) a.pw[j] = p->photons[P->pos_input[j]];
  a.dstride[0] = 1;
  int xoff = 0;
  for (int d = 0; d < a.nd; ++d) {
    a.drad[d] = a.pw[d + 1] + 1;
    a.doff[d] = xoff;
    xoff += a.drad[d];
    if ((double)a.dstride[d] * a.drad[d] > (double)GBSBIN_FOCK_MAX_NODES) {
      delete P;
      return GBSBIN_ERR_UNSUPPORTED;
    }
    a.dstride[d + 1] = a.dstride[d] * a.drad[d];
  }
  a.S = a.dstride[a.nd];
  // a shard walks the nodes [shard_begin, shard_end) only; its table is the partial sum of
  // their terms (normalised by the whole node count), so the shards' tables add up
  a.x_lo = 0;
  a.x_hi = a.S;
  if (opt.shard_end != 0 || opt.shard_begin != 0) {
    if (opt.shard_begin < 0 || opt.shard_end <= opt.shard_begin || opt.shard_end > a.S) {
      delete P;
      return GBSBIN_ERR_ARG;
    }
    a.x_lo = opt.shard_begin;
    a.x_hi = opt.shard_end;
  }
  const long long nodes = a.x_hi - a.x_lo;
  // output-group grid, as for Gaussian states
  GridDesc& g = a.grid;
  g.L = L;
  g.npts = 1;
  P->table_size = 1;
  a.roff[0] = 0;
  for (int l = 0; l < L; ++l) {
    g.radix[l] = opt.oversample * (p->cutoff[l] + 1);
    g.nout[l] = p->cutoff[l] + 1;
    g.npts *= g.radix[l];
    P->table_size *= g.nout[l];
    a.roff[l + 1] = a.roff[l] + g.radix[l];
  }
  a.rsum = a.roff[L];
  g.half = g.radix[L - 1] / 2 + 1;
  g.n_full = g.npts / g.radix[L - 1] * g.half;
  g.e_lo = 0;
  g.e_hi = g.n_full;
  g.n_eval = g.n_full;
  P->kernel = opt.tile_override ? opt.tile_override
                                : (opt.precision == GBSBIN_FP32_REFINE ? GBSBIN_KERNEL_FOCK_DF32 : GBSBIN_KERNEL_FOCK_FP64);
  P->df = P->kernel == GBSBIN_KERNEL_FOCK_DF32;
  // restarts bound the drift of the incrementally updated state (FP32 pairs drift faster)
  const long long chunk_max = P->df ? 256 : 1024;
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess ||
      cudaDeviceGetAttribute(&P->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
    cudaGetLastError();
    delete P;
    return GBSBIN_ERR_CUDA;
  }
  const size_t smem = fock_smem_bytes(a.nin, L, a.rsum);
  P->zt = fock_points_per_thread(P->df, g.n_full);
  const int per_sm = smem <= 200 * 1024 ? fock_ctas_per_sm(P->df, P->zt, smem) : 0;
  if (per_sm < 1) {
    delete P;
    return GBSBIN_ERR_UNSUPPORTED;
  }
  const long long per_cta = (long long)GBSBIN_FOCK_THREADS * P->zt;
  const long long tiles = (g.n_full + per_cta - 1) / per_cta;
  // node ranges: two whole waves of resident CTAs where the nodes allow (a partial last wave
  // idles SMs), each range at least 32 nodes; ranges longer than chunk_max are walked as
  // several restarts dealt cyclically
  const long long slots = (long long)per_sm * P->num_sms;
  long long xr = 2 * slots / tiles;
  const long long cap = (512LL << 20) / (16 * g.n_full);            // parts <= 512 MB
  if (xr > cap) xr = cap;
  if (xr > 65535) xr = 65535;
  if (xr > (nodes + 31) / 32) xr = (nodes + 31) / 32;
  if (xr < 1) xr = 1;
  a.chunk = (nodes + xr - 1) / xr;
  if (a.chunk > chunk_max) a.chunk = chunk_max;
  a.nchunks = (nodes + a.chunk - 1) / a.chunk;
  if (xr > a.nchunks) xr = a.nchunks;
  a.xr = (int)xr;
  P->coef_count = (size_t)(L + 1) * a.nin * a.nin;
  P->conv = opt.shard_end == 0 && opt.shard_begin == 0 && opt.tile_override == 0 && conv_layout(P);
  int st = GBSBIN_OK;
  const size_t walk_state = P->coef_count * (sizeof(double2) + sizeof(float4));
  // the convolution's tables and states; where the device has no room for them the walk serves the plan
  if (P->conv) {
    P->state_bytes = walk_state + (P->coef_count + 1) * sizeof(longlong2);   // and the exponent
    if ((st = conv_setup(P)) == GBSBIN_ERR_NOMEM) {
      P->conv = false;
      st = GBSBIN_OK;
    }
  }
  if (!P->conv) {
    P->state_bytes = walk_state;
    (st = dalloc(&P->d_state, P->state_bytes)) || (st = dalloc(&P->d_diag, GBSBIN_DIAG_DOUBLES)) ||
        (st = dalloc(&P->d_table, (size_t)P->table_size));
  }
  if (!st && !P->conv)                           // the walk's roots, partial sums and transform
    (st = dalloc(&P->d_xtw, (size_t)xoff)) || (st = dalloc(&P->d_xtw_df, (size_t)xoff)) ||
        (st = dalloc(&P->d_zr, (size_t)a.rsum)) || (st = dalloc(&P->d_zr_df, (size_t)a.rsum)) ||
        (st = dalloc(&P->d_tw, (size_t)a.rsum)) || (st = dalloc(&P->d_parts, (size_t)xr * g.n_full)) ||
        (st = dalloc(&P->d_bufA, (size_t)g.n_full)) || (st = dalloc(&P->d_bufB, (size_t)g.n_full)) ||
        (st = dalloc(&P->d_bar, 4));
  if (st) {
    free_all(P);
    delete P;
    return st;
  }
  if (cudaMallocHost(&P->h_stage, P->state_bytes ? P->state_bytes : 1) != cudaSuccess) {
    cudaGetLastError();
    P->h_stage = nullptr;
    free_all(P);
    delete P;
    return GBSBIN_ERR_NOMEM;
  }
  if (opt.want_timing &&
      (cudaEventCreate(&P->ev0) != cudaSuccess || cudaEventCreate(&P->ev1) != cudaSuccess)) {
    cudaGetLastError();
    free_all(P);
    delete P;
    return GBSBIN_ERR_CUDA;
  }
  a.coef = reinterpret_cast<const double2*>(P->d_state);
  a.coef_df = reinterpret_cast<const float4*>(P->d_state + P->coef_count * sizeof(double2));
  a.xtw = P->d_xtw;
  a.xtw_df = P->d_xtw_df;
  a.zr = P->d_zr;
  a.zr_df = P->d_zr_df;
  a.parts = P->d_parts;
  st = stage_transfer(P, p->T);
  if (!st && (cudaMemcpy(P->d_state, P->h_stage, P->state_bytes, cudaMemcpyHostToDevice) != cudaSuccess ||
              cudaMemset(P->d_diag, 0, GBSBIN_DIAG_DOUBLES * sizeof(double)) != cudaSuccess)) {
    cudaGetLastError();
    st = GBSBIN_ERR_CUDA;
  }
  if (!st && !P->conv) {
    // roots from exact integer indices
    const double TWO_PI = 6.283185307179586476925286766559;
    std::vector<double2> xtw((size_t)std::max(xoff, 1)), zr((size_t)a.rsum), tw((size_t)a.rsum);
    std::vector<float4> xtw_df((size_t)std::max(xoff, 1)), zr_df((size_t)a.rsum);
    for (int d = 0; d < a.nd; ++d)
      for (int q = 0; q < a.drad[d]; ++q) {
        const cd v = std::polar(1.0, TWO_PI * (double)q / (double)a.drad[d]);
        xtw[a.doff[d] + q] = make_double2(v.real(), v.imag());
        xtw_df[a.doff[d] + q] = split_df(v);
      }
    for (int l = 0; l < L; ++l)
      for (int q = 0; q < g.radix[l]; ++q) {
        const cd v = std::polar(1.0, TWO_PI * (double)q / (double)g.radix[l]);
        zr[a.roff[l] + q] = make_double2(v.real(), v.imag());
        zr_df[a.roff[l] + q] = split_df(v);
        tw[a.roff[l] + q] = make_double2(v.real(), -v.imag());
      }
    if (cudaMemcpy(P->d_xtw, xtw.data(), (size_t)xoff * sizeof(double2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(P->d_xtw_df, xtw_df.data(), (size_t)xoff * sizeof(float4), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(P->d_zr, zr.data(), zr.size() * sizeof(double2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(P->d_zr_df, zr_df.data(), zr_df.size() * sizeof(float4), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(P->d_tw, tw.data(), tw.size() * sizeof(double2), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemset(P->d_bar, 0, 4 * sizeof(unsigned)) != cudaSuccess) {
      cudaGetLastError();
      st = GBSBIN_ERR_CUDA;
    }
  }
  if (st) {
    free_all(P);
    delete P;
    return st;
  }
  *out = P;
  return GBSBIN_OK;
}

int gbsbin_fock_plan_set_transfer(gbsbin_fock_plan* P, const gbsbin_complex* T, void* stream) {
  if (!P || !T) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  // the staging block may still feed an earlier upload on this stream
  if (cudaStreamSynchronize(s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  int st = stage_transfer(P, T);
  if (st) return st;
  if (P->state_bytes &&
      cudaMemcpyAsync(P->d_state, P->h_stage, P->state_bytes, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return GBSBIN_ERR_CUDA;
  return GBSBIN_OK;
}

long long gbsbin_fock_plan_table_size(const gbsbin_fock_plan* P) { return P ? P->table_size : -1; }

long long gbsbin_fock_plan_nodes(const gbsbin_fock_plan* P) { return P ? P->args.S : -1; }

int gbsbin_fock_execute(gbsbin_fock_plan* P, double* P_out, void* stream) {
  if (!P || !P_out) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  if (P->ev0 && cudaEventRecord(P->ev0, s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  if (P->conv) {
    FockConvArgs c = P->cv;
    c.P = P_out;
    c.diag = P->opt.want_diagnostics ? P->d_diag : nullptr;
    if (launch_fock_conv(c, P->layers.data(), (int)P->layers.size(), P->num_sms, s, &P->last_launches) != cudaSuccess)
      return GBSBIN_ERR_CUDA;
    P->executed = true;
    return P->ev1 && cudaEventRecord(P->ev1, s) != cudaSuccess ? GBSBIN_ERR_CUDA : GBSBIN_OK;
  }
  if (launch_fock(P->args, P->df, P->zt, s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  P->executed = true;
  P->last_launches = 2;                           // the Fock kernel and the fused DFT
  if (P->ev1 && cudaEventRecord(P->ev1, s) != cudaSuccess) return GBSBIN_ERR_CUDA;
  DftArgs d{};
  d.grid = P->args.grid;
  d.parts = P->d_parts;
  d.nparts = P->args.xr;
  d.pscale = 1.0 / (double)P->args.S;
  d.tw = P->d_tw;
  d.bufA = P->d_bufA;
  d.bufB = P->d_bufB;
  d.P = P_out;
  d.diag = P->opt.want_diagnostics ? P->d_diag : nullptr;
  d.table_size = P->table_size;
  return launch_dft_fused(d, P->d_bar, P->num_sms, s) == cudaSuccess ? GBSBIN_OK : GBSBIN_ERR_CUDA;
}

int gbsbin_fock_execute_host(gbsbin_fock_plan* P, double* P_out_host, void* stream) {
  if (!P || !P_out_host) return GBSBIN_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  int st = gbsbin_fock_execute(P, P->d_table, stream);
  if (!st && cudaMemcpyAsync(P_out_host, P->d_table, (size_t)P->table_size * sizeof(double),
                             cudaMemcpyDeviceToHost, s) != cudaSuccess)
    st = GBSBIN_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess && !st) st = GBSBIN_ERR_CUDA;
  return st;
}

int gbsbin_fock_diagnostics(gbsbin_fock_plan* P, gbsbin_diag* out, void* stream) {
  if (!P || !out) return GBSBIN_ERR_ARG;
  std::vector<double> part(GBSBIN_DIAG_DOUBLES, 0.0);
  double sum = 0.0, im = 0.0;
  if (P->opt.want_diagnostics) {
    if (cudaMemcpyAsync(part.data(), P->d_diag, part.size() * sizeof(double), cudaMemcpyDeviceToHost,
                        (cudaStream_t)stream) != cudaSuccess ||
        cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess)
      return GBSBIN_ERR_CUDA;
    const int nblk = std::min(GBSBIN_DIAG_SLOTS, std::max(0, (int)part[4 * GBSBIN_DIAG_SLOTS + 2]));
    for (int b = 0; b < nblk; ++b) {   // fixed order: deterministic
      sum += part[4 * b];
      im = std::fmax(im, part[4 * b + 1]);
    }
  }
  out->sum_P = sum;
  out->max_imag = im;
  out->min_pivot_re = 1.0;
  out->n_bad_points = 0;
  out->log_q1_re = 0.0;
  out->n_points = P->args.grid.npts;
  out->n_evaluated = P->args.grid.n_full;
  out->table_size = P->table_size;
  out->n = P->args.nin;
  out->kernel = P->kernel;
  out->point_kernel_ms = 0.0;
  out->backward_kernel_ms = 0.0;
  out->backward_path = 0;
  out->state_upload_bytes = (long long)P->state_bytes;
  out->launches = P->last_launches;
  if (P->ev1 && P->executed) {
    float ms = 0.f;
    if (cudaEventSynchronize(P->ev1) != cudaSuccess || cudaEventElapsedTime(&ms, P->ev0, P->ev1) != cudaSuccess) {
      cudaGetLastError();
      return GBSBIN_ERR_CUDA;
    }
    out->point_kernel_ms = ms;
  }
  if (P->opt.want_diagnostics && part[4 * GBSBIN_DIAG_SLOTS + 1] != 0.0) return GBSBIN_ERR_CUDA;
  if (P->opt.want_diagnostics && !(std::isfinite(sum))) return GBSBIN_ERR_NUMERIC;
  return GBSBIN_OK;
}

int gbsbin_fock_plan_destroy(gbsbin_fock_plan* P) {
  if (!P) return GBSBIN_OK;
  cudaDeviceSynchronize();
  free_all(P);
  delete P;
  return GBSBIN_OK;
}

}  // extern "C"
