// Spectral form of a Hermitian matrix for the one-group plans, the small trees' first group and heralded states,
// FP64 on the host: Householder reduction to tridiagonal form, then the implicitly shifted QR iteration with
// Wilkinson's shift (Golub and Van Loan, Matrix Computations, 8.3), the unitary applied to given vectors instead
// of being formed: O(n^3) for the reduction, O(n^2) per vector for the rest.  The vectors are the columns of
// an n x m array held by rows, so that a reflector's products and a plane rotation run along contiguous entries.
#include <algorithm>
#include <cmath>
#include <limits>

#include "gbsbin_host_state.h"

namespace gbsbin {
namespace {

using cd = std::complex<double>;

// sum_j a_j v_j over [j0, n) of split rows, in four interleaved partial sums (fixed order)
inline void row_dot(const double* ar, const double* ai, const double* vr, const double* vi, int j0, int n, double* re,
                    double* im) {
  double r[4] = {0, 0, 0, 0}, m[4] = {0, 0, 0, 0};
  int j = j0;
  for (; j + 4 <= n; j += 4)
    for (int q = 0; q < 4; ++q) {
      r[q] += ar[j + q] * vr[j + q] - ai[j + q] * vi[j + q];
      m[q] += ar[j + q] * vi[j + q] + ai[j + q] * vr[j + q];
    }
  for (; j < n; ++j) {
    r[0] += ar[j] * vr[j] - ai[j] * vi[j];
    m[0] += ar[j] * vi[j] + ai[j] * vr[j];
  }
  *re = (r[0] + r[1]) + (r[2] + r[3]);
  *im = (m[0] + m[1]) + (m[2] + m[3]);
}

// y += a x of split rows (complex a)
inline void axpy(double ar, double ai, const double* __restrict__ xr, const double* __restrict__ xi,
                 double* __restrict__ yr, double* __restrict__ yi, int m) {
  for (int j = 0; j < m; ++j) {
    yr[j] += ar * xr[j] - ai * xi[j];
    yi[j] += ar * xi[j] + ai * xr[j];
  }
}

// |(x, z)|: the square root of the sum of squares where neither overflows nor loses digits
inline double norm2d(double x, double z) {
  const double q = x * x + z * z;
  return q > 1e-280 && q < 1e280 ? std::sqrt(q) : std::hypot(x, z);
}

// Eigenvalues of the real symmetric tridiagonal (d, e) into d; every plane rotation is also applied
// to the vectors' rows (which become Z^T X).  False if a block does not converge.
bool tridiagonal_qr(std::vector<double>& d, std::vector<double>& e, double* xr, double* xi, int m) {
  const int n = (int)d.size();
  const double eps = std::numeric_limits<double>::epsilon();
  auto rotate = [m](double c, double s, double* __restrict__ p, double* __restrict__ q) {
    for (int j = 0; j < m; ++j) {
      const double a = p[j], b = q[j];
      p[j] = c * a + s * b;
      q[j] = c * b - s * a;
    }
  };
  int hi = n - 1;
  long long budget = 60LL * n + 60;
  while (hi > 0) {
    int lo = hi;                                // the unreduced block ending at hi
    while (lo > 0) {
      if (std::fabs(e[lo - 1]) <= eps * (std::fabs(d[lo - 1]) + std::fabs(d[lo])) || std::fabs(e[lo - 1]) < std::numeric_limits<double>::min()) {
        e[lo - 1] = 0.0;
        break;
      }
      --lo;
    }
    if (lo == hi) {
      --hi;
      continue;
    }
    if (--budget < 0) return false;
    // Wilkinson's shift: the eigenvalue of the trailing 2 x 2 nearer to d[hi]
    const double b = e[hi - 1], g = 0.5 * (d[hi - 1] - d[hi]);
    const double mu = d[hi] - b * (b / (g + std::copysign(std::hypot(g, b), g)));
    double x = d[lo] - mu, z = e[lo];
    for (int k = lo; k < hi; ++k) {             // chase the bulge down the block
      const double h = norm2d(x, z);
      const double c = h > 0.0 ? x / h : 1.0, s = h > 0.0 ? z / h : 0.0;
      if (k > lo) e[k - 1] = h;
      const double t = s * (d[k + 1] - d[k]) + 2.0 * c * e[k];   // d_k' + d_{k+1}' = d_k + d_{k+1}
      d[k] += s * t;
      d[k + 1] -= s * t;
      e[k] = c * t - e[k];
      x = e[k];
      if (k + 1 < hi) {
        z = s * e[k + 1];
        e[k + 1] *= c;
      }
      rotate(c, s, xr + (size_t)k * m, xr + (size_t)(k + 1) * m);
      rotate(c, s, xi + (size_t)k * m, xi + (size_t)(k + 1) * m);
    }
  }
  return true;
}

}  // namespace

// Rows are updated and multiplied in one pass over the matrix per column: with the reflector of
// the next column known (its column updated first, O(n)), every remaining row takes the last
// column's rank-2 update and its product with the next reflector together; rows dealt cyclically
// to the host threads, each row's sums in a fixed order.
bool hermitian_spectrum(const std::vector<cd>& A, int n, std::vector<double>& lam, double* xr, double* xi, int m) {
  std::vector<double> re((size_t)n * n), im((size_t)n * n);
  for (size_t q = 0; q < re.size(); ++q) {
    re[q] = A[q].real();
    im[q] = A[q].imag();
  }
  const int nt = host_threads();
  std::vector<double> vr(n, 0.0), vi(n, 0.0), wr(n, 0.0), wi(n, 0.0), pr(n), pi(n), nvr(n, 0.0), nvi(n, 0.0);
  std::vector<double> tr(m), ti(m);             // v^H X
  std::vector<cd> sub(n, cd(0.0));              // sub[k] = entry (k + 1, k) of the tridiagonal form
  bool pending = false;                         // (v, w): the rank-2 update not yet applied
  for (int k = 0; k + 1 < n; ++k) {
    // column k below the diagonal, with the pending update: row k's conjugate
    double* rk = &re[(size_t)k * n];
    double* ik = &im[(size_t)k * n];
    if (pending)
      for (int j = k; j < n; ++j) {             // A_kj -= v_k conj(w_j) + w_k conj(v_j)
        rk[j] -= vr[k] * wr[j] + vi[k] * wi[j] + wr[k] * vr[j] + wi[k] * vi[j];
        ik[j] -= vi[k] * wr[j] - vr[k] * wi[j] + wi[k] * vr[j] - wr[k] * vi[j];
      }
    // the column scaled by a power of two (exact) that brings its largest component to [1/2, 1): the squares of
    // small entries and the square of beta leave FP64's range from magnitudes of 1e-77 on
    double big = 0.0;
    for (int j = k + 1; j < n; ++j) big = std::max(big, std::max(std::fabs(rk[j]), std::fabs(ik[j])));
    int ex = 0;
    std::frexp(big, &ex);
    ex = std::max(ex, -1000);
    const double up = std::ldexp(1.0, -ex);
    double nrm2 = 0.0;
    for (int j = k + 2; j < n; ++j) {
      nvr[j] = rk[j] * up;
      nvi[j] = -ik[j] * up;
      nrm2 += nvr[j] * nvr[j] + nvi[j] * nvi[j];
    }
    nvr[k] = nvi[k] = 0.0;
    const cd x0(rk[k + 1] * up, -ik[k + 1] * up);
    const double ax0 = std::abs(x0), nrm = std::sqrt(nrm2 + std::norm(x0));
    double beta = 0.0;
    if (nrm2 > 0.0) {                           // v = x - alpha e, alpha = -e^{i arg x0} |x|
      const cd alpha = (ax0 > 0.0 ? -x0 / ax0 : cd(-1.0, 0.0)) * nrm;
      nvr[k + 1] = x0.real() - alpha.real();
      nvi[k + 1] = x0.imag() - alpha.imag();
      beta = 2.0 / (nrm2 + nvr[k + 1] * nvr[k + 1] + nvi[k + 1] * nvi[k + 1]);
      sub[k] = std::ldexp(1.0, ex) * alpha;
    } else {
      sub[k] = cd(rk[k + 1], -ik[k + 1]);
    }
    auto rows = [&](int t, int nth) {           // the rows below: update, then p = A v
      for (int i = k + 1 + t; i < n; i += nth) {
        double* ri = &re[(size_t)i * n];
        double* ii = &im[(size_t)i * n];
        if (pending) {
          const double a = vr[i], b = vi[i], c = wr[i], d = wi[i];
          const double *w0 = wr.data(), *w1 = wi.data(), *v0 = vr.data(), *v1 = vi.data();
          for (int j = k + 1; j < n; ++j) {
            ri[j] -= a * w0[j] + b * w1[j] + c * v0[j] + d * v1[j];
            ii[j] -= b * w0[j] - a * w1[j] + d * v0[j] - c * v1[j];
          }
        }
        if (beta != 0.0) row_dot(ri, ii, nvr.data(), nvi.data(), k + 1, n, &pr[i], &pi[i]);
      }
    };
    if (n - k >= 160) parallel_run(nt, rows);
    else rows(0, 1);
    pending = beta != 0.0;
    if (!pending) continue;
    // w = beta p - (beta^2 (v^H p) / 2) v;  A <- A - v w^H - w v^H
    double h = 0.0;                             // v^H p, real for Hermitian A
    for (int j = k + 1; j < n; ++j) h += nvr[j] * pr[j] + nvi[j] * pi[j];
    const double half = 0.5 * beta * beta * h;
    for (int j = k + 1; j < n; ++j) {
      wr[j] = beta * pr[j] - half * nvr[j];
      wi[j] = beta * pi[j] - half * nvi[j];
    }
    wr[k] = wi[k] = 0.0;
    vr.swap(nvr);
    vi.swap(nvi);
    if (m > 0) {                                // X <- (I - beta v v^H) X
      std::fill(tr.begin(), tr.end(), 0.0);
      std::fill(ti.begin(), ti.end(), 0.0);
      for (int i = k + 1; i < n; ++i)
        axpy(vr[i], -vi[i], xr + (size_t)i * m, xi + (size_t)i * m, tr.data(), ti.data(), m);
      for (int i = k + 1; i < n; ++i)
        axpy(-beta * vr[i], -beta * vi[i], tr.data(), ti.data(), xr + (size_t)i * m, xi + (size_t)i * m, m);
    }
  }
  if (pending) {                                // the last diagonal entry
    const int k = n - 1;
    re[(size_t)k * n + k] -= 2.0 * (vr[k] * wr[k] + vi[k] * wi[k]);
  }
  // phases that make the subdiagonal real and non-negative: T = F |T| F^H
  std::vector<double> e(n, 0.0);
  lam.resize(n);
  cd f = 1.0;
  for (int k = 0; k < n; ++k) {
    lam[k] = re[(size_t)k * n + k];
    double* row_r = xr + (size_t)k * m;
    double* row_i = xi + (size_t)k * m;
    for (int j = 0; j < m; ++j) {               // times conj(f)
      const double a = row_r[j], b = row_i[j];
      row_r[j] = f.real() * a + f.imag() * b;
      row_i[j] = f.real() * b - f.imag() * a;
    }
    if (k + 1 < n) {
      const double g = std::abs(sub[k]);
      if (g > 0.0) f *= sub[k] / g;
      e[k] = g;
    }
  }
  return tridiagonal_qr(lam, e, xr, xi, m);
}

}  // namespace gbsbin
