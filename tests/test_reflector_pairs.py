"""The Householder reflector of the reductions to Hessenberg form in pairs of FP32: beta ||v||^2 = 2 to beta's own rounding,
so that the reflectors of a reduction do not add up the errors of their square roots.  The device header compiled on the
CPU, its intrinsics by their IEEE definitions."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_17742_gb300", "csrc")

MAIN = '''
#include <cuda_runtime.h>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
using std::fmaf; using std::fabs; using std::fma; using std::sqrt; using std::frexp; using std::ldexp;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fdiv_rn(float a, float b) { return a / b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline float __fsqrt_rn(float a) { return sqrtf(a); }
static inline float rsqrtf(float a) { return (float)(1.0 / std::sqrt((double)a)); }
static inline float __double2float_rn(double a) { return (float)a; }
static inline float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static inline unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static inline long long __double_as_longlong(double d) { long long u; std::memcpy(&u, &d, 8); return u; }
static inline double __longlong_as_double(long long u) { double d; std::memcpy(&d, &u, 8); return d; }
static inline float __shfl_sync(unsigned, float v, int) { return v; }
static inline double __shfl_sync(unsigned, double v, int) { return v; }
static inline float __shfl_xor_sync(unsigned, float v, int) { return v; }
static inline double __shfl_xor_sync(unsigned, double v, int) { return v; }
#include "gbsbin_hess.cuh"
using namespace gbsbin;
template <class Ar>
static void run(int m) {             // rms of beta ||v||^2 / 2 - 1 and of | |alpha| / ||x|| - 1 |, in extended precision
  std::mt19937_64 g(m);
  std::normal_distribution<double> d;
  long double su = 0, sa = 0;
  const int cases = 400;
  for (int c = 0; c < cases; ++c) {
    typename Ar::E x[128], rest = Ar::zero(), alpha, v0, beta;
    for (int i = 0; i < m; ++i) x[i] = Ar::from(make_double2(0.1 * d(g), 0.1 * d(g)));
    for (int i = 1; i < m; ++i) rest = Ar::add(rest, Ar::norm2(x[i]));
    reflector<Ar>(rest, x[0], alpha, v0, beta);
    auto sq = [](typename Ar::E e) { const double2 v = Ar::to(e); return (long double)v.x * v.x + (long double)v.y * v.y; };
    long double r = 0;
    for (int i = 1; i < m; ++i) r += sq(x[i]);
    const long double u = (long double)Ar::to(beta).x * (r + sq(v0)) / 2 - 1, a = sqrtl(sq(alpha) / (r + sq(x[0]))) - 1;
    su += u * u;
    sa += a * a;
  }
  std::printf("%Lg %Lg\\n", sqrtl(su / cases), sqrtl(sa / cases));
}
int main() { for (int m : {2, 3, 10, 100}) { run<ArDF>(m); run<ArF64>(m); } }
'''


def test_beta_belongs_to_v(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "reflector")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", str(tmp_path / "main.cpp"), "-I", CSRC, "-I",
                    os.path.join(cuda, "include"), "-o", exe], check=True)
    rows = [[float(v) for v in line.split()] for line in
            subprocess.run([exe], capture_output=True, text=True, check=True).stdout.splitlines()]
    for (pu, pa), (du, da) in zip(rows[0::2], rows[1::2]):
        # a rounding of beta (a pair keeps 2^-48) and of the sum ||v||^2, their errors independent
        assert pu < 2.0 ** -47.5 and pa < 2.0 ** -44
        assert du < 2.0 ** -52 and da < 2.0 ** -50
