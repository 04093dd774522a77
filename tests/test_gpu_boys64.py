"""The FP64 Boys function and reciprocal square root of the quartet kernels
(csrc/boys.cuh) against extended precision on the host: all orders, both table layouts,
T = 0, grid points and the midpoints between them (with the nearest neighbours of each),
both sides of the table's end at T = 36, and large T.

Bounds, in units of u = 2^-53, relative:
 * rsqrt_fp64: the last addition 1, the residual's rounding 1/2, the series 2^-5: 2.
 * T < 36: F_L by Horner's rule, table and sum 4; each downward step multiplies by
   1/(2n+1) (2) after one multiply-add (1), and averages over e^{-T}, itself within 4:
   4 + 3 (L - n).
 * T >= 36: F_0 is 2 from the root, 1 + 1 from the constant; h = rs^2 / 2 is 5, each
   upward step two roundings, h and one product: 4 + 8 n (e^{-T} is left out from T = 72
   on, where it is below 2^-59 of its term: 2^-6 a step).
 * e^{-T} of the large-T branch, 36 <= T < 72: the square of table 1, polynomial 2,
   truncation 1/4 and product 1, rounded: 10.
"""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2510_24968_gb300")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "fsim_internal.h"
using namespace fsim;

// one thread per argument; out[n * count + i]
template <int L, bool SCALED>
__global__ void boys_k(const double* T, int count, const double* tab, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  double F[L + 1];
  if (SCALED) boys_fp64_u<L, true>(-2.0 * T[i], F, tab + (size_t)L * kBoysOrderLd, kBoysK64 + 1, kBoysK64);
  else boys_fp64_u<L, false>(-2.0 * T[i], F, tab + L, kBoysCols, kBoysCols - 1 - L);
  for (int n = 0; n <= L; ++n) out[(size_t)n * count + i] = F[n];
}
__global__ void rsqrt_k(const double* x, int count, double* out, const double* tail) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  double d;
  const double* row;
  const double e = tail ? boys_exp(-2.0 * x[i], tail, kBoysCols, kBoysCols - 1, d, row) : 0.0;
  out[i] = tail ? e * e : rsqrt_fp64(x[i]);
}

static std::vector<long double> boys_ref(double T, int top) {
  const int M = top + 24;
  long double term = 1.0L / (2 * M + 1), sum = term;
  for (int k = 1; k < 20000; ++k) {
    term *= 2.0L * T / (2 * M + 2 * k + 1);
    sum += term;
    if (term < 1e-25L * sum) break;
  }
  std::vector<long double> F(M + 1);
  const long double e = expl(-(long double)T);
  F[M] = e * sum;
  for (int m = M - 1; m >= 0; --m) F[m] = (2.0L * T * F[m + 1] + e) / (2 * m + 1);
  return F;
}

static std::vector<double> args;
static double *d_T, *d_out;
static std::vector<std::vector<long double>> ref;
static int fail = 0;

template <int L, bool SCALED>
static void check(const double* tab) {
  const int n = (int)args.size();
  boys_k<L, SCALED><<<(n + 127) / 128, 128>>>(d_T, n, tab, d_out);
  std::vector<double> out((size_t)(L + 1) * n);
  if (cudaMemcpy(out.data(), d_out, sizeof(double) * out.size(), cudaMemcpyDeviceToHost) != cudaSuccess) fail = 1;
  double worst = 0.0, at = 0.0;
  int wn = 0;
  for (int m = 0; m <= L; ++m)
    for (int i = 0; i < n; ++i) {
      const double tol = ldexp(args[i] < 36.0 ? 4 + 3 * (L - m) : 4 + 8 * m, -53);
      const long double r = ref[i][m];
      const double err = (double)(fabsl(out[(size_t)m * n + i] - r) / r) / tol;
      if (!(err <= worst)) { worst = err; at = args[i]; wn = m; }
    }
  printf("boys L=%d scaled=%d worst/bound %.3f at T=%.17g n=%d\n", L, (int)SCALED, worst, at, wn);
  if (!(worst <= 1.0)) fail = 1;
  if constexpr (L < (SCALED ? 8 : 12)) check<L + 1, SCALED>(tab);
}

int main() {
  fsim_atom a{1, {0, 0, 0}};
  double al = 1.0, co = 1.0;
  fsim_shell_desc s{0, 0, 1, &al, &co};
  fsim_basis* b = nullptr;
  if (fsim_basis_create(&a, 1, &s, 1, &b) != FSIM_OK) return 2;
  auto around = [&](double T) {
    for (double t : {nextafter(T, 0.0), T, nextafter(T, 1e300)}) args.push_back(t);
  };
  args.push_back(0.0);
  args.push_back(1e-300);
  args.push_back(1e-20);
  for (int i = 0; i < 2 * 36 * 16; ++i) around((i + 1) / 32.0);  // midpoints and grid points, the last T = 36
  for (double T = 36.03; T < 1.0e3; T *= 1.007) around(T);
  for (int T = 37; T <= 90; ++T) around(T);  // e^{-T} is left out from 72 on
  for (double T : {1.0e-5, 0.01, 17.3, 35.99, 1.0e3, 2.0e3}) around(T);
  const int n = (int)args.size();
  for (double T : args) ref.push_back(boys_ref(T, 12));
  if (cudaMalloc(&d_T, sizeof(double) * n) || cudaMalloc(&d_out, sizeof(double) * 13 * n)) return 2;
  if (cudaMemcpy(d_T, args.data(), sizeof(double) * n, cudaMemcpyHostToDevice)) return 2;
  check<0, true>(b->d_boys64s);
  check<0, false>(b->d_boys64);
  std::vector<double> x, out;
  for (double T = 36.0; T < 72.0; T += 0.0073) x.push_back(T);
  x.push_back(nextafter(72.0, 0.0));
  for (int pass = 0; pass < 2; ++pass) {
    const int m = (int)x.size();
    double *dx, *dy;
    if (cudaMalloc(&dx, sizeof(double) * m) || cudaMalloc(&dy, sizeof(double) * m)) return 2;
    if (cudaMemcpy(dx, x.data(), sizeof(double) * m, cudaMemcpyHostToDevice)) return 2;
    rsqrt_k<<<(m + 127) / 128, 128>>>(dx, m, dy, pass == 0 ? b->d_boys64 : nullptr);
    out.resize(m);
    if (cudaMemcpy(out.data(), dy, sizeof(double) * m, cudaMemcpyDeviceToHost)) return 2;
    double worst = 0.0, at = 0.0;
    for (int i = 0; i < m; ++i) {
      const long double r = pass == 0 ? expl(-(long double)x[i]) : 1.0L / sqrtl((long double)x[i]);
      const double err = (double)(fabsl(out[i] - r) / r) / ldexp(pass == 0 ? 10 : 2, -53);
      if (!(err <= worst)) { worst = err; at = x[i]; }
    }
    printf("%s worst/bound %.3f at %.17g\n", pass == 0 ? "tail" : "rsqrt", worst, at);
    if (!(worst <= 1.0)) fail = 1;
    cudaFree(dx);
    cudaFree(dy);
    // rsqrt: mantissas over every exponent that two exponents' sum or T can have
    x.clear();
    unsigned long long r = 88172645463325252ull;
    for (int e = -300; e <= 300; ++e)
      for (int k = 0; k < 64; ++k) {
        r ^= r << 13; r ^= r >> 7; r ^= r << 17;
        x.push_back(ldexp(1.0 + (k < 2 ? k * (1 - ldexp(1.0, -52)) : (double)(r >> 12) * ldexp(1.0, -52)), e));
      }
  }
  fsim_basis_destroy(b);
  return fail;
}
"""


def test_boys_and_rsqrt_against_extended_precision(tmp_path):
    from paper_2510_24968_gb300.build import build
    build()
    src, exe = tmp_path / "boys.cu", tmp_path / "boys"
    src.write_text(PROGRAM)
    r = subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O3",
                        "--expt-relaxed-constexpr", "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"),
                        str(src), "-o", str(exe), "-L", PKG, "-lfsim", "-Xlinker", "-rpath=" + PKG],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
