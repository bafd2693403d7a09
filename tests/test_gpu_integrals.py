"""GPU test of the quadrature kernel's substep integrals (k_integrals), point by
point, with and without the FAS term, the residual and the forcing: a small
program built with nvcc launches the kernel and forms the same sums on the host
in FP64.

Tolerance: with B the sum of the magnitudes of a point's terms, each side rounds
every term and partial sum, at most ten of each, so the two are within 20 x
2^-53 B (a fixed-point sum is off by at most 6 x 2^-53 of its largest term)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "paper_1307_7867_gb300/csrc/kernels.cuh"
namespace h3d { void count_launch() {} }
using namespace h3d;
static unsigned long long seed = 1;
static double rnd() {  // uniform in [-1, 1)
  seed = seed * 6364136223846793005ull + 1442695040888963407ull;
  return (double)(long long)(seed >> 11) * (1.0 / 4503599627370496.0) - 1.0;
}
// argv: M N tau res spread; prints the largest error of I and of the residual's
// maximum over their tolerances
int main(int argc, char** argv) {
  const int M = atoi(argv[1]), N = atoi(argv[2]), tau = atoi(argv[3]), res = atoi(argv[4]), spread = atoi(argv[5]);
  const bool forced = argc > 6 && atoi(argv[6]);
  const int B = N > 127 ? 1 : 2, step = N > 127 ? 13 : N > 31 ? 3 : 1;
  const Grid g = make_grid(N);
  std::vector<ItemSDC> it(B);
  for (int b = 0; b < B; ++b) {
    memset(&it[b], 0, sizeof(ItemSDC));
    for (int m = 0; m + 1 < M; ++m) {
      it[b].dtm[m] = 0.01 * (1.5 + rnd());
      it[b].gS[m] = forced ? 0.03 * rnd() : 0.0;
      for (int j = 0; j < M; ++j) it[b].dtS[m][j] = 0.02 * rnd();
    }
    fix_coefficients(it[b], M);
  }
  std::vector<double> U((size_t)B * M * g.fs), F(U.size()), T((size_t)B * (M - 1) * g.fs), I(T.size(), 0.0), phi(N);
  for (double& x : U) x = rnd();
  for (double& x : F) x = 50.0 * rnd() * (spread ? std::ldexp(1.0, -(int)(seed >> 40) % 30) : 1.0);
  for (double& x : T) x = 0.1 * rnd();
  for (int i = 0; i < N; ++i) phi[i] = sin(M_PI * (i + 1) / (N + 1));
  double *dU, *dF, *dT, *dI, *dphi;
  ItemSDC* dit;
  unsigned long long* dn;
  auto up = [](auto*& d, const auto& h) {
    return cudaMalloc((void**)&d, h.size() * sizeof(h[0])) == cudaSuccess &&
           cudaMemcpy(d, h.data(), h.size() * sizeof(h[0]), cudaMemcpyHostToDevice) == cudaSuccess;
  };
  std::vector<unsigned long long> n(B, 0ull);
  if (!up(dU, U) || !up(dF, F) || !up(dT, T) || !up(dI, I) || !up(dphi, phi) || !up(dit, it) || !up(dn, n)) return 2;
  if (launch_integrals(M, g, B, dU, dF, tau ? dT : nullptr, dI, dit, dphi, res ? dn : nullptr, nullptr, 0) !=
          cudaSuccess ||
      cudaDeviceSynchronize() != cudaSuccess)
    return 3;
  cudaMemcpy(I.data(), dI, I.size() * 8, cudaMemcpyDeviceToHost);
  cudaMemcpy(n.data(), dn, B * 8, cudaMemcpyDeviceToHost);
  double worst = 0.0, rworst = 0.0;
  for (int b = 0; b < B; ++b) {
    double rmax = 0.0, rtol = 0.0;
    for (int k = 0; k < N; ++k)
      for (int j = 0; j < N; j += res ? 1 : step)
        for (int i = 0; i < N; ++i) {
          const size_t p = (size_t)k * g.plane + (size_t)j * g.px + i;
          const double ph = phi[i] * phi[j] * phi[k], u0 = U[(size_t)b * M * g.fs + p];
          double cum = 0.0, cumB = std::fabs(u0);
          for (int m = 0; m + 1 < M; ++m) {
            double J = it[b].gS[m] * ph, mag = std::fabs(J);
            for (int q = 0; q < M; ++q) {
              const double t = it[b].dtS[m][q] * F[((size_t)b * M + q) * g.fs + p];
              J += t;
              mag += std::fabs(t);
            }
            if (tau) {
              const double t = T[((size_t)b * (M - 1) + m) * g.fs + p];
              J += t;
              mag += std::fabs(t);
            }
            const double d = it[b].dtm[m] * F[((size_t)b * M + m + 1) * g.fs + p];
            const double want = J - d + (m == 0 ? u0 : 0.0);
            const double tol = 20 * std::ldexp(1.0, -53) * (mag + std::fabs(d) + (m == 0 ? std::fabs(u0) : 0.0));
            const double err = std::fabs(I[((size_t)b * (M - 1) + m) * g.fs + p] - want);
            if (!(err <= worst * tol)) worst = err / tol;
            cum += J;
            cumB += mag;
            const double um = U[((size_t)b * M + m + 1) * g.fs + p];
            rmax = std::fmax(rmax, std::fabs((u0 + cum) - um));
            rtol = std::fmax(rtol, 20 * std::ldexp(1.0, -53) * (cumB + std::fabs(um)));
          }
        }
    double got;
    memcpy(&got, &n[b], 8);
    if (res) rworst = std::fmax(rworst, std::fabs(got - rmax) / rtol);
  }
  printf("%g %g\n", worst, rworst);
  return 0;
}
'''


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("integrals")
    (d / "p.cu").write_text(PROGRAM)
    exe = str(d / "p")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", f"-I{ROOT}",
                    f"-I{ROOT}/include", "-o", exe, str(d / "p.cu"),
                    f"{ROOT}/paper_1307_7867_gb300/csrc/sdc_kernels.cu"], check=True, capture_output=True)
    return exe


@pytest.mark.parametrize("M", [2, 3, 4, 5])
@pytest.mark.parametrize("N,tau,res,spread,forced", [(31, 0, 0, 0, 1), (31, 1, 1, 0, 1), (31, 0, 1, 1, 0),
                                                     (63, 1, 0, 1, 1), (127, 1, 0, 0, 0), (127, 0, 1, 0, 1)])
def test_integrals_point_by_point(program, M, N, tau, res, spread, forced):
    out = subprocess.run([program, *map(str, (M, N, tau, res, spread, forced))], capture_output=True, text=True)
    assert out.returncode == 0, out
    err, rerr = map(float, out.stdout.split())
    assert err <= 1.0 and rerr <= 1.0


def test_integrals_of_the_largest_split(program):
    """255^3: eight planes a thread, with a remainder of seven."""
    out = subprocess.run([program, "3", "255", "1", "0", "0", "1"], capture_output=True, text=True)
    assert out.returncode == 0, out
    assert float(out.stdout.split()[0]) <= 1.0
