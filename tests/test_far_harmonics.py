"""The tables that every product uses (far_harmonics in farfield.cu: a node's
moments to the (P + 1)^2 coefficients of its far field), on the host: with
random moments the harmonic sum is the monomial one of far_tables, which
tests/test_far_table.py holds to the oracle's truncated expansion."""
import os
import subprocess

from paper_1506_03745_gb300 import build

# farfield.cu itself, with what it needs of the rest of the library and no device call
SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "farfield.cu"
namespace pgb {
thread_local cudaStream_t g_alloc_stream = nullptr;
thread_local bool g_alloc_scoped = false;
void note_alloc() {}
void cuda_check(cudaError_t, const char*) {}
void fail(int, const std::string&) { std::abort(); }
}
using namespace pgb;
static double uniform() { return 2.0 * std::rand() / RAND_MAX - 1.0; }
int main() {
    double worst = 0;
    for (int P = 0; P <= PGB_MAX_P; ++P)
        for (double kappa : {0.0, 0.125, 1.5}) {
            const int T = n_terms(P), TR = far_cols(P);
            std::vector<double> har, mono, M(T);
            far_harmonics(P, kappa, har);
            far_tables(P, kappa, mono);
            for (int trial = 0; trial < 4; ++trial) {
                for (double& m : M) m = uniform();
                const double R[3] = {3 * uniform(), 3 * uniform(), 2 + uniform()};
                const double r = std::sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]), x = kappa * r;
                std::vector<double> g(P + 2);
                g[0] = 1;
                g[1] = -(1 + x);
                for (int p = 2; p <= P; ++p) g[p] = x * x * g[p - 2] - (2 * p - 1) * g[p - 1];
                for (int lap = 0; lap < 2; ++lap) {
                    double a = 0, size = 0, b = 0;
                    int row = 0;
                    for (int i = 0; i <= P; ++i)
                        for (int j = 0; j <= P - i; ++j)
                            for (int k = 0; k <= P - i - j; ++k, ++row) {
                                double c = 0;
                                for (int t = 0; t < T; ++t) c += mono[(size_t)lap * T * T + (size_t)row * T + t] * M[t];
                                const double s = std::pow(R[0], i) * std::pow(R[1], j) * std::pow(R[2], k) / std::pow(r, 2 * (i + j + k));
                                const double v = c * s * (lap ? 1.0 : g[i + j + k]);
                                a += v;
                                size += std::fabs(v);
                            }
                    const double n[3] = {R[0] / r, R[1] / r, R[2] / r};
                    double X = 1, Y = 0;
                    for (int m = 0; m <= P; ++m) {
                        double q0 = 1, q1 = 0;
                        for (int l = m; l <= P; ++l) {
                            if (l > m) {
                                const double c = l > 1 ? (double)((l - 1) * (l - 1) - m * m) / (4.0 * (l - 1) * (l - 1) - 1.0) : 0.0;
                                const double q = l == m + 1 ? n[2] : n[2] * q0 - c * q1;
                                q1 = q0;
                                q0 = q;
                            }
                            for (int s = 0; s < (m ? 2 : 1); ++s) {
                                const int j = l * l + (m ? 2 * m - 1 + s : 0);
                                double c = 0;
                                for (int t = 0; t < T; ++t) c += har[((size_t)lap * T + t) * TR + j] * M[t];
                                const double v = c * q0 * (s ? Y : X) * (lap ? 1.0 : g[l]) / std::pow(r, l);
                                b += v;
                                size += std::fabs(v);
                            }
                        }
                        const double xn = n[0] * X - n[1] * Y;
                        Y = n[0] * Y + n[1] * X;
                        X = xn;
                    }
                    worst = std::fmax(worst, std::fabs(a - b) / size);
                }
            }
        }
    std::printf("%.3e\n", worst);
    return worst <= 1e-13 ? 0 : 1;
}
"""


def test_harmonic_tables_equal_the_monomial_ones(tmp_path):
    """To 1e-13 of the terms' magnitudes (some hundred roundings of 2^-53 on
    either side)."""
    src, exe = tmp_path / "tables.cu", tmp_path / "tables"
    src.write_text(SOURCE)
    include = os.path.join(os.path.dirname(build.HERE), "include")
    c = subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O1", "-I", build.CSRC, "-I", include, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert c.returncode == 0, c.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
