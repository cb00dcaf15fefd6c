"""The panel moments that a leaf's block reads (k_p2m), enumerated on the host
from the kernel's own index functions: at every compiled order each thread
stays inside the last panel's moments, and the threads of each share take
every moment once."""
import os
import subprocess

from paper_1506_03745_gb300 import build

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "treecode.cuh"
using namespace pgb;
int main() {
    for (int P = 0; P <= PGB_MAX_P; ++P) {
        if (!p_supported(P)) continue;
        const int T = n_terms(P), BT = p2m_threads(P), H = (T + BT - 1) / BT, NP = p2m_shares(P);
        const long n_pan = 5;
        std::vector<int> seen(NP * T, 0);
        for (int t = 0; t < BT; ++t)
            for (int h = 0; h < H; ++h) {
                const int k = p2m_index(P, t, h), s = p2m_share(P, t);
                if (k < 0) continue;
                if (k >= T || s >= NP || (n_pan - 1) * T + k >= n_pan * T) return std::printf("P %d thread %d reads %d of %d\n", P, t, k, T), 1;
                if (h > 0 && p2m_index(P, t, 0) < 0) return std::printf("P %d thread %d starts late\n", P, t), 1;
                ++seen[s * T + k];
            }
        for (int q : seen)
            if (q != 1) return std::printf("P %d: a moment is taken %d times\n", P, q), 1;
    }
    return 0;
}
"""


def test_every_read_is_inside_the_panel_moments(tmp_path):
    src, exe = tmp_path / "reads.cu", tmp_path / "reads"
    src.write_text(SOURCE)
    include = os.path.join(os.path.dirname(build.HERE), "include")
    subprocess.run([build.nvcc(), *build.ARCH, "-std=c++17", "-O0", "-I", build.CSRC, "-I", include, "-o", str(exe), str(src)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
