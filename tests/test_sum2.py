"""How the one-kernel GMRES joins its FP32 sums of 128 products (csrc/sum2.h, compiled for the
host): as exactly as the FP64 join of the kernels beyond its size, in any order of the
exchange.  Sums of 16 FP32 numbers per lane and 32 lanes that cancel to a small fraction
of their size, where a join in FP32 loses every digit."""
import os
import subprocess

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "sum2.h"
#include <cstdio>
#include <vector>
// stdin: 32 lanes of n floats (bytes); stdout: hi + lo of the lanes' sums after the exchange, in lane 0 and 31
int main(int argc, char** argv) {
    int n = 0;
    std::sscanf(argv[1], "%d", &n);
    std::vector<float> f(32 * n);
    if (std::fread(f.data(), 4, f.size(), stdin) != f.size()) return 1;
    Sum2 p[32], q[32];
    for (int l = 0; l < 32; ++l) {
        p[l] = {0.0f, 0.0f};
        for (int k = 0; k < n; ++k) p[l] = sum2_add(p[l], Sum2{f[l * n + k], 0.0f});
    }
    for (int o = 16; o > 0; o >>= 1) {
        for (int l = 0; l < 32; ++l) q[l] = sum2_add(p[l], p[l ^ o]);
        for (int l = 0; l < 32; ++l) p[l] = q[l];
    }
    std::printf("%.17g %.17g\n", (double)p[0].hi + (double)p[0].lo, (double)p[31].hi + (double)p[31].lo);
    return 0;
}
"""


def test_join_of_partial_sums(tmp_path):
    src, exe = tmp_path / "join.cpp", tmp_path / "join"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2204_13254_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    rng = np.random.default_rng(5)
    for n in (1, 2, 4):
        for _ in range(20):
            f = rng.standard_normal(32 * n).astype(np.float32)
            f[:16 * n] = -f[16 * n:][rng.permutation(16 * n)]     # cancels exactly
            f[rng.integers(32 * n)] += np.float32(1e-4)
            exact = float(np.sum(f.astype(np.float64)))           # (exact: 24-bit numbers of like size)
            got = [float(v) for v in subprocess.run([str(exe), str(n)], input=rng.permutation(f).tobytes(),
                                                    capture_output=True, check=True).stdout.split()]
            # each of the 32 n - 1 additions keeps its error in lo, whose own sum rounds at 2^-24 of that error
            bound = 32 * n * 2.0**-45 * float(np.abs(f).max()) * 32 * n
            assert all(abs(v - exact) <= bound for v in got)
            assert got[0] == got[1]                               # every lane, hence every CTA, has the same number
