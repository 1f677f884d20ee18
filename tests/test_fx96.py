"""The 96-bit sums of the fixed-point FP64 GEMV (csrc/fx96.h), compiled for the host, against
exact integers: sums of as many products of the largest size as a row can have (the sizes
that shared memory allows end at 8,192 columns), all of one sign or the other, and
random ones."""
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "fx96.h"
#include <cstdio>
// stdin: n, then n pairs h x (sums of 64 products); stdout: the high 64 and the low 32 bits
int main() {
    int n;
    if (std::scanf("%d", &n) != 1) return 1;
    uint64_t lo = 0;
    int32_t hi = 0;
    for (int k = 0; k < n; ++k) {
        long long h, x;
        if (std::scanf("%lld %lld", &h, &x) != 2) return 1;
        fx96_add(lo, hi, fx96_part(h, x));
    }
    std::printf("%lld %u\n", (long long)fx96_high(lo, hi), fx96_low(lo));
    return 0;
}
"""


def test_sums_of_the_largest_products(tmp_path):
    src, exe = tmp_path / "sums.cpp", tmp_path / "sums"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2204_13254_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)

    def run(parts):
        text = f"{len(parts)}\n" + "\n".join(f"{h} {x}" for h, x in parts) + "\n"
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()
        return (int(out[0]) << 32) + int(out[1])

    rng = random.Random(3)
    top = 64 << 56   # sum of 64 products hi hi' of the largest size (lo = 0 there)
    cross = 64 * ((1 << 57) - (1 << 29))
    for n in (1, 15, 16, 17, 29, 58, 128):          # parts of 64 products: 64 .. 8,192 columns
        for parts in ([(top - 1, 0)] * n, [(-top, 0)] * n, [(top - 1 - (64 << 29), cross)] * n,
                      [(rng.randint(-top, top - 1), rng.randint(-cross, cross)) for _ in range(n)]):
            exact = sum((h << 29) + x for h, x in parts)       # units of 2^29
            assert 0 <= exact - (run(parts) << 8) < n << 8      # eight bits of each part dropped
