"""The reductions of the one-kernel Schur CG go through a buffer in global memory with one
meeting of all CTAs between the writes and the reads of a reduction.  A model of that
exchange, compiled with the rows that the kernel uses (csrc/cg_rows.h): one CTA runs ahead
as far as the meetings allow, another reads as late as they allow.  Every CTA must read
what all of them wrote for the same reduction."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include "cg_rows.h"
#include <vector>
// Meetings are numbered; an event is a write (before its meeting) or a read (after it).
// Between two meetings a fast CTA does all of its events before a slow one does any.
int run(const std::vector<CgSums>& ops, const std::vector<int>& meetings_before) {
    double buf[kCgRows][2] = {};
    int bad = 0;
    auto write = [&](int cta, int k) {
        for (int i = 0; i < ops[k].n; ++i) buf[ops[k].row + i][cta] = 10.0 * k + i + 1;
    };
    auto read = [&](int k) {
        for (int i = 0; i < ops[k].n; ++i)
            for (int c = 0; c < 2; ++c) bad += buf[ops[k].row + i][c] != 10.0 * k + i + 1;
    };
    // fast CTA 0, slow CTA 1.  After the meeting of reduction k, CTA 0 reads it and, with no
    // meeting in front of reduction k + 1, already writes that one; then CTA 1 reads reduction k.
    write(0, 0);
    write(1, 0);
    for (size_t k = 0; k < ops.size(); ++k) {
        const bool next = k + 1 < ops.size(), ahead = next && meetings_before[k + 1] == 0;
        read(k);
        if (ahead) write(0, k + 1);
        read(k);
        if (next && !ahead) write(0, k + 1);
        if (next) write(1, k + 1);
    }
    return bad;
}
int main() {
    // start, then two iterations: the operator (at least one meeting) before every p . q, nothing
    // but arithmetic between p . q and the residual's sums
    std::vector<CgSums> ops{kCgStart, kCgPq, kCgRes, kCgPq, kCgRes};
    return run(ops, {0, 1, 0, 1, 0}) != 0;
}
"""


def test_no_sum_is_overwritten_before_every_cta_has_read_it(tmp_path):
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL)
    inc = os.path.join(ROOT, "paper_2204_13254_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", inc, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
    kernel = open(os.path.join(inc, "resident.cu")).read()
    for use in ("sums(kCgStart,", "sums(kCgPq,", "sums(kCgRes,"):   # the kernel takes its rows from there
        assert kernel.count(use) == 1
