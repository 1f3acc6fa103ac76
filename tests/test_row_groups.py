"""The refinement's split of partial rows stays inside its buffer.

cv_rows.h is plain C++, so the geometry the kernel uses is compiled for the
host and walked for every bin count, precision, row count and CTA size in
use: 512 threads (64 rows or more), 256 threads (batches and the server) and
the bins rounded up to warps, at least 64 (fewer rows).
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1408_6373_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "cv_rows.h"
int main()
{
    int bad = 0;
    for (int N = 2; N <= 256; ++N)
        for (int fp64 = 0; fp64 < 2; ++fp64)
            for (int cta = 0; cta < 3; ++cta) {
                const int threads = cta == 0 ? 512 : cta == 1 ? 256 : N <= 64 ? 64 : (N + 31) / 32 * 32;
                const int entries = cv::row_entries(cta == 1 ? 256 : 512, 256);
                const int V = cv::row_vector(N, fp64);
                for (int G = 1; G <= 2048; ++G) {
                    const cv::RowGroups g = cv::row_groups(threads, N, cv::row_reciprocal(N), fp64, G, entries);
                    const bool ok = g.R >= 1 && g.R <= G && g.stride >= N && (g.R - 1) * g.stride + N <= entries &&
                                    g.R * (N / V) <= threads && N % V == 0 && (N << g.lT) <= threads;
                    if (!ok && bad++ < 10)
                        printf("N %d fp64 %d threads %d G %d: R %d stride %d of %d\n", N, fp64, threads, G, g.R,
                               g.stride, entries);
                }
                // quotients by N of every value the kernel divides
                for (int x = 0; x < 65536; x += cta ? 65536 : 1)
                    if (cv::row_quotient(x, cv::row_reciprocal(N)) != x / N) ++bad;
            }
    return bad ? 1 : 0;
}
"""


def test_row_groups_fit_the_buffer(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "rows.cpp", tmp_path / "rows"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
