"""The refinement's split of partial rows, and its sums.

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
                    const cv::RowGroups g = cv::row_groups(threads, N, V, cv::row_reciprocal(N), fp64, G, entries);
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


# Rows added as the kernels do it (groups of every R-th row, 2^lT threads a
# bin, a tree), against their FP64 sum: rms relative error over 2000 columns.
SUMS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
#include "cv_rows.h"
int main(int argc, char **argv)
{
    const int G = atoi(argv[1]), R = atoi(argv[2]), T = atoi(argv[3]), M = 2000;
    std::mt19937 rng(1);
    std::uniform_real_distribution<float> uni(0.0f, 1.0f);
    double sq = 0.0;
    for (int m = 0; m < M; ++m) {
        std::vector<float> v(G);
        double exact = 0.0;
        for (float &x : v) exact += x = uni(rng);
        std::vector<float> s(R < T ? T : R, 0.0f), n(s.size(), 0.0f);
        for (int b = 0; b < G; ++b) cv::row_add(s[b % R], n[b % R], v[b]);
        for (int g = T; g < R; ++g) cv::pair_add(s[g % T], n[g % T], s[g], n[g]);
        for (int o = 1; o < T; o <<= 1)
            for (int j = 0; j < T; j += 2 * o) cv::pair_add(s[j], n[j], s[j + o], n[j + o]);
        const double e = ((double)s[0] + (double)n[0]) / exact - 1.0;
        sq += e * e;
    }
    printf("%.3e\n", std::sqrt(sq / M));
    return 0;
}
"""


# 2^-25 (a row's dropped rounding) over sqrt(rows) is 1.4e-9 of 456 rows, 2.4e-9 of
# 152 and 5.3e-9 of 32; sequential Kahan sums gave 3.8e-9, 5.2e-9 and 7.4e-9.
@pytest.mark.parametrize("rows,groups,threads,bound", [
    (456, 32, 32, 1.0e-9), (152, 32, 32, 1.7e-9),   # a standalone pass's bins
    (456, 16, 4, 3.8e-9), (152, 16, 4, 5.2e-9),     # one integral's refinement, 128 bins
    (32, 16, 4, 7.4e-9),                            # a batch item's, 64 bins
])
def test_row_sums_keep_their_compensation(tmp_path, rows, groups, threads, bound):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "sums.cpp", tmp_path / "sums"
    src.write_text(SUMS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe), str(rows), str(groups), str(threads)], capture_output=True, text=True, check=True)
    assert float(res.stdout) <= bound
