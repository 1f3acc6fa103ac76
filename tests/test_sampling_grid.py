"""The rules of cv_grid.h, compiled for the host: blocks of a pass, tiles of a batch.

For every kind of pass and 152 SMs: at least one block, at most one wave, never
fewer for more points; and where a point costs a warp's time rather than the
SM's (pseudo-random points, a shared histogram copy, delay chains) two blocks
per SM as early as the measurements ask for, so that no such pass leaves its
warps more blocks than the rule of sixteen per warp and two below it did.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1408_6373_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "cv_grid.h"
using namespace cv;
static int bad = 0;
static void check(bool ok, const char *what, long long n, int g)
{
    if (!ok && bad++ < 20) printf("%s: n %lld, %d blocks\n", what, n, g);
}
// 32-point blocks of a warp
static long long per_warp(long long n, int g) { return ((n + 63) / 32 + 8ll * g - 1) / (8ll * g); }
int main()
{
    const int sms = 152;
    for (int occ = 1; occ <= 4; ++occ)
        for (int b = 0; b < 8; ++b)
            for (long long chain : {0ll, 299ll, 300ll, 999ll, 1000ll, 1ll << 30}) {
                const PassKind k = {(b & 1) != 0, (b & 2) != 0, (b & 4) != 0, chain};
                int last = 0;
                for (long long n = 1; n < 20000000; n += 1 + n / 64) {
                    const int g = sampling_blocks(sms, occ, n, k);
                    check(g >= 1 && g <= sms * occ, "one wave", n, g);
                    check(g >= last, "monotone", n, g);
                    last = g;
                }
                check(last == sms * occ, "full wave", 20000000, last);
                check(sampling_blocks(sms, occ, 1ll << 52, k) == sms * occ, "full wave", 1ll << 52, 0);
            }
    const PassKind costly = {false, true, false, 0}, chain = {false, false, false, 1000};
    for (long long n = 30000; n < 20000000; n += 1 + n / 64) {
        const int g2 = sampling_blocks(sms, 2, n, costly), g3 = sampling_blocks(sms, 3, n, chain);
        check(g2 >= 2 * sms || per_warp(n, g2) <= 3, "pseudo-random, 9 dimensions on", n, g2);
        check(g3 >= 2 * sms || per_warp(n, g3) <= 3, "chain", n, g3);
        check(sampling_blocks(sms, 3, n, costly) >= 2 * sms || per_warp(n, sms) <= 6, "pseudo-random", n, 0);
        check(sampling_blocks(sms, 2, n, {false, false, true, 0}) >= 2 * sms || per_warp(n, sms) <= 8, "shared copy", n, 0);
    }
    return bad ? 1 : 0;
}
"""


def test_sampling_blocks(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "grid.cpp", tmp_path / "grid"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout


TILES = r"""
#include <initializer_list>
#include <cstdio>
#include "cv_grid.h"
int main()
{
    int bad = 0;
    for (int cap : {256, 1024, 2048, 4096})
        for (int split : {8, 16, 32})
            for (long long n = 1; n < (1ll << 45); n += 1 + n / 16) {
                const long long blocks = (n + 31) / 32 + 1, t = cv::tile_blocks_for(n, cap, split);
                const long long tiles = (blocks + t - 1) / t, most = (blocks + 2047) / 2048;
                const bool ok = t >= 64 && !(t & (t - 1)) && t <= (cap > 2048 ? cap : 2048) &&
                                tiles <= (most > 512 ? most : 512) && (blocks > 512 * (long long)cap || t <= cap);
                if (!ok && bad++ < 10) printf("n %lld cap %d split %d: tiles of %lld blocks\n", n, cap, split, t);
            }
    return bad ? 1 : 0;
}
"""


def test_tiles_leave_few_rows(tmp_path):
    # at most 512 rows an iteration, or those of tiles of 2^16 points
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "tiles.cpp", tmp_path / "tiles"
    src.write_text(TILES)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
