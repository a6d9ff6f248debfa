"""CPU checks of the rules that decide how a step is launched: few tiles shared
among the idle SMs, and which grids are chained."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def few(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    d = tmp_path_factory.mktemp("few_tiles")
    (d / "f.cpp").write_text(r"""
#include <cstdio>
#include <cstdlib>
#include "af_internal.h"
int main(int argc, char **argv) {
    int a[6];
    for (int i = 1; i + 5 < argc; i += 6) {
        for (int k = 0; k < 6; ++k) a[k] = atoi(argv[i + k]);
        printf("%d\n", af::few_tiles(a[0], a[1], af::tiling(a[2]), a[3], a[4], a[5]));
    }
}
""")
    exe = str(d / "f")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2205_07572_gb300", "csrc"), str(d / "f.cpp"), "-o", exe], check=True)

    def run(args):
        out = subprocess.run([exe] + [str(int(v)) for a in args for v in a], check=True, capture_output=True, text=True)
        return [int(v) for v in out.stdout.split()]
    return run


def test_bands_are_at_most_two_an_sm_of_two_rows_or_more(few):
    args = [(f64, ac, k, m, n, ad) for f64 in (0, 1) for ac in (0, 1) for k in range(10) for ad in (0, 1)
            for m in (1, 2, 37, 76, 77, 101, 102, 152, 153, 304, 10 ** 6) for n in (2, 3, 8, 16, 31, 64)]
    rows = [32, 16, 16, 8, 16, 8, 18, 10, 10, 18]
    for (f64, ac, k, m, n, ad), s in zip(args, few(args)):
        assert 1 <= s <= max(1, min(n + 2, rows[k]) // 2)
        assert s == 1 or m * s <= 304
        assert s == 1 or m <= 152


def test_tiles_that_bands_would_only_slow_down_stay_whole(few):
    """102 to 152 FP64 tiles took 10 to 45 % longer as two bands an SM, and so
    did the FP32 kernel that stages whole lattices in bulk."""
    for args in ([(1, ac, 0, m, n, 0) for ac in (0, 1) for m in (102, 128, 152) for n in (23, 32, 64)],
                 [(1, 1, 7, m, 16, 1) for m in (77, 100, 128, 152)], [(1, 1, 8, m, 8, ad) for m in (102, 152) for ad in (0, 1)],
                 [(0, 1, 6, m, 16, 1) for m in (77, 102, 128, 152)], [(0, 1, 0, m, 32, 0) for m in (102, 128, 152)]):
        assert few(args) == [1] * len(args), args
    # one 64 x 64 patch is four tiles: bands of two rows
    assert few([(1, 0, 0, 4, 64, 0)]) == [16]


def test_grids_that_a_chain_would_pile_up_are_not_chained(tmp_path):
    """(CTAs, resident CTAs an SM) that measured 10 to 50 % slower chained, and
    neighbours on either side that did not."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("needs nvcc")
    (tmp_path / "c.cu").write_text(r"""
#include <cstdio>
#include <cstdlib>
#include "af_launch.cuh"
int main(int argc, char **argv) {
    for (int i = 1; i + 1 < argc; i += 2) printf("%d\n", (int)af::chain_even(atoll(argv[i]), atoi(argv[i + 1])));
}
""")
    exe = str(tmp_path / "c")
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2205_07572_gb300", "csrc"), str(tmp_path / "c.cu"), "-o", exe], check=True)
    uneven = [(240, 3), (280, 3), (310, 4), (400, 4), (400, 5), (560, 5), (500, 6), (700, 6), (650, 8), (1000, 8), (760, 9)]
    even = [(1, 1), (152, 3), (228, 3), (310, 3), (304, 4), (500, 4), (350, 5), (650, 5), (456, 6), (800, 6), (608, 8),
            (1216, 8), (650, 9), (1, 2), (3000, 1), (10 ** 6, 12)]
    out = subprocess.run([exe] + [str(v) for e in uneven + even for v in e], check=True, capture_output=True, text=True)
    assert [int(v) for v in out.stdout.split()] == [0] * len(uneven) + [1] * len(even)
