"""CPU check of the flux-register indexing of the conservative fix, up to the
largest forest a GPU can hold."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_face_entries_of_the_largest_forests(tmp_path):
    """face_entry compiled for the host, at entries on both sides of 2^31: 2.4
    billion entries are 300 million patches of two cells (270 GB)."""
    if shutil.which("g++") is None:
        pytest.skip("needs g++")
    (tmp_path / "f.cpp").write_text(r"""
#include <cstdio>
#include <cstdlib>
#include "af_internal.h"
int main(int argc, char **argv) {
    int p, side, k;
    for (int a = 1; a + 1 < argc; a += 2) {
        af::face_entry(atoll(argv[a]), atoi(argv[a + 1]), p, side, k);
        printf("%d %d %d\n", p, side, k);
    }
}
""")
    exe = str(tmp_path / "f")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2205_07572_gb300", "csrc"), str(tmp_path / "f.cpp"), "-o", exe], check=True)
    at = [(t, n) for n in (2, 3, 16, 64) for t in (0, 1, 4 * n - 1, 4 * n, 2 ** 31 - 1, 2 ** 31, 2 ** 31 + 5, 2_400_000_001)]
    out = subprocess.run([exe] + [str(v) for e in at for v in e], check=True, capture_output=True, text=True).stdout
    got = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert got == [(t // (4 * n), t // n % 4, t % n) for t, n in at]
