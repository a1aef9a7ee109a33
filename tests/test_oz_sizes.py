"""The scratch planned for an exact-slicing product of K terms holds every product of fewer terms (a ragged last row block
of the adjoint has fewer, in other slabs)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_07731_gb300", "csrc")
MAIN = r"""
#include <stdio.h>
#include "oz_sizes.cuh"
int main()
{
    size_t last[4] = {0, 0, 0, 0}, s[4];
    for (int K = 1; K <= 200000; K += K < 30000 ? 1 : 7) {
        oz_sizes(320, 48, K, 1, &s[0], &s[1], &s[2], &s[3]);
        const long slab = oz_slab(K), kp = (2 * slab + 63) / 64 * 64, parts = (slab + 255) / 256;
        if (slab > 7168 || (slab < K && slab % 32) || s[0] < 7ul * 384 * kp || s[1] < 7ul * 128 * kp || s[2] < 320ul * (1 + parts) ||
            s[3] < 48ul * (1 + parts))
            return printf("K %d: slab %ld does not fit\n", K, slab), 1;
        for (int i = 0; i < 4; ++i) {
            if (s[i] < last[i]) return printf("K %d: size %d shrinks\n", K, i), 1;
            last[i] = s[i];
        }
    }
    return 0;
}
"""


def test_sizes_grow_with_k(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "m.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(tmp_path / "m.cpp"), "-o", str(tmp_path / "m")], check=True)
    r = subprocess.run([str(tmp_path / "m")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
