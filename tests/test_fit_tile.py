"""The tile shapes of thin volumes (csrc/host_logic.h, fit_tile): always one
thread per voxel of a block of 256, the wanted shape where the volume is as
large, and no axis padded beyond its size while another could take the
lanes."""
import ctypes
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2102_01604_gb300", "csrc")

HARNESS = """
#include "host_logic.h"
extern "C" void fit(const int* n, int* l)
{
    const int m[3] = {n[0], n[1], n[2]};
    int k[3] = {l[0], l[1], l[2]};
    mpm::fit_tile(m, k);
    for (int d = 0; d < 3; ++d) l[d] = k[d];
}
"""


def test_fit_tile(tmp_path):
    src = tmp_path / "tile.cpp"
    src.write_text(HARNESS)
    so = str(tmp_path / "tile.so")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so],
                   check=True)
    h = ctypes.CDLL(so)
    A = ctypes.c_int * 3

    def fit(n, want):
        l = A(*want)
        h.fit(A(*n), l)
        return tuple(l)

    assert fit((512, 512, 1), (3, 2, 3)) == (4, 4, 0)
    assert fit((1, 256, 256), (3, 2, 3)) == (0, 4, 4)
    assert fit((8, 512, 512), (5, 2, 1)) == (3, 3, 2)
    assert fit((5, 512, 512), (3, 2, 3)) == (3, 2, 3)
    rng = random.Random(2)
    for _ in range(2000):
        want = rng.choice(((3, 2, 3), (5, 2, 1)))
        n = tuple(int(2 ** rng.uniform(0, 10)) for _ in range(3))
        l = fit(n, want)
        assert sum(l) == 8
        if all(v > 1 << (w - 1) for v, w in zip(n, want)):
            assert l == want, (n, l)
        covered = [1 << k >= v for k, v in zip(l, n)]
        for d in range(3):        # an axis runs over its end by less than a factor of two
            assert (1 << l[d]) < 2 * n[d] or all(covered), (n, l)
