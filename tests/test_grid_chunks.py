"""The z split of the staged JTV kernel's grid: as tma_chunks', but never more
blocks than the reduction has partials for (32768), whatever the volume."""
import ctypes
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2102_01604_gb300", "csrc")

HARNESS = """
#include "host_logic.h"
extern "C" int plain(long long t, int nz, long long w) { return mpm::tma_chunks(t, nz, w); }
extern "C" int capped(long long t, int nz, long long w, long long m) { return mpm::grid_chunks(t, nz, w, m); }
"""
MOST = 32768


def test_blocks_stay_within_the_partials(tmp_path):
    src = tmp_path / "chunks.cpp"
    src.write_text(HARNESS)
    so = str(tmp_path / "chunks.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src),
                    "-o", so], check=True)
    h = ctypes.CDLL(so)
    LL = ctypes.c_longlong
    h.plain.argtypes = [LL, ctypes.c_int, LL]
    h.capped.argtypes = [LL, ctypes.c_int, LL, LL]
    assert 3364 * h.plain(3364, 1221, 304) > MOST
    rng = random.Random(1)
    cases = [(3364, 1221, 304), (8192, 1024, 152), (1, 1, 1), (8192, 1, 304)]
    cases += [(int(2 ** rng.uniform(0, 13)), int(2 ** rng.uniform(0, 12)), rng.choice((1, 76, 152, 304)))
              for _ in range(300)]
    for t, nz, w in cases:
        c, p = h.capped(t, nz, w, MOST), h.plain(t, nz, w)
        assert 1 <= c <= nz and t * c <= MOST, (t, nz, w)
        assert c == p or t * p > MOST, (t, nz, w)      # the same split wherever it fits
