"""Kernel attributes (the opt-in to more than 48 KB of dynamic shared memory)
hold for one device, so they are set once on each device of the process, not
once per process: a second GPU's first launch would otherwise be refused.  The
bookkeeping is csrc/host_logic.h's OncePerDevice, driven here with made-up
device numbers."""
import ctypes
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2102_01604_gb300", "csrc")

HARNESS = """
#include "host_logic.h"
static mpm::OncePerDevice once;
static int calls;
extern "C" int visit(int dev, int error) { return once.run(dev, [&] { ++calls; return error; }); }
extern "C" int count() { return calls; }
"""


def test_once_per_device(tmp_path):
    src = tmp_path / "once.cpp"
    src.write_text(HARNESS)
    so = str(tmp_path / "once.so")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", so],
                   check=True)
    h = ctypes.CDLL(so)
    assert h.visit(0, 7) == 7 and h.count() == 1          # failed: tried again
    assert h.visit(0, 0) == 0 and h.count() == 2
    assert h.visit(0, 7) == 0 and h.count() == 2          # done there
    assert h.visit(1, 0) == 0 and h.count() == 3          # another device
    assert h.visit(63, 0) == 0 and h.visit(63, 0) == 0 and h.count() == 4
    assert h.visit(64, 0) == 0 and h.visit(64, 0) == 0 and h.count() == 6   # beyond the record: every time


def test_no_opt_in_is_kept_per_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        assert not re.search(r"static bool (attr|done)\b", open(path).read()), path
