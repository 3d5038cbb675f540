"""The float32 uncertainty pass's distance from 64 bits, per output, on the
seeded 64^3 volume of the speed cases.  The bits are the same on every run, so
the bounds lie just above what the pass gives: rounding the equilibrated
diagonal by itself (one rounding more) puts map 3's variance at 1.18e-7, eight
logarithms summed put the determinant at 3.80e-8."""
import importlib.util
import os

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_error_against_64_bits():
    spec = importlib.util.spec_from_file_location("speed_cases", os.path.join(ROOT, "perf", "cases.py"))
    cases = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(cases)
    case = next(c for c in cases.listed() if c["kind"] == "uncertainty")
    case = {**case, "nx": 64, "ny": 64, "nz": 64}
    got, ref = cases.run(cases.prepare(case, 3)), cases.exact(case, 3)

    def err(a, b):
        return ((a.double() - b).norm() / b.norm()).item()

    for k, bound in enumerate((2.75e-7, 2.0e-7, 1.45e-7, 1.165e-7)):
        assert err(got["var"][k], ref["var"][k]) <= bound, k
    assert err(got["logdet"], ref["logdet"]) <= 3.5e-8
    assert err(got["moments"], ref["moments"]) <= 4.0e-8
