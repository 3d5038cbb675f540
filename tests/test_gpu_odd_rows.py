"""The staged PCG iteration on volumes whose x size is not a multiple of 4 (w
and H copied with padded rows by the PCG start): every residue, the smallest
volumes each tile shape takes and one voxel less (the plain iteration), three
and four maps, against the oracle at the bounds of the solve's parity tests."""
import numpy as np
import pytest

import oracle as orc
from cases import assert_close_scaled, dataset, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,contrasts", [
    ((41, 11, 6), ("PDw", "T1w", "MTw")),
    ((42, 21, 5), ("PDw", "T1w")),
    ((75, 34, 7), ("PDw", "T1w", "MTw")),
    ((25, 18, 9), ("PDw", "T1w", "MTw")),      # 16 x 16 tiles' smallest
    ((25, 17, 9), ("PDw", "T1w")),             # plain
    ((41, 9, 4), ("PDw", "T1w", "MTw")),       # plain
    ((131, 19, 1), ("PDw", "T1w", "MTw")),
])
def test_solve_odd_rows(shape, contrasts):
    import paper_2102_01604_gb300 as mpm
    d = dataset(shape, seed=21, contrasts=contrasts, n_echoes=(4,) * len(contrasts))
    pg, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    rng = np.random.default_rng(22)
    y = (d["y_true"] + 0.05 * rng.standard_normal(d["y_true"].shape)).astype(np.float32)
    _, g, h = orc.grad_hess(po, d["x"], y, d["b1p"], d["b1m"])
    _, w = orc.jtv(po, y)
    h, w, g = h.astype(np.float32), w.astype(np.float32), g.astype(np.float32)
    delta, resid = mpm.mpm_solve(pg, mpm.make_opts(cg_iters=30), to_dev(h), to_dev(w), to_dev(g), to_dev(y))
    d_o, _, r_o = orc.solve(po, h, w, g, y, 30)
    assert_close_scaled(to_np(delta), d_o, 2e-4, "delta")
    np.testing.assert_allclose(to_np(resid), r_o, rtol=2e-4, atol=1e-6 * r_o[0])
