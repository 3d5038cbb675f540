"""The multigrid solve over more tiles than one launch has blocks (1216 of 256
voxels), on odd and unequal sizes, on thin volumes, whose tiles take other
shapes (pairs along fewer axes in the restriction), and with one level in each
of its forms (up to 512 voxels, up to 8192, larger), against the oracle at the
bounds of the multigrid parity tests."""
import numpy as np
import pytest

import oracle as orc
from cases import assert_close_scaled, dataset, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,levels,nu,cg,contrasts", [
    ((97, 83, 61), 8, 1, 4, ("PDw", "MTw")),
    ((97, 83, 61), 3, 2, 2, ("PDw", "T1w")),
    ((67, 45, 1), 8, 1, 6, ("PDw", "MTw")),
    ((1, 45, 38), 8, 1, 6, ("PDw", "MTw")),
    ((3, 50, 21), 8, 2, 5, ("PDw", "MTw")),
    ((50, 1, 30), 8, 1, 5, ("PDw", "T1w")),
    ((600, 2, 2), 8, 1, 5, ("PDw", "MTw")),
    ((1, 1, 900), 8, 1, 5, ("PDw", "MTw")),
    ((9, 8, 7), 1, 1, 6, ("PDw", "MTw")),          # one level, 504 voxels
    ((13, 12, 9), 1, 1, 6, ("PDw", "T1w")),        # 1404
    ((31, 22, 15), 1, 1, 6, ("PDw", "MTw")),       # 10230: a launch per sweep
])
def test_mg_solve(shape, levels, nu, cg, contrasts):
    import paper_2102_01604_gb300 as mpm
    d = dataset(shape, seed=19, contrasts=contrasts, n_echoes=(3, 3))
    pg, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    rng = np.random.default_rng(20)
    y = (d["y_true"] + 0.05 * rng.standard_normal(d["y_true"].shape)).astype(np.float32)
    _, g, h = orc.grad_hess(po, d["x"], y, d["b1p"], d["b1m"])
    _, w = orc.jtv(po, y)
    h, w, g = h.astype(np.float32), w.astype(np.float32), g.astype(np.float32)
    kw = dict(mg_levels=levels, mg_nu=nu, mg_omega=0.7, mg_coarse_sweeps=20)
    delta, resid = mpm.mpm_solve(pg, mpm.make_opts(cg_iters=cg, **kw), to_dev(h), to_dev(w), to_dev(g), to_dev(y))
    d_o, it, r_o = orc.mg_solve(po, h, w, g, y, cg, orc.make_mg(levels, nu, 0.7, 20))
    assert it == cg
    assert_close_scaled(to_np(delta), d_o, 2e-4, "delta")
    np.testing.assert_allclose(to_np(resid)[:it + 1], r_o, rtol=2e-4 * cg ** 0.5 + 1e-5, atol=1e-6 * r_o[0])
