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


def _least(mpm, pg, opts, call):
    """Smallest workspace of a call without room for the padded rows: the padded
    rows are the last part of the solve's region and only they depend on nx % 4."""
    import torch
    lo, hi = 0, mpm.mpm_workspace_size(pg, opts, mpm._lib.CALL_SOLVE)
    full = hi
    N = pg.nx * pg.ny * pg.nz
    z = torch.zeros((10, N), device="cuda")
    h = z.clone()
    h[:pg.n_maps] = 1.0
    w = torch.ones(N, device="cuda")
    ws = torch.empty(hi, dtype=torch.uint8, device="cuda")
    one = mpm.make_opts(cg_iters=1)
    while hi - lo > 1:
        mid = (lo + hi) // 2
        try:
            mpm.mpm_solve(pg, one, h[:pg.n_maps * (pg.n_maps + 1) // 2].contiguous(), w,
                          z[:pg.n_maps].contiguous(), z[:pg.n_maps].contiguous(), ws=ws[:mid])
            hi = mid
        except mpm.MPMError as e:
            assert e.status == mpm._lib.ERR_WORKSPACE_TOO_SMALL
            lo = mid
    return mpm.mpm_workspace_size(pg, opts, call) - (full - hi)


def test_odd_rows_without_room_for_the_copies():
    """A workspace or arena that holds everything but the padded copies still
    solves, fits and serves (the plain iteration); one byte less is refused."""
    import torch
    import paper_2102_01604_gb300 as mpm
    shape = (41, 11, 6)
    d = dataset(shape, seed=23)
    pg, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    opts = mpm.make_opts(gn_iters=3, cg_iters=12)
    sizes = {c: (_least(mpm, pg, opts, c), mpm.mpm_workspace_size(pg, opts, c))
             for c in (mpm._lib.CALL_SOLVE, mpm._lib.CALL_FIT)}
    assert all(least < full for least, full in sizes.values())

    def buf(n):
        return torch.empty(n, dtype=torch.uint8, device="cuda")

    _, g, h = orc.grad_hess(po, d["x"], d["y_true"].astype(np.float32), d["b1p"], d["b1m"])
    _, w = orc.jtv(po, d["y_true"].astype(np.float32))
    h, w, g = h.astype(np.float32), w.astype(np.float32), g.astype(np.float32)
    y = d["y_true"].astype(np.float32)
    args = [to_dev(a) for a in (h, w, g, y)]
    n = sizes[mpm._lib.CALL_SOLVE][0]
    delta, _ = mpm.mpm_solve(pg, opts, *args, ws=buf(n))
    d_o, _, _ = orc.solve(po, h, w, g, y, 12)
    assert_close_scaled(to_np(delta), d_o, 2e-4, "delta")
    with pytest.raises(mpm.MPMError):
        mpm.mpm_solve(pg, opts, *args, ws=buf(n - 1))

    n = sizes[mpm._lib.CALL_FIT][0]
    x, b1p, b1m = (to_dev(d[k]) for k in ("x", "b1p", "b1m"))
    y_fit, y_srv = (torch.zeros((pg.n_maps, d["y_true"].shape[1]), device="cuda") for _ in range(2))
    mpm.mpm_fit(pg, opts, x, y_fit, b1p, b1m, ws=buf(n))
    srv = mpm.Server(buf(n), max_slots=1)
    t = srv.submit(pg, opts, x, y_srv, b1p, b1m)
    while srv.poll(t)[0] < mpm._lib.REQ_DONE:
        srv.step()
    srv.close()
    assert torch.equal(y_fit, y_srv)
