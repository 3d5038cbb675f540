"""Which kernel a call takes, seen from outside: with the copies of the staged
kernels withheld (mpm_test_copy_timeout, waits of 1 ms), a staged pass reports
the timeout and a plain one runs as ever."""
import contextlib

import numpy as np
import pytest

import oracle as orc
from cases import assert_close_scaled, dataset, map_error, to_dev, to_np

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def withheld(mpm):
    mpm.mpm_test_copy_timeout(True, 1000.0)
    try:
        yield
    finally:
        mpm.mpm_test_copy_timeout(False, 0.0)


def _staged(mpm, ws):
    st = mpm.mpm_workspace_status(ws)
    assert st in (mpm._lib.OK, mpm._lib.ERR_NUMERIC)
    return st != mpm._lib.OK


def _nan_ws(mpm, problem, opts, call):
    import torch
    ws = mpm.workspace(problem, opts, call)
    ws[:ws.numel() // 4 * 4].view(torch.float32).fill_(float("nan"))
    ws[:4096].zero_()                           # the header: counters are zero between calls
    return ws


@pytest.mark.parametrize("shape,contrasts,staged", [
    ((40, 10, 5), ("PDw", "T1w", "MTw"), True),
    ((41, 11, 6), ("PDw", "T1w", "MTw"), True),
    ((42, 21, 5), ("PDw", "T1w"), True),
    ((75, 34, 7), ("PDw", "T1w", "MTw"), True),
    ((25, 18, 9), ("PDw", "T1w", "MTw"), True),
    ((25, 17, 9), ("PDw", "T1w"), False),
    ((41, 9, 4), ("PDw", "T1w", "MTw"), False),
    ((23, 18, 9), ("PDw", "T1w", "MTw"), False),
    ((131, 19, 1), ("PDw", "T1w", "MTw"), True),
])
def test_solve_route(shape, contrasts, staged):
    """The iteration's route with the full workspace (filled with NaN: nothing
    in it may be read before it is written), and the plain one where an odd
    volume's workspace lacks room for the padded copies."""
    import paper_2102_01604_gb300 as mpm
    d = dataset(shape, seed=21, contrasts=contrasts, n_echoes=(4,) * len(contrasts))
    pg, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    y = d["y_true"].astype(np.float32)
    _, g, h = orc.grad_hess(po, d["x"], y, d["b1p"], d["b1m"])
    _, w = orc.jtv(po, y)
    h, w, g = h.astype(np.float32), w.astype(np.float32), g.astype(np.float32)
    args = [to_dev(a) for a in (h, w, g, y)]
    opts = mpm.make_opts(cg_iters=12)
    d_o, _, _ = orc.solve(po, h, w, g, y, 12)
    ws = _nan_ws(mpm, pg, opts, mpm._lib.CALL_SOLVE)
    delta, _ = mpm.mpm_solve(pg, opts, *args, ws=ws)
    assert not _staged(mpm, ws)                 # status OK
    assert_close_scaled(to_np(delta), d_o, 2e-4, "delta")
    with withheld(mpm):
        mpm.mpm_solve(pg, opts, *args, ws=ws)
        assert _staged(mpm, ws) == staged
    if shape[0] % 4:
        small = _nan_ws(mpm, pg, opts, mpm._lib.CALL_SOLVE)[:-1]
        with withheld(mpm):
            delta, _ = mpm.mpm_solve(pg, opts, *args, ws=small)
            assert not _staged(mpm, small)
        assert_close_scaled(to_np(delta), d_o, 2e-4, "delta without padded rows")


def test_fit_without_padded_rows_matches_the_oracle():
    import torch
    import paper_2102_01604_gb300 as mpm
    shape = (41, 11, 6)
    d = dataset(shape, seed=23)
    pg, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    opts = mpm.make_opts(gn_iters=4, cg_iters=30)
    ref = orc.fit(po, d["x"], None, d["b1p"], d["b1m"], gn_iters=4, cg_iters=30)
    for cut in (0, 1):
        ws = _nan_ws(mpm, pg, opts, mpm._lib.CALL_FIT)
        y = torch.zeros((pg.n_maps, int(np.prod(shape))), device="cuda")
        _, rep = mpm.mpm_fit(pg, opts, to_dev(d["x"]), y, to_dev(d["b1p"]), to_dev(d["b1m"]),
                             ws=ws[:ws.numel() - cut])
        np.testing.assert_allclose(np.array(rep.F[:5]), ref["F"], rtol=1e-5)
        assert map_error(to_np(y), ref["y"]).max() <= 1e-3


@pytest.mark.parametrize("shape,offset,staged", [
    ((64, 64, 33), 0, True),
    ((60, 47, 49), 0, True),
    ((64, 64, 31), 0, False),           # below 2^17 voxels
    ((64, 64, 33), 1, False),
    ((128, 96, 86), 3, True),
    ((129, 95, 87), 0, True),
    ((129, 95, 87), 2, True),
    ((129, 95, 85), 0, False),          # below 2^20
    ((3, 5, 70001), 1, False),          # planes of one tile
    ((8, 8, 4096), 0, False),
    ((16, 16, 4096), 0, True),          # two, and not longer than 2^20 voxels
    ((16, 16, 4097), 0, False),
    ((16, 20, 4097), 0, True),          # three
    ((15, 17, 4200), 0, True),
    ((13, 15, 5500), 0, False),
    ((1500, 7, 101), 0, True),
    ((1828, 3, 200), 0, True),          # the widest row of its kind
    ((1832, 3, 200), 0, False),
])
def test_jtv_route(shape, offset, staged):
    import torch
    import paper_2102_01604_gb300 as mpm
    d = dataset((4, 4, 4), seed=11)
    p = mpm.make_problem(d["prot"], shape)
    N = int(np.prod(shape))
    y = torch.zeros(4 * N + 8, device="cuda")[offset:offset + 4 * N].view(4, N)
    ws = mpm.workspace(p, None, mpm._lib.CALL_JTV)
    with withheld(mpm):
        mpm.mpm_jtv_weights(p, y, w=torch.zeros(N + 8, device="cuda")[offset:offset + N], ws=ws)
        assert _staged(mpm, ws) == staged
