"""Stiff Newton systems (lambda = 1e5 on flat maps: directions hundreds of
times longer than the preconditioned residual), solved to convergence.  The
iteration forms z from the last two directions only while |p| <= 8 |z| in the
norm of M (pcg_step.cuh), so each of J iterations rounds z to within 8 * 2^-24
of its size, and J independent roundings stay within 8 * 2^-24 sqrt(J).  A z
that is always formed from p ends 1e-4 off here, one that is always stored
1e-6 to 3e-6."""
import numpy as np
import pytest

import oracle as orc
from cases import dataset, to_dev, to_np

pytestmark = pytest.mark.gpu

ITERS = 700
BOUND = 8 * 2.0 ** -24 * ITERS ** 0.5


def _flat(d):
    return np.repeat(d["y_true"].mean(axis=1, keepdims=True), d["y_true"].shape[1], 1).astype(np.float32)


@pytest.mark.parametrize("shape,contrasts", [
    ((28, 18, 10), ("PDw", "T1w", "MTw")),     # 16 x 16 tiles
    ((44, 12, 8), ("PDw", "T1w")),             # 32 x 8 tiles, three maps
    ((41, 11, 6), ("PDw", "T1w", "MTw")),      # padded rows
    ((20, 16, 12), ("PDw", "T1w", "MTw")),     # the plain iteration
    ((24, 18, 1), ("PDw", "T1w", "MTw")),      # at most 512 voxels: z[1] among the partials
])
def test_stiff_solve(shape, contrasts):
    import torch
    import paper_2102_01604_gb300 as mpm
    d = dataset(shape, seed=3, contrasts=contrasts, n_echoes=(6,) * len(contrasts))
    pg, po = (m.make_problem(d["prot"], shape, lam=1e5) for m in (mpm, orc))
    y = _flat(d)
    _, g, h = orc.grad_hess(po, d["x"], y, d["b1p"], d["b1m"])
    _, w = orc.jtv(po, y)
    h, w, g = h.astype(np.float32), w.astype(np.float32), g.astype(np.float32)
    opts = mpm.make_opts(cg_iters=ITERS)
    ws = mpm.workspace(pg, opts, mpm._lib.CALL_SOLVE)
    ws[:ws.numel() // 4 * 4].view(torch.float32).fill_(float("nan"))
    ws[:4096].zero_()                           # the header: counters are zero between calls
    delta, resid = mpm.mpm_solve(pg, opts, to_dev(h), to_dev(w), to_dev(g), to_dev(y), ws=ws)
    d_o, _, _ = orc.solve(po, h, w, g, y, 3000)
    err = np.linalg.norm(to_np(delta) - d_o) / np.linalg.norm(d_o)
    assert err <= BOUND, err


def test_stiff_update_in_a_group():
    """The same in one launch for two subjects: one update of each against its
    own solo update, each within the bound of the exact one."""
    import torch
    import paper_2102_01604_gb300 as mpm
    opts = mpm.make_opts(gn_iters=1, cg_iters=ITERS, init=False, graph="phased")
    subs = []
    for shape, seed in (((28, 18, 10), 3), ((32, 20, 7), 4)):
        d = dataset(shape, seed=seed, n_echoes=(6, 6, 6))
        subs.append((d, mpm.make_problem(d["prot"], shape, lam=1e5), to_dev(_flat(d))))
    ys = [y.clone() for _, _, y in subs]
    mpm.mpm_fit_batch([p for _, p, _ in subs], opts, [to_dev(d["x"]) for d, _, _ in subs], ys,
                      b1ps=[to_dev(d["b1p"]) for d, _, _ in subs],
                      b1ms=[to_dev(d["b1m"]) for d, _, _ in subs])
    for (d, p, y0), yb in zip(subs, ys):
        y = y0.clone()
        mpm.mpm_fit(p, mpm.make_opts(gn_iters=1, cg_iters=ITERS, init=False), to_dev(d["x"]), y,
                    to_dev(d["b1p"]), to_dev(d["b1m"]))
        step = to_np(y) - to_np(y0)
        assert np.linalg.norm(to_np(yb) - to_np(y)) <= (2 * BOUND + 2.0 ** -23) * np.linalg.norm(step) \
            + 2.0 ** -23 * np.linalg.norm(to_np(y))
