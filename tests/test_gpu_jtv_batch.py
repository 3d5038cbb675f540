"""The JTV pass of phase-batched fits at sizes where the group takes the staged
kernel: runs of four for 16-byte rows (from 2^17 voxels), single voxels where
one subject's maps lie off the boundary (the group from 2^20), the tile kernel
where a group of the latter kind has a smaller subject.  The objective of one
update's two evaluations and the maps after it against each subject's own fit
(the reductions run over other blocks: 1e-6 relative, and 1e-5 in the maps
after 3 PCG iterations), and the first objective's prior against the
oracle's (a compensated sum: 2e-6)."""
import numpy as np
import pytest

import oracle as orc
from cases import dataset, to_dev, to_np

pytestmark = pytest.mark.gpu

SMALL, LARGE = (64, 64, 33), (128, 96, 86)      # 1.03 x 2^17 and 1.01 x 2^20 voxels


@pytest.mark.parametrize("shapes,offsets", [
    ((SMALL, SMALL), (0, 0)),          # staged, runs of four
    ((SMALL, SMALL), (0, 1)),          # tile kernel
    ((LARGE, LARGE), (3, 0)),          # staged, single voxels
    ((LARGE, SMALL), (1, 0)),          # tile kernel: one subject too small for single voxels
])
def test_group_matches_solo(shapes, offsets):
    import torch
    import paper_2102_01604_gb300 as mpm
    subs, keep = [], []
    rng = np.random.default_rng(4)
    d = dataset((4, 4, 4), seed=11, n_echoes=(2, 2, 2))
    for shape, off in zip(shapes, offsets):
        N = int(np.prod(shape))
        y0 = np.repeat(d["y_true"].mean(axis=1, keepdims=True), N, 1) + 0.05 * rng.standard_normal((4, N))
        y0 = y0.astype(np.float32)
        x = torch.rand((6, N), device="cuda") * 100.0 + 400.0
        subs.append((mpm.make_problem(d["prot"], shape), orc.make_problem(d["prot"], shape), x, y0, off))

    def maps(y0, off):
        buf = torch.full((y0.size + 8,), float("nan"), device="cuda")
        v = buf[off:off + y0.size].view(y0.shape)
        v.copy_(to_dev(y0))
        keep.append(buf)
        return v

    opts = dict(gn_iters=1, cg_iters=3, init=False)
    ys = [maps(y0, off) for _, _, _, y0, off in subs]
    _, reps = mpm.mpm_fit_batch([p for p, *_ in subs], mpm.make_opts(graph="phased", **opts),
                                [x for _, _, x, _, _ in subs], ys)
    for (p, po, x, y0, off), yb, rb in zip(subs, ys, reps):
        ysolo = maps(y0, off)
        _, rep = mpm.mpm_fit(p, mpm.make_opts(**opts), x, ysolo)
        np.testing.assert_allclose(np.array(rb.F[:2]), np.array(rep.F[:2]), rtol=1e-6)
        np.testing.assert_allclose(to_np(yb), to_np(ysolo), rtol=1e-5, atol=1e-5)
        e_o, _ = orc.jtv(po, y0)
        assert abs(rb.jtv[0] - e_o) <= 2e-6 * e_o
    for buf, off, n in zip(keep, offsets, [s[3].size for s in subs]):
        assert torch.isnan(buf[:off]).all() and torch.isnan(buf[off + n:]).all()
