"""The staged JTV kernel at the edges of its dispatch, against the oracle:
volumes just large enough for it with and without 16-byte rows, arrays at every
4-byte offset from a 16-byte boundary (whose first and last granules it must
not read whole), planes smaller than a granule, rows that leave one block per
SM and rows too wide for it.  Bounds as in the parity tests: a weight is a
chain of about 30 float32 operations (1e-5 relative), the energy a compensated
sum of positive terms (2e-6)."""
import numpy as np
import pytest

import oracle as orc
from cases import dataset, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,offset", [
    ((64, 64, 33), 0),          # 16-byte rows: runs of four
    ((60, 47, 49), 0),          # the last block of a plane partly empty
    ((64, 64, 33), 1),          # too small for single voxels: the tile kernel
    ((128, 96, 86), 3),         # 16-byte rows, arrays off the boundary
    ((129, 95, 87), 0),
    ((129, 95, 87), 2),
    ((3, 5, 70001), 1),         # a plane of 15 voxels
    ((1500, 7, 101), 0),        # one block per SM
    ((2400, 3, 150), 0),        # rows too wide: the tile kernel
])
def test_jtv_staged(shape, offset):
    import torch

    import paper_2102_01604_gb300 as mpm
    vx = (0.8, 1.0, 1.25)
    d = dataset((4, 4, 4), seed=11)
    p, po = (m.make_problem(d["prot"], shape, vx=vx) for m in (mpm, orc))
    N = int(np.prod(shape))
    rng = np.random.default_rng(12)
    y = rng.standard_normal((4, N)).astype(np.float32)
    y *= np.where(rng.random(N) < 0.5, 1e-4, 1.0).astype(np.float32)   # flat and rough neighbourhoods
    buf = torch.full((4 * N + 8,), float("nan"), device="cuda")
    yd = buf[offset:offset + 4 * N].view(4, N)
    yd.copy_(to_dev(y))
    wbuf = torch.zeros(N + 8, device="cuda")
    w, e = mpm.mpm_jtv_weights(p, yd, w=wbuf[offset:offset + N])
    e_o, w_o = orc.jtv(po, y)
    np.testing.assert_allclose(to_np(w), w_o, rtol=1e-5)
    assert abs(e.item() - e_o) <= 2e-6 * e_o
    assert not wbuf[:offset].any() and not wbuf[offset + N:].any()


def test_jtv_staged_infinite_and_nan_maps():
    """A NaN or an infinity reaches the weights of its voxel and its
    neighbours only, on the staged kernel (2 x 2 x 2 of them at a corner)."""
    import torch

    import paper_2102_01604_gb300 as mpm
    shape = (64, 64, 33)
    nx, ny, nz = shape
    d = dataset((4, 4, 4), seed=11)
    p = mpm.make_problem(d["prot"], shape)
    for bad, centre in ((float("nan"), float("nan")), (float("inf"), 0.0)):
        y = torch.randn((4, nz, ny, nx), generator=torch.Generator().manual_seed(3))
        y[2, 0, 0, 0] = bad
        w, e = mpm.mpm_jtv_weights(p, y.cuda().view(4, -1))
        w = w.cpu().view(nz, ny, nx)
        near = [(0, 0, 0), (0, 0, 1), (0, 1, 0), (1, 0, 0)]
        for n in near:
            v = w[n].item()
            assert (np.isnan(v) if np.isnan(centre) else v == 0.0), n
        rest = w.clone()
        for n in near:
            rest[n] = 1.0
        assert torch.isfinite(rest).all() and (rest > 0).all()
        assert not np.isfinite(e.item())


@pytest.mark.parametrize("shape", [(64, 64, 33), (129, 95, 87)])
def test_jtv_staged_copy_timeout(shape):
    """Copies that never land (the test hook withholds them): the call returns,
    the workspace records the timeout, and the next call on the same context
    gives the weights again."""
    import torch

    import paper_2102_01604_gb300 as mpm
    from paper_2102_01604_gb300 import _lib
    p = mpm.make_problem(dataset((4, 4, 4), seed=11)["prot"], shape)
    y = torch.randn((4, int(np.prod(shape))), device="cuda")
    ws = mpm.workspace(p, None, _lib.CALL_JTV)
    w0, e0 = (t.clone() for t in mpm.mpm_jtv_weights(p, y, ws=ws))
    assert mpm.mpm_workspace_status(ws) == _lib.OK
    mpm.mpm_test_copy_timeout(True, 1000.0)
    try:
        mpm.mpm_jtv_weights(p, y, ws=ws)
        st = mpm.mpm_workspace_status(ws)
        msg = _lib.load().mpm_last_error().decode()
    finally:
        mpm.mpm_test_copy_timeout(False, 0.0)
    assert st == _lib.ERR_NUMERIC and "copy wait timed out" in msg
    w, e = mpm.mpm_jtv_weights(p, y, ws=ws)
    assert mpm.mpm_workspace_status(ws) == _lib.OK
    assert torch.equal(w, w0) and torch.equal(e, e0)
