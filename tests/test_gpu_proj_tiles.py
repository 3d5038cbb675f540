"""The moved scans' kernels over more tiles than one launch has blocks (1216 of
256 voxels), on odd and unequal sizes, and on thin grids, whose tiles take
other shapes, against the oracle.  Dyadic affines, bounds as in the projected
voxel pass's parity test."""
import numpy as np
import pytest

import oracle as orc
from cases import assert_close_scaled, moved_dataset, to_dev, to_np

pytestmark = pytest.mark.gpu

TURN = [[0.9375, -0.25, 0.0], [0.25, 0.9375, 0.0], [0.0, 0.0, 1.0]]     # in the x, y plane
TILT = [[1.0, 0.0, 0.0], [0.0, 0.9375, -0.25], [0.0, 0.25, 0.9375]]     # in the y, z plane


def _aff(lin, t):
    A = np.eye(4)
    A[:3, :3] = lin
    A[:3, 3] = t
    return A


@pytest.mark.parametrize("recon,grids,affines", [
    ((97, 83, 61), ((95, 84, 59), (97, 83, 61)), (_aff(TURN, (9.5, -8.25, 1.375)), _aff(TILT, (0.5, 7.75, -9.25)))),
    ((67, 45, 1), ((67, 45, 1), (70, 41, 1)), (_aff(np.eye(3), (0, 0, 0)), _aff(TURN, (5.5, -6.25, 0)))),
    ((1, 45, 38), ((1, 45, 38), (1, 44, 40)), (_aff(np.eye(3), (0, 0, 0)), _aff(TILT, (0, 4.75, -5.25)))),
    ((3, 50, 21), ((2, 51, 23), (5, 50, 19)), (_aff(TILT, (0.5, 3.5, -5.5)), _aff(np.eye(3), (-1, 0, 1)))),
    ((150, 2, 2), ((151, 2, 3), (2, 2, 2)), (_aff(np.eye(3), (-0.5, 0.25, -0.125)), _aff(np.eye(3), (7, 0, 0)))),
])
def test_projected_voxel_pass(recon, grids, affines):
    import paper_2102_01604_gb300 as mpm
    d = moved_dataset(recon, list(grids), list(affines), seed=17, contrasts=("PDw", "MTw"), n_echoes=(3, 2))
    pg, po = mpm.make_problem(d["prot"], recon), orc.make_problem(d["prot"], recon)
    qg, qo = (m.make_projection(d["grids"], d["affines"]) for m in (mpm, orc))
    rng = np.random.default_rng(18)
    y = (d["y_true"] + 0.05 * rng.standard_normal(d["y_true"].shape)).astype(np.float32)
    nll_o, g_o, h_o = orc.grad_hess_proj(po, qo, d["xs"], y.astype(np.float64), d["b1ps"], d["b1ms"])
    g, h, nll = mpm.mpm_grad_hess_proj(pg, qg, [to_dev(x) for x in d["xs"]], to_dev(y),
                                       [to_dev(b) for b in d["b1ps"]], [to_dev(b) for b in d["b1ms"]])
    assert abs(float(nll) - nll_o) <= 1e-5 * nll_o
    assert_close_scaled(to_np(g), g_o, 1e-4, "g")
    assert_close_scaled(to_np(h), h_o, 1e-4, "h")
