"""The push's search for the points that pull a voxel, on the affines where it
takes another way: shifts by whole voxels (in and out of the grid), the same
shift made of fractions, axes swapped and mirrored (lines that do not run along
x), acquisition grids finer and coarser than the reconstruction, a volume one
voxel thick.  The push must be the pull's exact adjoint (float32 sums of the
same products: 1e-5 of the sum of their magnitudes) and agree with the
oracle's."""
import numpy as np
import pytest

import oracle as orc
from cases import dataset, to_dev, to_np

pytestmark = pytest.mark.gpu

I3 = np.eye(3)


def _affine(R, t):
    return np.concatenate([np.asarray(R, dtype=np.float64), np.asarray(t, dtype=np.float64)[:, None]], axis=1)


@pytest.mark.parametrize("shape,grid,A", [
    ((21, 14, 9), (21, 14, 9), _affine(I3, (0, 0, 0))),
    ((21, 14, 9), (17, 15, 11), _affine(I3, (3, -2, 1))),
    ((21, 14, 9), (21, 14, 9), _affine(I3, (30, 0, 0))),                          # nothing inside
    ((21, 14, 9), (21, 14, 9), _affine(I3, (0.5, -0.25, 0.125))),
    ((21, 14, 9), (14, 21, 9), _affine([[0, 1, 0], [1, 0, 0], [0, 0, 1]], (0, 0, 0))),
    ((21, 14, 9), (21, 14, 9), _affine(np.diag([-1.0, 1.0, -1.0]), (20, 0, 8))),
    ((21, 14, 9), (40, 26, 17), _affine(0.5 * I3, (0.25, 0.25, 0.25))),           # finer
    ((21, 14, 9), (9, 8, 5), _affine(2.0 * I3, (1, 0, 0.5))),                     # coarser
    ((21, 14, 1), (21, 14, 1), _affine([[0.9375, 0.25, 0], [-0.25, 0.9375, 0], [0, 0, 1]], (0, 2, 0))),
    ((1, 14, 9), (3, 14, 9), _affine([[0.5, 0, 0], [0, 1, 0.125], [0, -0.125, 1]], (0, 0, 0.5))),
])
def test_push_is_the_adjoint_of_the_pull(shape, grid, A):
    import paper_2102_01604_gb300 as mpm
    d = dataset((4, 4, 4), seed=5, contrasts=("PDw", "T1w"), n_echoes=(2, 2))
    p, po = (m.make_problem(d["prot"], shape) for m in (mpm, orc))
    proj = mpm.make_projection([grid, grid], [A, A])
    rng = np.random.default_rng(6)
    u = rng.standard_normal((2, int(np.prod(shape)))).astype(np.float32)
    v = rng.standard_normal((2, int(np.prod(grid)))).astype(np.float32)
    pu = to_np(mpm.mpm_pull(p, proj, 0, to_dev(u)))
    pv = to_np(mpm.mpm_push(p, proj, 0, to_dev(v)))
    a, b = np.sum(pu * v), np.sum(u * pv)
    assert abs(a - b) <= 1e-5 * (np.sum(np.abs(pu * v)) + 1e-30)
    np.testing.assert_allclose(pv, orc.push(po, grid, A, v), rtol=1e-5, atol=1e-5)
