"""The bytes the PCG iteration moves (bench.moved_step_bytes, behind the
roofline figure), against its operands written out: vectors of four floats per
voxel, w and the packed H."""
import bench

V, W = 16, 4


def test_moved_step_bytes():
    for K, H in ((4, 40), (3, 24)):
        assert bench.moved_step_bytes(0, K) == V + W + H + V                 # p_0; v_0
        assert bench.moved_step_bytes(1, K) == 2 * V + W + H + 2 * V         # p_0, v_0; p_1, v_1
        assert bench.moved_step_bytes(3, K) == 3 * V + W + H + 2 * V         # p_2, v_2, p_1; p_3, v_3
        assert bench.moved_step_bytes(2, K) == 3 * V + W + H + 3 * V         # p_1, v_1, p_0; p_2, v_2, x
        assert bench.moved_step_bytes(4, K) == 4 * V + W + H + 3 * V         # x too
    mean = sum(bench.moved_step_bytes(j, 4) for j in range(30)) / 30
    assert abs(mean - 136.3) < 0.05
