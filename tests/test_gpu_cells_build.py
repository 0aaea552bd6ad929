"""Builds of the matching cells that the other tests do not reach: clouds beyond the sizes whose verdicts are kept in
shared memory, up to the largest and one above; more objects than one launch takes, of uneven sizes; a new cloud in a
context whose cells are in use; a cloud padded with copies of a point.  Each test waits until the matching
does go through the cells (the exact choice is no longer launched) and compares with the float32 kernel, and with the
nearest points in float64."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

CELLS = asicp.FWD_SHAPES - 1
EXACT = asicp.KERNEL_KINDS.index("exact")


class _Context:
    def __init__(self, clouds, K, N, shape):
        g = np.random.default_rng(N)
        self.K, self.N, self.clouds = K, N, list(clouds)
        cfg = asicp.asicp_config_default(P=1, K=K, k_max=2, k_stein=0, conv_tol=-1.0, debug=1, profile=1, fwd_shape=shape,
                                         n_objects=len(clouds), cuda_stream=torch.cuda.current_stream().cuda_stream)
        self.ctx = asicp.asicp_create(cfg)
        asicp.asicp_set_gripper_sdf(self.ctx, 0, g.uniform(-0.04, 0.04, (N, 3)).astype(np.float32), -np.ones((6, 6, 6), np.float32),
                                    np.full(3, -0.1, np.float32), np.float32(0.04))
        for o, R in enumerate(clouds):
            asicp.asicp_set_object_at(self.ctx, o, R)

    def close(self):
        asicp.asicp_destroy(self.ctx)

    def replace(self, o, R):
        self.clouds[o] = R
        asicp.asicp_set_object_at(self.ctx, o, R)

    def step(self):
        """(nearest points, transformed gripper points, whether the exact choice ran) of one step."""
        g = np.random.default_rng(3)
        theta = []
        for R in self.clouds:
            q = g.normal(size=(self.K, 4))
            theta.append(np.concatenate([R.mean(0, dtype=np.float64) + g.normal(size=(self.K, 3)) * 0.05,
                                         q / np.linalg.norm(q, axis=1, keepdims=True)], 1))
        T = self.K * len(self.clouds)
        asicp.asicp_kernel_times(self.ctx, reset=True)
        asicp.asicp_set_state(self.ctx, np.concatenate(theta).astype(np.float32), 0)
        asicp.asicp_step(self.ctx, 0)
        idx, sp = np.zeros((T, self.N), np.int32), np.zeros((T, self.N, 3), np.float32)
        asicp.asicp_get_state(self.ctx, nn_idx=idx, s_prime=sp)
        return idx, sp, asicp.asicp_kernel_times(self.ctx)[1][EXACT] > 0

    def until_cells(self, most=400):
        for n in range(most):
            idx, sp, screened = self.step()
            if not screened:
                return idx, sp, n
        return idx, sp, None


def _check(clouds, K, N, idx, sp):
    other = _Context(clouds, K, N, 0)
    try:
        want, sp0, _ = other.step()
    finally:
        other.close()
    assert np.array_equal(sp, sp0)
    assert np.array_equal(idx, want)
    for o, R in enumerate(clouds):
        rows = slice(o * K, o * K + 2)             # (two particles each: the search in float64 is slow)
        tl.check_nn(sp[rows].reshape(-1, 3), R, idx[rows].reshape(-1), {})


@pytest.mark.parametrize("M,cells", [(65537, True), (131071, True), (1 << 18, True), ((1 << 18) + 1, False)])
def test_large_clouds(M, cells):
    R = synth.partial_object(M, 21).points
    c = _Context([R], 16, 512, CELLS)
    try:
        idx, sp, n = c.until_cells(120)
    finally:
        c.close()
    assert (n is not None) == cells
    assert n != 0                                  # (the build is not due at once)
    _check([R], 16, 512, idx, sp)


def test_more_objects_than_a_launch_takes():
    g = np.random.default_rng(9)
    sizes = [1, 2, 13, 33, 700, 1023, 4097] + [int(m) for m in g.integers(50, 2500, 34)]
    clouds = [synth.partial_object(m, 60 + o).points for o, m in enumerate(sizes)]
    c = _Context(clouds, 32, 300, CELLS)
    try:
        idx, sp, n = c.until_cells()
        assert n
        _check(clouds, 32, 300, idx, sp)
        # some of them replaced, by clouds of the same and of other sizes
        for o, m in ((0, 1), (5, 1023), (6, 5000), (40, 64)):
            c.replace(o, synth.partial_object(m, 900 + o).points)
        idx, sp, n = c.until_cells()
        assert n
        _check(c.clouds, 32, 300, idx, sp)
    finally:
        c.close()


def test_a_new_cloud_while_cells_are_in_use():
    clouds = [synth.partial_object(2000, 70 + k).points for k in range(3)]
    clouds[2] = np.concatenate([clouds[2][:1900], np.repeat(clouds[2][:1], 100, 0)])     # padded with copies
    c = _Context(clouds[:1], 64, 500, CELLS)
    try:
        for k, R in enumerate(clouds):
            if k:
                c.replace(0, R)
                idx, sp, screened = c.step()
                assert screened                    # the old cloud's cells are not used
                _check([R], 64, 500, idx, sp)
            idx, sp, n = c.until_cells()
            assert n is not None
            _check([R], 64, 500, idx, sp)
    finally:
        c.close()
