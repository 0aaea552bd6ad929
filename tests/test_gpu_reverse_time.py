"""The reverse matching is never much slower through the gripper clouds' cells than by brute force, and finds the same
points: an object far from its frame's origin (the cells do not hold there), and a contact cloud that covers a small part
of the gripper's body (colliding points lie far from it)."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

REVERSE = asicp.KERNEL_KINDS.index("collide_nn")


@pytest.mark.parametrize("offset,pads", [(0.0, 1.0), (30.0, 1.0), (0.0, 0.2), (0.0, 0.03)])
def test_cells_are_no_slower_than_brute_force(offset, pads):
    P, K, N, M = 2, 256, 2048, 8192
    w = synth.custom_case(P=P, K=K, N=N, M=M, grid=48, k_max=4, seed=19, k_stein=0)
    R = (w.objects[0].points + np.float32(offset)).astype(np.float32)
    g = np.random.default_rng(6)
    q = g.normal(size=(P * K, 4))
    theta = np.concatenate([R.mean(0, dtype=np.float64) + g.normal(size=(P * K, 3)) * 0.02,
                            q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    ctx = asicp.asicp_create(tl.make_config(w, torch.cuda.current_stream().cuda_stream, profile=True))

    def steps(n):
        """Shortest reverse matching of n equal steps, in ms, and the state after the last."""
        times = []
        for _ in range(n):
            asicp.asicp_kernel_times(ctx, reset=True)
            asicp.asicp_set_state(ctx, theta, 0)
            asicp.asicp_step(ctx, 0)
            times.append(asicp.asicp_kernel_times(ctx)[0][REVERSE])
        return min(times), tl.read_state(ctx, P, K, N, M)

    try:
        asicp.asicp_set_object(ctx, R)
        for p, pre in enumerate(w.preshapes):
            S = ((pre.S - pre.S.mean(0)) * np.float32(pads) + pre.S.mean(0)).astype(np.float32)
            asicp.asicp_set_gripper_sdf(ctx, p, S, pre.sdf, pre.origin, pre.voxel)
        brute, a = steps(2)                        # the build is not due yet
        steps(80)
        later, b = steps(5)
    finally:
        asicp.asicp_destroy(ctx)
    assert a["ncol"].sum() > 50000
    for pk in range(P * K):
        n = a["ncol"][pk]
        assert np.array_equal(a["col_nn"][pk, :n], b["col_nn"][pk, :n])
    for key in ("ncol", "cost", "grad", "theta"):
        assert np.array_equal(a[key], b[key]), key
    assert later <= 1.5 * brute, (later, brute)
