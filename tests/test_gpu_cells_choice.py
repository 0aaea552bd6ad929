"""Which clouds are matched through cells: those whose cells' lists are short; on others (points on a common
sphere or cylinder, copies of one point) the screening goes on, which is faster there.  With kernel timers the
exact choice after the screening is counted and the matching through cells has none."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

P, K, N, M = 2, 96, 1024, 8192
EXACT = asicp.KERNEL_KINDS.index("exact")


def _cloud(kind):
    g = np.random.default_rng(5)
    if kind == "sphere":
        R = g.normal(size=(M, 3))
        R *= 0.05 / np.linalg.norm(R, axis=1, keepdims=True)
    elif kind == "cylinder":
        a = g.uniform(0, 2 * np.pi, M)
        R = np.stack([0.03 * np.cos(a), 0.03 * np.sin(a), g.uniform(-0.06, 0.06, M)], 1)
    elif kind == "one point":
        R = np.tile([[0.01, 0.02, 0.03]], (M, 1))
    else:
        R = synth.partial_object(M, 7 if kind == "object" else 8).points
    return np.ascontiguousarray(R, dtype=np.float32)


@pytest.mark.parametrize("kind,cells", [("object", True), ("sphere", False), ("cylinder", False), ("one point", False)])
def test_cells_only_where_their_lists_are_short(kind, cells):
    g = np.random.default_rng(1)
    q = g.normal(size=(P * K, 4))
    theta = np.concatenate([g.normal(size=(P * K, 3)) * 0.01, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    S = g.uniform(-0.02, 0.02, (P, N, 3)).astype(np.float32)
    cfg = asicp.asicp_config_default(P=P, K=K, k_max=2, k_stein=0, conv_tol=-1.0, debug=1, profile=1,
                                     fwd_shape=asicp.FWD_SHAPES - 1, cuda_stream=torch.cuda.current_stream().cuda_stream)
    ctx = asicp.asicp_create(cfg)

    def steps(n):
        """State after the last of n equal steps, and whether it ran the exact choice."""
        for _ in range(n):
            asicp.asicp_kernel_times(ctx, reset=True)
            asicp.asicp_set_state(ctx, theta, 0)
            asicp.asicp_step(ctx, 0)
        st = tl.read_state(ctx, P, K, N, M)
        return st, asicp.asicp_kernel_times(ctx)[1][EXACT] > 0

    try:
        for p in range(P):
            asicp.asicp_set_gripper_sdf(ctx, p, S[p], -np.ones((8, 8, 8), np.float32), np.full(3, -0.1, np.float32),
                                        np.float32(0.2 / 7))
        asicp.asicp_set_object(ctx, _cloud(kind))
        first, screened = steps(1)
        assert screened                            # the build is not due yet
        last, screened = steps(60)
        assert screened != cells
        for key in ("nn_idx", "cost", "grad"):
            assert np.array_equal(first[key], last[key]), key
        # the next cloud is looked at anew (after a refusal the build has to pay several times over)
        asicp.asicp_set_object(ctx, _cloud("another object"))
        first, screened = steps(1)
        assert screened
        last, screened = steps(120)
        assert not screened
        for key in ("nn_idx", "cost", "grad"):
            assert np.array_equal(first[key], last[key]), key
    finally:
        asicp.asicp_destroy(ctx)
