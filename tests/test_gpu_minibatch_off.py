"""Mini-batches end with the call that switches them off: a step that ran on one leaves nothing behind for the
steps and runs after asicp_set_minibatch(None), or after a new object of the same size."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

P, K, N, M = 2, 9, 130, 700


def _context(w, R):
    ctx = asicp.asicp_create(tl.make_config(w, torch.cuda.current_stream().cuda_stream))
    asicp.asicp_set_object(ctx, R)
    for p, pre in enumerate(w.preshapes):
        asicp.asicp_set_gripper_sdf(ctx, p, pre.S, pre.sdf, pre.origin, pre.voxel)
    return ctx


def _step_and_run(ctx, theta):
    asicp.asicp_set_state(ctx, theta, 1)
    asicp.asicp_step(ctx, 1)
    st = tl.read_state(ctx, P, K, N, M)
    asicp.asicp_run(ctx, theta)
    out = tl.read_state(ctx, P, K, N, M)
    return [st[k] for k in ("nn_idx", "cost", "theta")] + [out[k] for k in ("nn_idx", "cost", "theta")]


@pytest.mark.parametrize("how", ["off", "new object", "new object, run first"])
def test_no_step_matches_against_a_mini_batch_that_is_off(how):
    w = synth.custom_case(P=P, K=K, N=N, M=M, grid=24, k_max=12, seed=77, k_stein=0)
    R, other = w.objects[0].points, synth.partial_object(M, 12).points
    g = np.random.default_rng(2)
    q = g.normal(size=(P * K, 4))
    theta = np.concatenate([g.normal(size=(P * K, 3)) * 0.08, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    ctx = _context(w, R)
    fresh = _context(w, R if how == "off" else other)
    try:
        asicp.asicp_set_minibatch(ctx, *synth.minibatch_ramp(M, w.k_max, 5))
        asicp.asicp_set_state(ctx, theta, 1)
        asicp.asicp_step(ctx, 1)
        assert tl.read_state(ctx, P, K, N, M)["nn_idx"].max() < M // 2      # it did run on a mini-batch
        if how == "off":
            asicp.asicp_set_minibatch(ctx, None, None)
        else:
            asicp.asicp_set_object(ctx, other)
        if how.endswith("run first"):
            for c in (ctx, fresh):
                asicp.asicp_run(c, theta)
        for a, b in zip(_step_and_run(ctx, theta), _step_and_run(fresh, theta)):
            assert np.array_equal(a, b)
    finally:
        asicp.asicp_destroy(ctx)
        asicp.asicp_destroy(fresh)
