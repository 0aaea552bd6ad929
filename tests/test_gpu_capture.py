"""asicp_step inside the caller's own stream capture: launches only, nothing counts as prepared before a replay
has run, and every replay computes the step on the clouds and grippers that the context then holds."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

KEYS = ("grad", "theta")           # (what can be read back when only a replay has run since the poses were set)


def _context(w, R, pre, shape, stream):
    ctx = asicp.asicp_create(tl.make_config(w, stream.cuda_stream, fwd_shape=shape))
    asicp.asicp_set_object(ctx, R)
    _grip(ctx, pre)
    return ctx


def _grip(ctx, pre):
    for p, x in enumerate(pre):
        asicp.asicp_set_gripper_sdf(ctx, p, x.S, x.sdf, x.origin, x.voxel)


# (the second size runs the collision test beside the matching; both build cells in direct steps)
@pytest.mark.parametrize("K,N", [(16, 600), (256, 2100)])
@pytest.mark.parametrize("shape", [0, asicp.FWD_SHAPES - 1])
def test_replays_follow_the_context(K, N, shape):
    P, M = 2, 1500
    w = synth.custom_case(P=P, K=K, N=N, M=M, grid=24, k_max=4, seed=31, k_stein=0)
    R, R2 = w.objects[0].points, synth.partial_object(M, 44).points
    pre, pre2 = w.preshapes, synth.make_preshapes(P, N, 24, 99)
    g = np.random.default_rng(4)
    q = g.normal(size=(P * K, 4))
    theta = np.concatenate([R.mean(0) + g.normal(size=(P * K, 3)) * 0.03, q / np.linalg.norm(q, axis=1, keepdims=True)],
                           1).astype(np.float32)
    stream = torch.cuda.Stream()

    def state(ctx):
        out = {"theta": np.zeros((P * K, 7), np.float32), "grad": np.zeros((P * K, 7))}
        asicp.asicp_get_state(ctx, **out)
        return out

    def step(ctx):
        asicp.asicp_set_state(ctx, theta, 1)
        asicp.asicp_step(ctx, 1)
        return state(ctx)

    def capture(ctx):
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            asicp.asicp_step(ctx, 1)
        return graph

    def replay(ctx, graph):
        asicp.asicp_set_state(ctx, theta, 1)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            graph.replay()
        stream.synchronize()
        return state(ctx)

    want = {}
    for name, r, x in (("first", R, pre), ("object", R2, pre), ("both", R2, pre2)):
        ctx = _context(w, r, x, shape, stream)
        want[name] = step(ctx)
        collide = tl.read_state(ctx, P, K, N, M)["ncol"]
        assert collide.any() and not collide.all()
        asicp.asicp_destroy(ctx)

    def same(got, name):
        for key in KEYS:
            assert np.array_equal(got[key], want[name][key]), (name, key)

    ctx = _context(w, R, pre, shape, stream)
    try:
        asicp.asicp_set_state(ctx, theta, 1)
        early = capture(ctx)                       # before anything has been prepared
        same(step(ctx), "first")                   # (a direct step prepares for itself)
        same(replay(ctx, early), "first")
        for _ in range(120):                       # cells are built on the way
            last = step(ctx)
        same(last, "first")
        late = capture(ctx)
        for graph in (early, late):
            same(replay(ctx, graph), "first")
        asicp.asicp_set_object(ctx, R2)
        for graph in (late, early):
            same(replay(ctx, graph), "object")
        same(step(ctx), "object")
        _grip(ctx, pre2)
        for graph in (late, early):
            same(replay(ctx, graph), "both")
        same(step(ctx), "both")
        del early, late
    finally:
        torch.cuda.synchronize()
        asicp.asicp_destroy(ctx)
