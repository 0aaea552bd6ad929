"""Gradients of the proposal network at the edges of its kernels' tiles, for inputs on which no stored activation lands on
the other side of a bfloat16 boundary than float64 puts it (where one does, outputs and gradients are
another point's and are not compared): of six clouds' seeds per size at least one has to be such an input."""
import numpy as np
import pytest

from paper_2412_08346_gb300 import proposal, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import proposal as orc  # noqa: E402
from test_gpu_proposal import ELEM_ULPS, F32_REL, FLOOR_ULPS  # noqa: E402


@pytest.mark.parametrize("P,points,T", [(1, 16, 1), (2, 127, 7), (4, 128, 128), (3, 129, 5), (3, 1001, 16), (16, 300, 3)])
def test_gradients_where_nothing_crossed(P, points, T):
    compared = 0
    for seed in range(6):
        g = np.random.default_rng(1000 * points + seed)
        cloud = synth.partial_object(points, 50 + 7 * points + seed).points.astype(np.float32)[None]
        tg = np.zeros((1, P, T, 7), np.float32)
        tg[..., :3] = cloud.mean(1)[:, None, None, :] + g.normal(0, 0.06, (1, P, T, 3))
        q = g.normal(size=(1, P, T, 4))
        tg[..., 3:] = q / np.linalg.norm(q, axis=-1, keepdims=True)
        params = synth.proposal_params(P, points + seed)
        net = proposal.Proposal(P, points, 1, torch.cuda.current_stream().cuda_stream)
        try:
            net.set_params(params)
            out, _ = net.forward(cloud, 1)
            loss, grad = net.loss_grad(cloud, tg, 1, T, want_grad=True)
        finally:
            net.close()
        o = orc.forward(params, cloud[0], P)[0].ravel()
        if np.any(np.abs(out.ravel() - o) > F32_REL * (np.abs(o) + np.sqrt(np.mean(o ** 2)))):
            continue
        compared += 1
        lo, go = orc.loss_and_grad(params, list(cloud), list(tg), P)
        assert abs(loss - lo) <= 1e-3 * abs(lo)
        start = 0
        for layer, (rows, cols) in enumerate(orc.layer_shapes(P)):
            for kind, n in (("W", rows * cols), ("b", rows)):
                a, b = grad[start:start + n].astype(np.float64), np.asarray(go[start:start + n], np.float64)
                bound = 2.0 ** -8 * (ELEM_ULPS * np.abs(b) + FLOOR_ULPS * np.sqrt(np.mean(b ** 2))) + 1e-30
                assert np.all(np.abs(a - b) <= bound), (seed, f"d{kind}{layer + 1}", float((np.abs(a - b) / bound).max()))
                start += n
    assert compared > 0
