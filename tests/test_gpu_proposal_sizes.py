"""The proposal network at the edges of its kernels' tiles: clouds of a part of a 128-point tile, one tile
and a ragged last one, batches that leave head rows over, one to sixteen preshapes; outputs and every
gradient against the FP64 oracle, every element within test_gpu_proposal's bound.  Where
a stored activation lands on the other side of a bfloat16 boundary than float64 puts it (with 16 points
one does), all outputs follow it and the gradients are another point's: they are then not compared."""
import numpy as np
import pytest

from paper_2412_08346_gb300 import proposal, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import proposal as orc  # noqa: E402
from test_gpu_proposal import ELEM_ULPS, F32_REL, FLOOR_ULPS  # noqa: E402


def _within(a, b, what):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    bound = 2.0 ** -8 * (ELEM_ULPS * np.abs(b) + FLOOR_ULPS * np.sqrt(np.mean(b ** 2))) + 1e-30
    assert np.all(np.abs(a - b) <= bound), (what, float((np.abs(a - b) / bound).max()))


@pytest.mark.parametrize("P,points,B,T", [(1, 16, 1, 1), (2, 127, 3, 7), (4, 128, 5, 128), (3, 1001, 2, 16), (16, 300, 1, 3)])
def test_forward_and_gradients_at_tile_edges(P, points, B, T):
    g = np.random.default_rng(points)
    clouds = np.stack([synth.partial_object(points, points + 100 * b).points for b in range(B)]).astype(np.float32)
    tg = np.zeros((B, P, T, 7), np.float32)
    tg[..., :3] = clouds.mean(1)[:, None, None, :] + g.normal(0, 0.06, (B, P, T, 3))
    q = g.normal(size=(B, P, T, 4))
    tg[..., 3:] = q / np.linalg.norm(q, axis=-1, keepdims=True)
    params = synth.proposal_params(P, points)
    net = proposal.Proposal(P, points, B + 1, torch.cuda.current_stream().cuda_stream)
    try:
        net.set_params(params)
        out, cen = net.forward(clouds, B)
        loss, grad = net.loss_grad(clouds, tg, B, T, want_grad=True)
        again, _ = net.forward(clouds, B)
    finally:
        net.close()
    assert np.array_equal(out, again)
    crossed = False
    for b in range(B):
        o, _, c = orc.forward(params, clouds[b], P)
        assert np.allclose(cen[b], c, rtol=0, atol=1e-6)
        _within(out[b], o, f"object {b} outputs")
        crossed |= bool(np.any(np.abs(out[b].ravel() - o.ravel()) > F32_REL * (np.abs(o.ravel()) + np.sqrt(np.mean(o ** 2)))))
    lo, go = orc.loss_and_grad(params, list(clouds), list(tg), P)
    assert abs(loss - lo) <= 1e-3 * abs(lo), (loss, lo)
    if crossed:
        return
    start = 0
    for layer, (o, i) in enumerate(orc.layer_shapes(P)):
        for kind, n in (("W", o * i), ("b", o)):
            _within(grad[start:start + n], go[start:start + n], f"d{kind}{layer + 1}")
            start += n
