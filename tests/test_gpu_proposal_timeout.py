"""An expired wait of the proposal network's encoder: the call returns TIMEOUT, the backward kernels leave their
arrays alone (no pooled point is known), and the next calls compute what a fresh handle computes."""
import numpy as np
import pytest

from paper_2412_08346_gb300 import asicp, proposal, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


@pytest.mark.parametrize("points,B", [(128, 1), (300, 3)])
def test_expired_wait_is_reported_and_the_handle_recovers(points, B):
    P, T = 2, 5
    g = np.random.default_rng(points)
    clouds = np.stack([synth.partial_object(points, 40 + b).points for b in range(B)]).astype(np.float32)
    tg = np.zeros((B, P, T, 7), np.float32)
    tg[..., :3] = g.normal(0, 0.06, (B, P, T, 3))
    tg[..., 3] = 1.0
    params = synth.proposal_params(P, 9)
    results = []
    for expire in (True, False):
        net = proposal.Proposal(P, points, B, torch.cuda.current_stream().cuda_stream)
        try:
            net.set_params(params)
            if expire:
                net.test_expire_waits(True)
                for call in (lambda: net.loss_grad(clouds, tg, B, T, want_grad=True), lambda: net.forward(clouds, B)):
                    with pytest.raises(asicp.AsicpError) as e:
                        call()
                    assert e.value.status == asicp.ASICP_ERR_TIMEOUT
                net.test_expire_waits(False)
            results.append((net.forward(clouds, B)[0], *net.loss_grad(clouds, tg, B, T, want_grad=True)))
        finally:
            net.close()
    for a, b in zip(*results):
        assert np.array_equal(a, b)
