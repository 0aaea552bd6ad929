"""Matching through the objects' cells (the tensor-core shape on clouds of 1024 points and more)
against the float32 kernel and the FP64 nearest neighbour, on clouds where a cell's list is hard to
keep short (exact planes, a sphere seen from its centre, duplicates), at the smallest size that uses
cells and one below, and on queries near, far and beyond the outermost cells."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)


def _cloud(kind, M):
    g = np.random.default_rng(M)
    if kind == "plane":
        R = np.concatenate([g.uniform(-0.05, 0.05, (M, 2)), np.zeros((M, 1))], 1)
    elif kind == "grid":
        R = np.stack(np.meshgrid(*[np.arange(int(np.ceil(M ** (1 / 3)))) * 0.004] * 3), -1).reshape(-1, 3)[:M]
    elif kind == "sphere":
        R = g.normal(size=(M, 3))
        R *= 0.05 / np.linalg.norm(R, axis=1, keepdims=True)
    elif kind == "duplicates":
        R = g.uniform(-0.05, 0.05, (64, 3))[g.integers(0, 64, M)]
    elif kind == "shifted":
        R = synth.partial_object(M, 5).points + np.float32([3.0, -2.0, 8.0])
    else:
        R = synth.partial_object(M, 7).points
    return np.ascontiguousarray(R, dtype=np.float32)


def _indices(R, S, theta, P, shape):
    N = S.shape[1]
    cfg = asicp.asicp_config_default(P=P, K=len(theta) // P, k_max=2, k_stein=0, conv_tol=-1.0, debug=1, fwd_shape=shape,
                                     cuda_stream=torch.cuda.current_stream().cuda_stream)
    ctx = asicp.asicp_create(cfg)
    try:
        asicp.asicp_set_object(ctx, R)
        for p in range(P):
            asicp.asicp_set_gripper_sdf(ctx, p, S[p], -np.ones((8, 8, 8), np.float32), np.full(3, -0.1, np.float32),
                                        np.float32(0.2 / 7))
        for _ in range(100 if shape else 1):         # the build waits until the steps would have paid for it
            asicp.asicp_set_state(ctx, theta, 0)
            asicp.asicp_step(ctx, 0)
        return tl.read_state(ctx, P, len(theta) // P, N, len(R))
    finally:
        asicp.asicp_destroy(ctx)


@pytest.mark.parametrize("kind,M", [("partial", 1023), ("partial", 1024), ("partial", 9001), ("shifted", 4099),
                                    ("plane", 2000), ("grid", 1728), ("sphere", 1500), ("duplicates", 1100)])
def test_cells_find_the_nearest_points(kind, M):
    R = _cloud(kind, M)
    g = np.random.default_rng(3)
    P, N, K = 2, 203, 64
    S = g.uniform(-0.05, 0.05, (P, N, 3)).astype(np.float32)
    S[:, :40] = R[g.integers(0, M, (P, 40))] - R.mean(0)       # on object points (when the pose is the identity)
    S[:, 40] = 0.0
    c = (R.max(0) + R.min(0)) / 2
    t = np.stack([R.mean(0), c, c + [0.1, 0, 0], c - [0, 0.3, 0.1], c + [0, 0, 1.5], c + [4, 4, -4], c - [9, 0, 30],
                  c + [0.02, 0.03, -0.01]])
    t = np.tile(t, (K // 8, 1))
    q = g.normal(size=(K, 4))
    q[::8] = q[1::8] = [1, 0, 0, 0]
    theta = np.tile(np.concatenate([t, q / np.linalg.norm(q, axis=1, keepdims=True)], 1), (P, 1)).astype(np.float32)
    a, b = (_indices(R, S, theta, P, v) for v in (0, asicp.FWD_SHAPES - 1))
    assert np.array_equal(a["s_prime"], b["s_prime"])
    tl.check_nn(b["s_prime"].reshape(-1, 3), R, b["nn_idx"].reshape(-1), {})
    d = b["s_prime"].astype(np.float64) - R[b["nn_idx"]]
    assert np.allclose(b["nn_d2"], (d ** 2).sum(-1), rtol=1e-6, atol=0)
    # the cells give the lowest index of the smallest float32 distance over the whole cloud; the float32
    # kernel the same, but for points whose distances differ by less than their rounding
    for pk in range(P * K):
        diff = np.nonzero(a["nn_idx"][pk] != b["nn_idx"][pk])[0]
        assert np.all(b["nn_d2"][pk][diff] <= a["nn_d2"][pk][diff])
        tie = diff[b["nn_d2"][pk][diff] == a["nn_d2"][pk][diff]]
        assert np.all(b["nn_idx"][pk][tie] < a["nn_idx"][pk][tie])
        if np.abs(t[pk % K] - c).max() < 1.0:
            assert len(diff) == 0


@pytest.mark.parametrize("N,offset", [(511, 0.0), (512, 0.0), (2047, 0.0), (1000, 3.0), (1000, 30.0)])
def test_gripper_cells_give_the_same_reverse_matches(N, offset):
    """Reverse matching through the gripper clouds' cells (512 points and more, once the steps have paid for
    their build; an object metres away is beyond their tolerance and compares the whole cloud)
    against the brute-force kernel of a context's first step: every output of the step the same."""
    w = synth.custom_case(P=2, K=24, N=N, M=1500, grid=40, k_max=4, seed=83, k_stein=0)
    w.objects[0].points = (w.objects[0].points + np.float32(offset)).astype(np.float32)
    g = np.random.default_rng(N)
    t = w.objects[0].points.mean(0, dtype=np.float64) + g.normal(size=(48, 3)) * 0.02
    q = g.normal(size=(48, 4))
    theta = np.concatenate([t, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    states = []
    for steps in (1, 80):
        ctx = asicp.asicp_create(tl.make_config(w, torch.cuda.current_stream().cuda_stream))
        try:
            keep = tl.upload(ctx, w)
            for _ in range(steps):
                asicp.asicp_set_state(ctx, theta, 0)
                asicp.asicp_step(ctx, 0)
            states.append(tl.read_state(ctx, 2, 24, N, 1500))
            del keep
        finally:
            asicp.asicp_destroy(ctx)
    a, b = states
    assert a["ncol"].max() > 64
    for pk in range(48):
        n = a["ncol"][pk]
        assert np.array_equal(a["col_list"][pk, :n], b["col_list"][pk, :n])
        assert np.array_equal(a["col_nn"][pk, :n], b["col_nn"][pk, :n])
    for key in ("theta", "cost", "grad", "ncol"):
        assert np.array_equal(a[key], b[key]), key


@pytest.mark.parametrize("Mc", [1, 31, 33, 4096, 65537, 131072 + 45])
def test_collision_test_skips_no_colliding_point(Mc):
    """The collision test skips chunks of the spatially sorted collision cloud that are clear of the gripper:
    the colliding points, ascending, are the oracle's (but for values within 1e-6 m of zero), for
    clouds of one point to several segments of the sort and a grid of three different sides."""
    import oracle
    w = synth.custom_case(P=2, K=6, N=64, M=300, grid=28, k_max=2, seed=91, k_stein=0)
    g = np.random.default_rng(Mc)
    for pre in w.preshapes:
        pre.sdf = np.ascontiguousarray(pre.sdf[2:, 1:, :])
        pre.origin = (pre.origin + pre.voxel * np.float32([0, 1, 2])).astype(np.float32)
    C = (w.objects[0].points.mean(0) + g.uniform(-0.12, 0.12, (Mc, 3))).astype(np.float32)
    t = C.mean(0, dtype=np.float64) + g.normal(size=(12, 3)) * 0.04
    q = g.normal(size=(12, 4))
    theta = np.concatenate([t, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    theta[3, :3] += 5.0                                        # nowhere near
    ctx = asicp.asicp_create(tl.make_config(w, torch.cuda.current_stream().cuda_stream))
    try:
        asicp.asicp_set_object(ctx, w.objects[0].points, C)
        for p, pre in enumerate(w.preshapes):
            asicp.asicp_set_gripper_sdf(ctx, p, pre.S, pre.sdf, pre.origin, pre.voxel)
        asicp.asicp_set_state(ctx, theta, 0)
        before = tl.read_theta(ctx, 12)
        asicp.asicp_step(ctx, 0)
        st = tl.read_state(ctx, 2, 6, 64, Mc)
    finally:
        asicp.asicp_destroy(ctx)
    orc = oracle.Oracle(np.stack([pre.S for pre in w.preshapes]), [(pre.sdf, pre.origin, pre.voxel) for pre in w.preshapes],
                        w.objects[0].points, Cc=C, K=6)
    for pk in range(12):
        want, vals = orc.collision_points(pk // 6, before[pk].astype(np.float64))
        got = st["col_list"][pk, :st["ncol"][pk]]
        assert np.all(np.diff(got) > 0)
        diff = np.setxor1d(got, want)
        assert np.all(np.abs(np.asarray(vals)[diff]) <= tl.PHI_TOL), (pk, len(diff))
    assert st["ncol"][3] == 0 and st["ncol"].max() >= Mc // 200       # (the gripper fills 0.75 % of the cube)


@pytest.mark.parametrize("M", [1, 63, 64, 65, 255, 257, 1025, 2048, 2049])
def test_every_shape_at_the_edges_of_chunks_and_tiles(M):
    """Clouds that end inside, at and just past a screening chunk or tile (only whole chunks up to the last
    point are read), prepared by several CTAs: every matching shape finds the nearest points, and the
    no-allocation entry point the same ones."""
    R = _cloud("partial", M)
    g = np.random.default_rng(M)
    S = g.uniform(-0.05, 0.05, (2, 70, 3)).astype(np.float32)
    q = g.normal(size=(8, 4))
    theta = np.concatenate([g.normal(size=(8, 3)) * 0.05, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)
    stream = torch.cuda.current_stream().cuda_stream
    out = torch.full((8 * 70,), -1, dtype=torch.int32, device="cuda")
    asicp.asicp_match_noalloc(theta, S.reshape(-1, 3), R, out, 2, 4, stream)
    got = [out.cpu().numpy().reshape(8, 70)]
    for shape in range(asicp.FWD_SHAPES):
        cfg = asicp.asicp_config_default(P=2, K=4, k_max=1, k_stein=0, conv_tol=-1.0, debug=1, fwd_shape=shape, cuda_stream=stream)
        ctx = asicp.asicp_create(cfg)
        try:
            asicp.asicp_set_object(ctx, R)
            for p in range(2):
                asicp.asicp_set_gripper_sdf(ctx, p, S[p], -np.ones((8, 8, 8), np.float32), np.full(3, -0.1, np.float32),
                                            np.float32(0.2 / 7))
            asicp.asicp_set_state(ctx, theta, 0)
            asicp.asicp_step(ctx, 0)
            st = tl.read_state(ctx, 2, 4, 70, M)
        finally:
            asicp.asicp_destroy(ctx)
        got.append(st["nn_idx"])
        if shape == 0:
            tl.check_nn(st["s_prime"].reshape(-1, 3), R, st["nn_idx"].reshape(-1), {})
    for idx in got:
        assert np.array_equal(idx, got[1])


@pytest.mark.parametrize("K,N,shape", [(7, 33, 0), (256, 4095, 7), (256, 4096, 7), (257, 4096, 0)])
def test_collision_test_beside_the_matching_gives_the_same_pass(K, N, shape):
    """A pass with kernel timers runs its kernels one after the other, one without runs the collision test beside
    the matching (in a captured loop, and directly from 2^20 gripper points on): the same poses and costs, also
    after a matching whose waits expired while the collision test beside it ran."""
    w = synth.custom_case(P=1, K=K, N=N, M=1500, grid=24, k_max=3, seed=5, k_stein=1)
    out = []
    for profile in (1, 0):
        cfg = asicp.asicp_config_default(P=1, K=K, k_max=3, k_stein=1, conv_tol=-1.0, init_radius=0.05, profile=profile,
                                         fwd_shape=shape, cuda_stream=torch.cuda.current_stream().cuda_stream)
        ctx = asicp.asicp_create(cfg)
        try:
            keep = tl.upload(ctx, w)
            if shape == 0 and profile == 0:
                asicp.asicp_test_expire_waits(ctx, True)
                asicp.asicp_run(ctx)
                with pytest.raises(asicp.AsicpError):
                    asicp.asicp_get_state(ctx, theta=np.zeros((K, 7), np.float32))
                asicp.asicp_test_expire_waits(ctx, False)
            asicp.asicp_run(ctx)
            state = [np.zeros((K, 7), np.float32), np.zeros(K), np.zeros(K, np.int32)]
            asicp.asicp_get_state(ctx, theta=state[0], cost=state[1], ncol=state[2])
            asicp.asicp_step(ctx, 2)
            more = [np.zeros((K, 7), np.float32), np.zeros(K), np.zeros(K, np.int32)]
            asicp.asicp_get_state(ctx, theta=more[0], cost=more[1], ncol=more[2])
            out.append(state + more)
            del keep
        finally:
            asicp.asicp_destroy(ctx)
    assert out[0][2].any()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
