"""Cells without memory: the context goes on without them, with the same results, and keeps nothing of what it had
taken; and they leave the memory alone when little is free."""
import numpy as np
import pytest

import asicp_testlib as tl
from paper_2412_08346_gb300 import asicp, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

OBJECTS, P, K, N, M = 24, 1, 64, 700, 1100
MB = 1 << 20


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _run(arm):
    """Best poses and costs of two runs (the second on new clouds of the same sizes); arm(ctx) is called before the
    first.  Also the free memory around the first run."""
    w = synth.custom_case(P=P, K=K, N=N, M=M, grid=24, k_max=60, seed=3, k_stein=2)
    cfg = asicp.asicp_config_default(P=P, K=K, k_max=60, k_stein=2, conv_tol=-1.0, init_radius=0.05, n_objects=OBJECTS,
                                     fwd_shape=asicp.FWD_SHAPES - 1, cuda_stream=torch.cuda.current_stream().cuda_stream)
    ctx = asicp.asicp_create(cfg)
    out = []
    try:
        for p, x in enumerate(w.preshapes):
            asicp.asicp_set_gripper_sdf(ctx, p, x.S, x.sdf, x.origin, x.voxel)
        arm(ctx)
        for again in range(2):
            for o in range(OBJECTS):
                asicp.asicp_set_object_at(ctx, o, synth.partial_object(M, 100 * again + o).points)
            before = _free()
            asicp.asicp_run(ctx)
            if again == 0:
                taken = before - _free()
            for o in (0, OBJECTS - 1):
                th, cost = np.zeros((K, 7), np.float32), np.zeros(K, np.float32)
                asicp.asicp_best_grasps_at(ctx, o, K, th, cost)
                out += [th, cost]
    finally:
        asicp.asicp_destroy(ctx)
    return out, taken


def test_failed_allocations_keep_nothing():
    want, taken = _run(lambda ctx: None)
    assert taken > 200 * MB                       # both kinds of cells were built
    # the scratch; an object's nodes or leaves; the reverse matching's list, scratch and tables
    n = 1 + 2 * OBJECTS
    for after in (0, 1, 2, 20, n - 1, n, n + 1, n + 2, n + 3):
        got, kept = _run(lambda ctx: asicp.asicp_test_fail_cell_memory(ctx, after))
        for a, b in zip(got, want):
            assert np.array_equal(a, b), after
        assert kept < taken - (200 * MB if after < n else 10 * MB), (after, kept / MB, taken / MB)


def test_cells_leave_a_nearly_full_device_alone():
    want, taken = _run(lambda ctx: None)
    torch.cuda.empty_cache()
    hold, room = [], 2200 * MB                    # an eighth: less than the objects' cells, more than the gripper's
    while _free() > room + 64 * MB:
        hold.append(torch.empty(min(_free() - room, 32 << 30), dtype=torch.uint8, device="cuda"))
    got, kept = _run(lambda ctx: None)
    del hold
    torch.cuda.empty_cache()
    for a, b in zip(got, want):
        assert np.array_equal(a, b)
    assert kept < taken - 200 * MB
