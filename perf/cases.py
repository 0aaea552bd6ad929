"""The library's work as its users have it done, as cases that can be prepared, run and checked.

A case is a dict of plain values whose "kind" says which public calls it goes through:

run      a grasp set: every object's cloud is set, the loop runs from the Fibonacci poses (or given
         ones) and all particles are read back ranked, as asicp_set_object / asicp_run /
         asicp_best_grasps are used for a freshly seen object; the gripper is set up once
step     one teacher-forced iteration of a warm context: asicp_set_state / asicp_step /
         asicp_get_state
match    asicp_match_noalloc on device memory, as a control loop without allocations calls it
propose  the learned proposal: network forward pass and sampled initial poses
train    one training step of the proposal network: loss, gradient and Adam update

Inputs are the seeded procedural workloads of paper_2412_08346_gb300.synth; exact() restates an
iteration and the network in float64 with torch alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2412_08346_gb300 import asicp, proposal, synth

FASTEST = asicp.FWD_SHAPES - 1        # the matching shape learned_init takes and the autotuner picks
DEFAULT = 0                           # what a caller gets who leaves the configuration alone
RUN = dict(kind="run", P=3, K=256, N=2048, M=8192, objects=1, uneven=False, table=0, grid=64, k_max=100, k_stein=-1,
           schedule=0, radius=0.15, given=False, minibatch=False, freeze=False, shape=FASTEST, host=True)
STEP = dict(kind="step", P=3, K=256, N=2048, M=8192, table=0, grid=64, k_max=100, k=20, radius=0.06, shape=FASTEST)


def listed():
    return [
        # the smallest whole call: a noisy box, 32 poses, 50 linearly annealed Stein iterations; launches
        # and the latency of each small kernel count
        dict(RUN, name="grasp-small", P=1, K=32, N=256, M=512, grid=32, k_max=50, k_stein=50, schedule=1, shape=DEFAULT),
        # the paper's Table I: about 30 poses a preshape, a cloud of 1100-1900 points, 15 + 25
        # iterations on the mini-batch ramp, particles freezing on convergence
        dict(RUN, name="grasp-table1-ramp", K=30, N=777, M=1499, grid=32, k_max=40, minibatch=True, freeze=True, shape=DEFAULT),
        # a grasp on a table: the collision cloud is the object and the table under it
        dict(RUN, name="grasp-on-table", P=2, K=64, N=1024, M=3001, table=1500, grid=48, k_max=40, freeze=True, host=False),
        # the paper-scale grasp set of the benchmark
        dict(RUN, name="grasp-paper-scale"),
        # several objects in one pass, uneven clouds (1k-32k points) and particle counts (128-512)
        dict(RUN, name="grasp-batch", objects=8, uneven=True, M=32768, K=512, k_max=40),
        # learned initial poses refined by a few SGD iterations, sixteen clouds at a time
        dict(RUN, name="refine-proposals", objects=16, K=64, M=2048, k_max=10, k_stein=0, radius=0.05, given=True),
        # one Stein iteration at the paper's scale, state in and out
        dict(STEP, name="step-stein"),
        # one SGD iteration at odd sizes, most particles in collision
        dict(STEP, name="step-sgd-odd", P=2, K=77, N=1023, M=5003, grid=41, k=60, radius=0.04),
        # the largest object: 65536 points, 3 x 1024 particles, 128^3 SDF
        dict(STEP, name="step-large", K=1024, N=4096, M=65536, grid=128, k=60),
        # correspondences alone in a control loop that must not allocate
        dict(kind="match", name="match-noalloc", P=2, K=64, N=1024, M=4096, radius=0.08),
        # poses proposed for one freshly seen cloud
        dict(kind="propose", name="propose-one", P=3, B=1, points=2048, K=64),
        # a training step on the batch the network is trained with
        dict(kind="train", name="train-batch", P=3, B=32, points=2048, T=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "step", "step", "match", "propose", "train"])
    if kind in ("run", "batch"):
        c = dict(RUN, P=rng.randint(1, 4), K=_log(rng, 16, 512), N=_log(rng, 200, 4096), M=_log(rng, 500, 32768),
                 grid=rng.randint(24, 72), k_max=rng.randint(8, 100), freeze=rng.random() < 0.5,
                 host=rng.random() < 0.5, schedule=rng.randint(0, 1))
        if kind == "batch":
            c.update(objects=rng.randint(2, 16), uneven=rng.random() < 0.5, given=rng.random() < 0.5, k_max=rng.randint(4, 20))
        elif rng.random() < 0.3:
            c.update(table=_log(rng, 200, 4000))
        elif rng.random() < 0.2:
            c.update(minibatch=True, shape=DEFAULT, M=_log(rng, 500, 4000))
        if c["objects"] == 1 and c["P"] * c["K"] * c["N"] * c["M"] < 2e8:
            c.update(shape=rng.choice([DEFAULT, FASTEST]) if not c["minibatch"] else DEFAULT)
        while c["objects"] * c["P"] * c["K"] * c["N"] * c["M"] * (c["k_max"] + 1) > 1e12:
            c.update(K=max(16, c["K"] // 2), k_max=max(4, c["k_max"] * 3 // 4))
        return c
    if kind == "step":
        c = dict(STEP, P=rng.randint(1, 4), K=_log(rng, 16, 1024), N=_log(rng, 200, 4096), M=_log(rng, 500, 65536),
                 grid=rng.randint(24, 96), k=rng.randint(0, 99), radius=rng.uniform(0.03, 0.15),
                 table=rng.choice([0, 0, _log(rng, 200, 4000)]))
        while c["P"] * c["K"] * c["N"] * c["M"] > 4e11:
            c["K"] = max(16, c["K"] // 2)
        return c
    if kind == "match":
        c = dict(kind="match", P=rng.randint(1, 4), K=_log(rng, 8, 256), N=_log(rng, 100, 4096), M=_log(rng, 300, 65536),
                 radius=rng.uniform(0.03, 0.15))
        while c["P"] * c["K"] * c["N"] * c["M"] > 4e11:
            c["K"] = max(8, c["K"] // 2)
        return c
    P, points = rng.randint(1, 4), _log(rng, 256, 8192)
    if kind == "propose":
        return dict(kind="propose", P=P, B=_log(rng, 1, 64), points=points, K=_log(rng, 16, 512))
    return dict(kind="train", P=P, B=_log(rng, 2, 48), points=min(points, 3000), T=rng.randint(4, 64))


# ---------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _sdf(tilt, grid):
    return synth.sdf_grid(tilt, grid)


def _gripper(case, seed):
    """Contact clouds (a new sampling per seed) and the gripper's distance fields (one hand)."""
    P = case["P"]
    tilts = synth.DEFAULT_TILTS_DEG[:P] if P <= 3 else [20.0 * p / (P - 1) for p in range(P)]
    S = [synth.gripper_contact_cloud(case["N"], t, 5 * seed + 17 * p + 1) for p, t in enumerate(tilts)]
    return S, [_sdf(t, case["grid"]) if "grid" in case else None for t in tilts]


def _cloud(m, seed, box=False):
    return (synth.box_object(m, seed) if box else synth.partial_object(m, seed)).points


def _poses(g, n, centre, radius):
    """n poses around a point: positions scattered about a sphere, any rotation."""
    u = g.normal(size=(n, 3))
    t = centre + u / np.linalg.norm(u, axis=1, keepdims=True) * radius * g.uniform(0.5, 1.2, (n, 1))
    q = g.normal(size=(n, 4))
    return np.concatenate([t, q / np.linalg.norm(q, axis=1, keepdims=True)], 1).astype(np.float32)


def _inputs(case, seed):
    g = np.random.default_rng([seed, 11])
    x = {}
    if case["kind"] in ("propose", "train"):
        x["params"] = synth.proposal_params(case["P"], seed + 7)
        x["clouds"] = np.stack([_cloud(case["points"], 31 * seed + b) for b in range(case["B"])])
        if case["kind"] == "propose":
            n = (case["B"], case["P"], case["K"])
            x["draws"] = np.concatenate([g.uniform(0, 1, n + (1,)), g.normal(size=n + (7,))], -1).astype(np.float32)
        else:
            tg = [_poses(g, case["P"] * case["T"], c.mean(0, dtype=np.float64), 0.08) for c in x["clouds"]]
            x["targets"] = np.stack(tg).reshape(case["B"], case["P"], case["T"], 7)
        return x
    x["S"], x["sdf"] = _gripper(case, seed)
    n_obj, P, K = case.get("objects", 1), case["P"], case["K"]
    Ms, x["K"] = [case["M"]] * n_obj, np.full(n_obj * P, K, np.int32)
    if case.get("uneven"):                           # the sizes are the case's, the points the seed's
        sizes = np.random.default_rng(n_obj)
        Ms = [int(case["M"] / 32.0 ** u) + 1 for u in sizes.uniform(0, 1, n_obj)]
        x["K"] = sizes.choice(np.array([K // 4, K // 2, K], np.int32), size=n_obj * P).astype(np.int32)
    small_box = case["kind"] == "run" and case["M"] == 512 and n_obj == 1
    x["R"] = [_cloud(int(m), 1009 * seed + o, small_box) for o, m in enumerate(Ms)]
    x["C"] = [np.concatenate([r, synth.table_points(case["table"], r, seed + 3)]) if case.get("table") else None for r in x["R"]]
    per_obj = x["K"].reshape(n_obj, P).sum(1)
    if case["kind"] != "run" or case["given"]:
        x["theta"] = np.concatenate([_poses(g, int(k), r.mean(0, dtype=np.float64), case["radius"]) for k, r in zip(per_obj, x["R"])])
    if case.get("minibatch"):
        x["ramp"] = synth.minibatch_ramp(case["M"], case["k_max"], seed + 5)
    return x


def _k_stein(case):
    k = case.get("k_stein", -1)
    return synth.k_stein_for(case["k_max"]) if k < 0 else k


# ---------------------------------------------------------------------------- preparing and running
class _State:
    """What the caller keeps between passes; the handle goes with it."""
    ctx = net = None

    def __del__(self):
        if self.ctx:
            asicp.asicp_destroy(self.ctx)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    x, s = _inputs(case, seed), _State()
    s.case = case
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] in ("propose", "train"):
        s.net = proposal.Proposal(case["P"], case["points"], case["B"], stream)
        s.net.set_params(x["params"])
        s.x = {k: v for k, v in x.items() if k != "params"}
        return s
    if case["kind"] == "match":
        s.theta, s.S, s.R = _dev(x["theta"]), _dev(np.concatenate(x["S"])), _dev(x["R"][0])
        s.out = torch.empty(case["P"] * case["K"] * case["N"], dtype=torch.int32, device="cuda")
        return s
    cfg = asicp.asicp_config_default(P=case["P"], K=case["K"], k_max=case["k_max"], k_stein=_k_stein(case),
                                     schedule=case.get("schedule", 0), init_radius=case["radius"],
                                     conv_tol=2e-4 if case.get("freeze") else -1.0, cuda_stream=stream,
                                     n_objects=case.get("objects", 1), fwd_shape=case["shape"])
    s.ctx = asicp.asicp_create(cfg)
    if case.get("uneven"):
        asicp.asicp_set_particle_counts(s.ctx, x["K"])
    for p, (S, (sdf, origin, voxel)) in enumerate(zip(x["S"], x["sdf"])):
        asicp.asicp_set_gripper_sdf(s.ctx, p, S, sdf, origin, voxel)
    s.n = [int(k) for k in x["K"].reshape(-1, case["P"]).sum(1)]
    s.ramp = x.get("ramp")
    s.theta = x.get("theta")
    host = case.get("host", True)
    s.clouds = [(r if host else _dev(r), c if host or c is None else _dev(c)) for r, c in zip(x["R"], x["C"])]
    if case["kind"] == "step":
        asicp.asicp_set_object(s.ctx, *s.clouds[0])
    return s


def run(s):
    case = s.case
    if case["kind"] == "run":
        for o, (R, C) in enumerate(s.clouds):
            asicp.asicp_set_object_at(s.ctx, o, R, C)
        if s.ramp is not None:
            asicp.asicp_set_minibatch(s.ctx, *s.ramp)
        asicp.asicp_run(s.ctx, s.theta)
        out = []
        for o, n in enumerate(s.n):
            theta, cost, pre = np.empty((n, 7), np.float32), np.empty(n, np.float32), np.empty(n, np.int32)
            asicp.asicp_best_grasps_at(s.ctx, o, n, theta, cost, pre)
            out.append({"cost": cost, "preshape": pre, "theta": theta})
        return out
    if case["kind"] == "step":
        n = s.n[0]
        asicp.asicp_set_state(s.ctx, s.theta, case["k"])
        asicp.asicp_step(s.ctx, case["k"])
        out = {"theta": np.empty((n, 7), np.float32), "cost": np.empty(n), "grad": np.empty((n, 7)),
               "phi": np.empty((n, 7), np.float32), "ncol": np.empty(n, np.int32), "frozen": np.empty(n, np.int32),
               "h": np.empty(case["P"], np.float32)}
        asicp.asicp_get_state(s.ctx, **out)
        return out
    if case["kind"] == "match":
        asicp.asicp_match_noalloc(s.theta, s.S, s.R, s.out, case["P"], case["K"], torch.cuda.current_stream().cuda_stream)
        return s.out
    B, x = case["B"], s.x
    if case["kind"] == "propose":
        out, cen = s.net.forward(x["clouds"], B)
        return {"mixture": out, "centroid": cen, "theta": s.net.sample(out, cen, B, case["K"], x["draws"])}
    loss, grad = s.net.loss_grad(x["clouds"], x["targets"], B, case["T"], want_grad=True)
    s.net.adam_step(1e-3)
    return {"loss": loss, "grad": grad, "params": s.net.get_params()}


def work(case):
    """Linear in the points: any exact nearest-neighbour search has to transform each gripper point, form
    one distance and add its pair to the sums, and to map each collision point into the gripper frame
    and test it; how many distances it forms beyond that is the algorithm's affair."""
    if case["kind"] in ("propose", "train"):
        rows, head = case["B"] * case["points"], case["B"] * (256 * 256 + 256 * case["P"] * 160)
        params = proposal.num_params(case["P"])
        fwd = 2.0 * (rows * (3 * 64 + 64 * 128 + 128 * 256) + head)
        if case["kind"] == "propose":
            n = case["B"] * case["P"]
            return {"bytes": 4.0 * (params + 3 * rows + 160 * n + n * case["K"] * 15), "flops": fwd}
        # the max-pool passes gradients to at most 256 points of a cloud
        live = case["B"] * min(case["points"], 256)
        back = 4.0 * (live * (3 * 64 + 64 * 128 + 128 * 256) + head)
        return {"bytes": 4.0 * (7 * params + 3 * rows + case["B"] * case["P"] * case["T"] * 7), "flops": fwd + back}
    pairs, tests = case["P"] * case["K"] * case["N"], case["P"] * case["K"] * (case["M"] + case.get("table", 0))
    clouds = 12.0 * (case["P"] * case["N"] + case["M"] + case.get("table", 0))
    if case["kind"] == "match":
        return {"bytes": clouds + 28.0 * case["P"] * case["K"] + 4.0 * pairs, "flops": 26.0 * pairs}
    share = (7 / 12 if case.get("uneven") else 1.0) * case.get("objects", 1)
    points = 0.29 if case.get("uneven") else 1.0        # mean cloud of a log-uniform draw over a factor of 32
    passes = case["k_max"] + 1 if case["kind"] == "run" else 1
    grids = 4.0 * case["P"] * case["grid"] ** 3
    return {"bytes": clouds * case.get("objects", 1) + grids + 32.0 * case["P"] * case["K"] * share,
            "flops": passes * share * (52.0 * pairs + 40.0 * tests * points)}


# ---------------------------------------------------------------------------- the method in float64
def _t64(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().double()


def _f32(t):
    return t.float().double()


def _rot(q):
    w, x, y, z = q.unbind(-1)
    a = w * w - x * x - y * y - z * z
    return torch.stack([a + 2 * x * x, 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), a + 2 * y * y, 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), a + 2 * z * z], -1).reshape(q.shape[:-1] + (3, 3))


def _nearest(q, r):
    """Index of the nearest of r [M, 3] for every row of q [n, 3]."""
    w, out = (r * r).sum(1), []
    step = max(1, (1 << 28) // len(r))
    for a in range(0, len(q), step):
        out.append(torch.addmm(w, q[a:a + step], r.T, alpha=-2.0).argmin(1))
    return torch.cat(out)


def _inside(sdf, origin, voxel, x):
    """Trilinear value of the distance field at x [..., 3] is positive (outside the grid: no)."""
    dims = torch.tensor(sdf.shape[::-1], device=x.device)
    u = (x - origin) / voxel
    ok = ((u >= 0) & (u <= dims - 1)).all(-1)
    i = torch.minimum(u.floor().clamp(min=0).long(), dims - 2)
    f = u - i
    nx, ny = int(dims[0]), int(dims[1])
    flat, base, v = sdf.reshape(-1), (i[..., 2] * ny + i[..., 1]) * nx + i[..., 0], 0.0
    for c in range(8):
        d = [(c >> k) & 1 for k in range(3)]
        wgt = math.prod((f[..., k] if d[k] else 1 - f[..., k]) for k in range(3))
        v = v + wgt * flat[base + (d[2] * ny + d[1]) * nx + d[0]]
    return ok & (v > 0)


def _evaluate(th, S, sdf, R, C, com):
    """Cost [K], gradient [K, 7] and number of colliding points [K] of one preshape's poses."""
    t, q, N = th[:, :3], th[:, 3:], len(S)
    rot, tcp = _rot(q), S.mean(0)
    x = torch.einsum("kab,nb->kna", rot, S) + t[:, None]
    e = x - R[_nearest(x.reshape(-1, 3), R)].reshape(x.shape)
    ec = rot @ tcp + t - com
    se2 = (e * e).sum((1, 2)) + (ec * ec).sum(1)
    Se = e.sum(1) + ec
    E = torch.einsum("kna,nb->kab", e, S) + ec[:, :, None] * tcp
    cnt = torch.full((len(th),), float(N), device=th.device, dtype=torch.float64)
    hit, step = [], max(1, (1 << 22) // len(C))
    for a in range(0, len(th), step):
        local = torch.einsum("kba,kmb->kma", rot[a:a + step], C - t[a:a + step, None])
        hit.append(_inside(*sdf, local))
    hit = torch.cat(hit)
    ncol = hit.sum(1)
    for k in ncol.nonzero()[:, 0].tolist():
        c = C[hit[k]]
        i = _nearest(c, x[k])
        e1 = x[k][i] - c
        se2[k], Se[k], E[k], cnt[k] = (e1 * e1).sum(), e1.sum(0), e1.T @ S[i], float(len(c))
    w, v = q[:, :1], q[:, 1:]
    tr = E.diagonal(dim1=1, dim2=2).sum(1, keepdim=True)
    axial = torch.stack([E[:, 2, 1] - E[:, 1, 2], E[:, 0, 2] - E[:, 2, 0], E[:, 1, 0] - E[:, 0, 1]], 1)
    gw = 2 * w * tr + 2 * (v * axial).sum(1, keepdim=True)
    gv = -2 * v * tr + 2 * ((E @ v[:, :, None])[:, :, 0] + (E.mT @ v[:, :, None])[:, :, 0]) + 2 * w * axial
    gq = torch.cat([gw, gv], 1) / cnt[:, None]
    gq = gq - (gq * q).sum(1, keepdim=True) * q
    return se2 / cnt, torch.cat([Se / cnt[:, None], gq], 1), ncol


def _stein(th, grad, gamma, N):
    """Bandwidth and Stein direction of one preshape's poses."""
    K, t, q = len(th), th[:, :3], th[:, 3:]
    d2 = ((t[:, None] - t[None]) ** 2).sum(2)
    h = 1.0
    if K > 1:
        i, j = torch.triu_indices(K, K, 1, device=th.device)
        h = max(float(d2[i, j].sort().values[(K * (K - 1) // 2 - 1) // 2]) / math.log(K), 1e-12)
    kt, drive = torch.exp(-d2 / h), -gamma * N * grad
    ft = kt @ drive[:, :3] + 2 / h * (kt.sum(1, keepdim=True) * t - kt @ t)
    c = q @ q.T
    sign = torch.where(c < 0, -1.0, 1.0).sum(1, keepdim=True)
    fq = (c @ drive[:, 3:] + sign * q) / K
    return h, torch.cat([ft / K, fq - (fq * q).sum(1, keepdim=True) * q], 1)


def _moved(th, d, eta):
    th = th + eta * d
    return _f32(torch.cat([th[:, :3], th[:, 3:] / th[:, 3:].norm(dim=1, keepdim=True)], 1))


def _gamma(case, k):
    period = case["k_max"] / 5.0
    return float(np.float32((math.fmod(k, period) / period) ** 2))


def _exact_step(case, x):
    P, K, N = case["P"], case["K"], case["N"]
    R = _t64(x["R"][0])
    C = R if x["C"][0] is None else _t64(x["C"][0])
    got = {"theta": [], "cost": [], "grad": [], "phi": [], "h": []}
    for p in range(P):
        th = _t64(x["theta"][p * K:(p + 1) * K])
        th = _f32(torch.cat([th[:, :3], th[:, 3:] / th[:, 3:].norm(dim=1, keepdim=True)], 1))
        sdf, origin, voxel = x["sdf"][p]
        parts, step = [], max(1, (1 << 21) // N)
        for a in range(0, K, step):
            parts.append(_evaluate(th[a:a + step], _t64(x["S"][p]), (_t64(sdf), _t64(origin), float(voxel)), R, C, R.mean(0)))
        cost, grad = torch.cat([v[0] for v in parts]), torch.cat([v[1] for v in parts])
        h, phi = _stein(th, grad, _gamma(case, case["k"]), N)
        if case["k"] < _k_stein(case):
            th = _moved(th, phi, float(np.float32(1.0 / N)))
        else:
            h, phi, th = 0.0, torch.zeros_like(phi), _moved(th, -grad, 1.0)
        for key, v in (("theta", th), ("cost", cost), ("grad", grad), ("phi", phi), ("h", torch.tensor([h], dtype=torch.float64, device="cuda"))):
            got[key].append(v)
    return {**{k: torch.cat(v) for k, v in got.items()}, "ncol": None, "frozen": None}


def _exact_net(case, x):
    """The network in float64 on the weights and activations it stores (bfloat16), gradients passed
    straight through the rounding; ties of the max-pool go to the lowest point."""
    dims, at, W = [(64, 3), (128, 64), (256, 128), (256, 256), (case["P"] * 160, 256)], 0, []
    for o, i in dims:
        for shape in ((o, i), (o,)):
            n = math.prod(shape)
            v = torch.from_numpy(x["params"][at:at + n].reshape(shape)).cuda()
            W.append((v.bfloat16() if len(shape) == 2 else v).double().requires_grad_())
            at += n

    def kept(v):
        return v + (v.float().bfloat16().double() - v).detach()

    outs, cens, loss = [], [], 0.0
    for b, cloud in enumerate(x["clouds"]):
        pts = _t64(cloud)
        cen = pts.mean(0)
        hid = kept(pts - cen)
        for layer in range(3):
            hid = kept(torch.relu(hid @ W[2 * layer].T + W[2 * layer + 1]))
        top = hid.detach().amax(0)
        rows = torch.arange(len(hid), device="cuda")[:, None]
        first = torch.where(hid.detach() == top, rows, len(hid)).amin(0)
        pooled = hid[first, torch.arange(256, device="cuda")]
        z = kept(torch.relu(pooled @ W[6].T + W[7]))
        o = (z @ W[8].T + W[9]).reshape(case["P"], 16, 10)
        outs.append(o.detach())
        cens.append(cen)
        if case["kind"] == "train":
            tg = _t64(x["targets"][b])
            logpi = torch.log_softmax(o[..., 0], -1)
            sigma, kappa = 0.1 * torch.exp(o[..., 4].clamp(-4, 1)), 4 * torch.exp(o[..., 9].clamp(-2, 3))
            nu = o[..., 5:9] / o[..., 5:9].norm(dim=-1, keepdim=True).clamp(min=1e-6)
            d2 = ((tg[:, :, None, :3] - _f32(cen) - 0.1 * o[:, None, :, 1:4]) ** 2).sum(-1)
            dot = torch.einsum("ptk,pck->ptc", tg[..., 3:], nu)
            term, series = torch.ones_like(kappa), torch.ones_like(kappa)
            for n in range(400):                     # Kummer's M(1/2, 2, kappa)
                term = term * (0.5 + n) / (2.0 + n) * kappa / (n + 1)
                series = series + term
            ell = (logpi - 3 * torch.log(sigma) - torch.log(series))[:, None] - d2 / (2 * sigma[:, None] ** 2) + kappa[:, None] * dot ** 2
            loss = loss - (torch.logsumexp(ell, -1) - 1.5 * math.log(2 * math.pi) - math.log(2 * math.pi ** 2)).mean() / case["B"]
    if case["kind"] == "propose":
        o, cen = torch.stack(outs), torch.stack(cens)
        draws = _t64(x["draws"])
        cdf = torch.softmax(o[..., 0], -1).cumsum(-1)
        pick = (cdf[:, :, None] <= draws[..., :1]).sum(-1).clamp(max=15)
        oc = torch.gather(o, 2, pick[..., None].expand(-1, -1, -1, 10))
        t = cen[:, None, None] + 0.1 * oc[..., 1:4] + 0.1 * torch.exp(oc[..., 4:5].clamp(-4, 1)) * draws[..., 1:4]
        q = oc[..., 5:9] / oc[..., 5:9].norm(dim=-1, keepdim=True).clamp(min=1e-6)
        q = q + draws[..., 4:] / torch.sqrt(8 * torch.exp(oc[..., 9:].clamp(-2, 3)))
        return {"mixture": o, "centroid": cen, "theta": torch.cat([t, q / q.norm(dim=-1, keepdim=True)], -1)}
    grad = torch.cat([g.reshape(-1) for g in torch.autograd.grad(loss, W)])
    return {"loss": float(loss.detach()), "grad": grad, "params": _t64(x["params"]) - 1e-3 * grad / (grad.abs() + 1e-8)}


def exact(case, seed):
    if case["kind"] in ("run", "match"):
        # indices have to be equal anyway, and a whole run has no such value: its particles pass through
        # near-tied correspondences and collision flags, where a rounding decides which way they go (each
        # single iteration, from given poses, has one)
        return None
    x = _inputs(case, seed)
    return _exact_step(case, x) if case["kind"] == "step" else _exact_net(case, x)
