"""The calls whose speed is measured, and the inputs they are measured on.

Every case goes through the public entry points of paper_2204_03139_gb300, as a program that
fits cloth parameters to observed point clouds uses them: single calls on trajectories, the
autograd loss, plain point clouds, batches of uneven trajectories, and the pipeline from and to
host memory. Sizes are those of the repository's workloads and tests. Inputs are made on the GPU
from the seed: a square cloth whose corner is lifted along an arc, seeded uniform draws, and
target clouds with sensor noise and outliers taken from a copy of the motion with other
parameters. `fit` says how far those parameters are off: 0.1 (the workloads' value) is late in an
optimisation, larger values its start.
"""
import math

import numpy as np
import torch

from paper_2204_03139_gb300 import (BIDIR_MEAN, UNIDIR_SUM, dc_chamfer_bwd, dc_chamfer_fwd,
                                    dc_loss_traj, dc_sample)
from paper_2204_03139_gb300.autograd import loss_traj
from paper_2204_03139_gb300.batch import BatchedLoss, DeviceTrajectory
from paper_2204_03139_gb300.pipeline import LossPipeline

DEV = "cuda:0"
MODES = {"eq1": BIDIR_MEAN, "eq2": UNIDIR_SUM}


def listed():
    return [
        # the smallest call: one frame of a coarse mesh, loss, gradient and neighbours; a fit to
        # one observed frame makes one such call per optimiser step
        {"name": "single_frame", "kind": "call", "T": 1, "grid": 25, "N": 2048, "M": 2048,
         "mode": "eq1", "fit": 0.1, "nn": True},
        # one frame of a fine mesh against a dense merged cloud
        {"name": "dense_frame", "kind": "call", "T": 1, "grid": 100, "N": 32768, "M": 32768,
         "mode": "eq1", "fit": 0.1, "nn": True},
        # the ordinary call: a whole recorded trajectory, bidirectional loss and gradient
        {"name": "trajectory", "kind": "call", "T": 40, "grid": 50, "N": 10000, "M": 10000,
         "mode": "eq1", "fit": 0.1, "nn": True},
        # the same in the one-directional form, without returning the neighbours
        {"name": "trajectory_eq2", "kind": "call", "T": 40, "grid": 50, "N": 10000, "M": 10000,
         "mode": "eq2", "fit": 0.1, "nn": False},
        # one optimiser step on the last frame only, at the start of a fit (parameters far off),
        # forward and backward through autograd; frames of weight 0 cost nothing
        {"name": "last_frame_step", "kind": "autograd", "T": 40, "grid": 50, "N": 10000,
         "M": 10000, "mode": "eq1", "fit": 0.5, "last": True},
        # forward and backward through autograd on the largest single trajectory
        {"name": "autograd_large", "kind": "autograd", "T": 100, "grid": 100, "N": 32768,
         "M": 32768, "mode": "eq1", "fit": 0.1, "last": False},
        # Chamfer distance and its gradient of clouds that the caller sampled, odd sizes
        {"name": "clouds_odd", "kind": "clouds", "T": 7, "N": 4097, "M": 3001, "mode": "eq1",
         "fit": 0.1, "volume": False},
        # the sampler alone, on the visible half of the cloth: points, faces and weights
        {"name": "sample_half", "kind": "sample", "T": 40, "grid": 50, "N": 10000, "half": True},
        # many optimisations at once: a planned batch of uneven trajectories, run again and again
        {"name": "batch_uneven", "kind": "batch", "traj": 64, "grid_lo": 15, "grid_hi": 80,
         "T_lo": 20, "T_hi": 100, "M_lo": 2000, "M_hi": 30000, "sizes": 1, "mode": "eq1",
         "graph": True},
        # a batch as a server forms it: other trajectories every time, planned and run once
        {"name": "batch_formed", "kind": "form", "traj": 6, "grid_lo": 15, "grid_hi": 50,
         "T_lo": 5, "T_hi": 40, "M_lo": 1000, "M_hi": 10000, "sizes": 2, "mode": "eq1"},
        # from pinned host memory to pinned host memory: what a caller without device data pays
        {"name": "host_pipeline", "kind": "pipeline", "T": 40, "grid": 50, "N": 10000,
         "M": 10000, "mode": "eq1", "fit": 0.1},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the same kinds over the whole range of frame counts, meshes and clouds."""
    kind = rng.choice(["call", "call", "call", "autograd", "autograd", "clouds", "clouds",
                       "sample", "batch", "form", "pipeline"])
    mode = rng.choice(["eq1", "eq1", "eq2"])
    if kind in ("batch", "form"):
        c = {"kind": kind, "traj": _log(rng, 2, 24), "grid_lo": 15, "grid_hi": rng.randint(20, 80),
             "T_lo": rng.randint(1, 20), "T_hi": rng.randint(20, 60),
             "M_lo": rng.randint(500, 2000), "M_hi": _log(rng, 2500, 30000),
             "sizes": rng.randrange(1 << 20), "mode": mode}
        if kind == "batch":
            c["graph"] = rng.random() < 0.5
        return c
    c = {"kind": kind, "T": _log(rng, 1, 100)}
    if kind != "clouds":
        c["grid"] = _log(rng, 8, 110)
    c["N"] = _log(rng, 300, 33000)
    if kind == "sample":
        c["half"] = rng.random() < 0.5
        return c
    c["M"] = c["N"] if rng.random() < 0.3 else _log(rng, 300, 33000)
    c["mode"] = mode
    c["fit"] = round(math.exp(rng.uniform(math.log(0.02), math.log(0.6))), 3)
    if kind == "call":
        c["nn"] = rng.random() < 0.5
    elif kind == "autograd":
        c["last"] = rng.random() < 0.3
    elif kind == "clouds":
        c["volume"] = rng.random() < 0.4
    return c


# ---- inputs -----------------------------------------------------------------------------------
def _faces(n):
    ix, iy = np.meshgrid(np.arange(n - 1), np.arange(n - 1), indexing="xy")
    a = (iy * n + ix).ravel()
    f = np.empty((2 * a.size, 3), np.int32)
    f[0::2] = np.stack([a, a + 1, a + n + 1], axis=1)
    f[1::2] = np.stack([a, a + n + 1, a + n], axis=1)
    return f


def _motion(u, v, s, a, lift):
    """Points (u, v) of the cloth at phase s (broadcast) of the lift: the grasped corner follows
    an arc, the rest hangs below it as a catenary of parameter a."""
    cz = lift * (0.6 * s - 0.1 * s * s)
    rho = torch.hypot(u, v)
    h = torch.clamp(cz - a * (torch.cosh(rho / a) - 1.0), min=0.0)
    inv = torch.where(rho > 0, 1.0 / rho.clamp(min=1e-12), torch.zeros_like(rho))
    pull = torch.minimum(0.5 * h, 0.5 * rho)
    frac = torch.where(cz > 0, h / cz.clamp(min=1e-12), torch.zeros_like(h))
    return torch.stack([u - pull * u * inv + frac * 0.2 * s, v - pull * v * inv + frac * 0.2 * s,
                        h], dim=-1)


def _phase(T):
    s = torch.arange(T, dtype=torch.float64, device=DEV) / (T - 1) if T > 1 else \
        torch.ones(1, dtype=torch.float64, device=DEV)
    return s[:, None]


def _verts(gen, T, grid, a=0.35, lift=1.0):
    g = torch.linspace(0.0, 1.0, grid, dtype=torch.float64, device=DEV)
    v, u = torch.meshgrid(g, g, indexing="ij")
    p = _motion(u.reshape(1, -1), v.reshape(1, -1), _phase(T), a, lift)
    p = p + 1e-3 * torch.randn(p.shape, generator=gen, dtype=torch.float64, device=DEV)
    return p.float().contiguous()


def _areas(verts, faces, mask=None):
    """[T, F] float64 face areas (0 outside the mask)."""
    p = verts.double()[:, faces.long()]
    area = 0.5 * torch.linalg.cross(p[:, :, 1] - p[:, :, 0], p[:, :, 2] - p[:, :, 0]).norm(dim=2)
    return area if mask is None else area * (mask != 0)


def _draws(gen, n, verts, faces, mask=None):
    """[T, n, 3] uniform draws. A draw within 1e-6 of a boundary between two faces, where the
    picked face is a matter of rounding, is moved to the middle of its face's interval."""
    r = torch.rand(verts.shape[0], n, 3, generator=gen, device=DEV).clamp_(max=1 - 2 ** -24)
    cdf = torch.cumsum(_areas(verts, faces, mask), 1)
    cdf = torch.cat([torch.zeros_like(cdf[:, :1]), cdf / cdf[:, -1:]], 1)
    u = r[..., 0].double()
    f = torch.searchsorted(cdf, u, right=True).clamp(1, cdf.shape[1] - 1)
    lo, hi = cdf.gather(1, f - 1), cdf.gather(1, f)
    near = torch.minimum(u - lo, hi - u) < 1e-6
    r[..., 0] = torch.where(near, 0.5 * (lo + hi), u).float()
    return r


def _cloud(gen, T, m, fit, a=0.35, lift=1.0, noise=2e-3, outliers=0.03):
    """[T, m, 3] observed clouds of the motion with parameters off by `fit`."""
    uv = torch.rand(2, T, m, generator=gen, dtype=torch.float64, device=DEV)
    p = _motion(uv[0], uv[1], _phase(T), (1.0 + fit) * a, (1.0 - 0.5 * fit) * lift)
    p = p + noise * torch.randn(p.shape, generator=gen, dtype=torch.float64, device=DEV)
    if outliers > 0:
        lo, hi = p.amin(1, keepdim=True), p.amax(1, keepdim=True)
        q = lo + (hi - lo) * torch.rand(p.shape, generator=gen, dtype=torch.float64, device=DEV)
        out = torch.rand(T, m, 1, generator=gen, device=DEV) < outliers
        p = torch.where(out, q, p)
    return p.float().contiguous()


def _sizes(case):
    """Per trajectory of a batch: (grid, T, M of every frame, catenary, lift). Each frame loses
    up to a fifth of its trajectory's points, as a depth camera's cloud does."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["traj"]):
        grid = int(rng.integers(case["grid_lo"], case["grid_hi"] + 1))
        T = int(rng.integers(case["T_lo"], case["T_hi"] + 1))
        m = int(rng.integers(case["M_lo"], case["M_hi"] + 1))
        ms = np.ceil(m * (1.0 - rng.uniform(0.0, 0.2, T))).astype(np.int64)
        out.append((grid, T, ms, float(rng.uniform(0.3, 0.4)), float(rng.uniform(0.8, 1.2))))
    return out


def _trajectories(case, gen):
    trajs = []
    for grid, T, ms, a, lift in _sizes(case):
        verts = _verts(gen, T, grid, a, lift)
        m_max = int(np.max(ms))
        y = _cloud(gen, T, m_max, 0.1, a, lift, noise=3e-3, outliers=0.0)
        # the points beyond a plane are missing: those furthest along a random direction
        d = torch.randn(T, 3, 1, generator=gen, dtype=torch.float64, device=DEV)
        rank = torch.bmm(y.double(), d)[..., 0].argsort(1).argsort(1)
        keep = rank < torch.as_tensor(ms, device=DEV)[:, None]
        off = np.concatenate([[0], np.cumsum(ms)]).astype(np.int64)
        faces = torch.from_numpy(_faces(grid)).to(DEV)
        draws = _draws(gen, m_max, verts, faces)[keep].contiguous()
        trajs.append(DeviceTrajectory(verts, faces, draws, y[keep].contiguous(), off, off))
    return trajs


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    kind = case["kind"]
    if kind in ("batch", "form"):
        return {"trajs": _trajectories(case, gen)}
    T, N = case["T"], case["N"]
    x = {}
    if kind == "clouds":
        if case["volume"]:
            x["a"] = torch.rand(T, N, 3, generator=gen, device=DEV)
            x["b"] = torch.rand(T, case["M"], 3, generator=gen, device=DEV)
        else:
            x["a"] = _cloud(gen, T, N, 0.0, noise=0.0, outliers=0.0)
            x["b"] = _cloud(gen, T, case["M"], case["fit"])
        x["g"] = torch.rand(T, generator=gen, device=DEV) + 0.5
        return x
    x["verts"] = _verts(gen, T, case["grid"])
    x["faces"] = torch.from_numpy(_faces(case["grid"])).to(DEV)
    if kind == "sample":
        n = case["grid"] - 1
        upper = np.repeat(np.arange(n) >= n // 2, 2 * n).astype(np.uint8)
        x["mask"] = torch.from_numpy(upper).to(DEV) if case["half"] else None
    x["draws"] = _draws(gen, N, x["verts"], x["faces"], x.get("mask"))
    if kind != "sample":
        x["targets"] = _cloud(gen, T, case["M"], case["fit"])
    if case.get("last"):
        x["weights"] = torch.zeros(T, device=DEV)
        x["weights"][-1] = 1.0
    return x


# ---- the measured calls -----------------------------------------------------------------------
def _flat_outputs(trajs):
    """One tensor for all trajectories' losses and one for their gradients, with the views that
    the batch writes into."""
    shapes = [(t.T, t.verts.shape[1]) for t in trajs]
    losses = torch.zeros(sum(T for T, _ in shapes), device=DEV)
    grads = torch.zeros(sum(T * V * 3 for T, V in shapes), device=DEV)
    views, i, j = [], 0, 0
    for T, V in shapes:
        views.append((losses[i:i + T], grads[j:j + T * V * 3].view(T, V, 3)))
        i, j = i + T, j + T * V * 3
    return losses, grads, views


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    kind = case["kind"]
    if kind in ("batch", "form"):
        state["losses"], state["grads"], state["views"] = _flat_outputs(state["trajs"])
    if kind == "batch":
        state["plan"] = BatchedLoss(state["trajs"], mode=MODES[case["mode"]], grad=True,
                                    graph=case["graph"], outputs=state["views"])
    if kind == "pipeline":
        T, N, M = case["T"], case["N"], case["M"]
        V, F = state["verts"].shape[1], state["faces"].shape[0]
        state["pipe"] = LossPipeline(T, V, F, N, M, device=DEV, mode=MODES[case["mode"]])
        for k in ("verts", "faces", "draws", "targets"):
            state[k] = state[k].cpu().pin_memory()
        state["grad_out"] = LossPipeline.pinned((T, V, 3))
        state["loss_out"] = LossPipeline.pinned((1,))
        state["frames_out"] = LossPipeline.pinned((T,))
    if kind == "autograd":
        state["verts"].requires_grad_(True)
    return state


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "call":
        r = dc_loss_traj(s["verts"], s["faces"], s["draws"], s["targets"],
                         mode=MODES[case["mode"]], nn=case["nn"])
        return [r["loss_total"], r["loss_frames"], r["grad_verts"], r["nn_ab"], r["nn_ba"]]
    if kind == "autograd":
        s["verts"].grad = None
        total, frames = loss_traj(s["verts"], s["faces"], s["draws"], s["targets"],
                                  mode=MODES[case["mode"]], frame_w=s.get("weights"))
        total.backward()
        return [total.detach(), frames.detach(), s["verts"].grad]
    if kind == "clouds":
        mode = MODES[case["mode"]]
        loss, nn_ab, nn_ba = dc_chamfer_fwd(s["a"], s["b"], mode=mode)
        grad = dc_chamfer_bwd(s["a"], s["b"], nn_ab, nn_ba, s["g"], mode=mode)
        return [loss, grad, nn_ab, nn_ba]
    if kind == "sample":
        points, face, bary = dc_sample(s["verts"], s["faces"], s["draws"], face_mask=s["mask"])
        return [points, bary, face]
    if kind == "batch":
        total = s["plan"].run()
        return [total, s["losses"], s["grads"]]
    if kind == "form":
        total = BatchedLoss(s["trajs"], mode=MODES[case["mode"]], grad=True, outputs=s["views"],
                            async_plan=True).run()
        return [total, s["losses"], s["grads"]]
    done = s["pipe"].submit(s["verts"], s["faces"], s["draws"], s["targets"], s["grad_out"],
                            s["loss_out"], s["frames_out"])
    done.synchronize()  # the caller reads the results on the host
    return [s["loss_out"], s["frames_out"], s["grad_out"]]


# ---- what a pass cannot do without ------------------------------------------------------------
def _frame_work(grid, N, M, mode, nn):
    """Bytes and floating-point operations of one frame: the mesh, the draws and the targets read
    once, the gradient (and the neighbours, if returned) written once; the area of every face, one
    point per draw, one squared distance per query point (that of its nearest neighbour: how the
    neighbour is searched is not part of the result) and its gradient on three vertices."""
    V, F = grid * grid, 2 * (grid - 1) ** 2
    q = N + (M if mode == "eq1" else 0)
    b = 12 * V + 12 * N + 12 * M + 12 * V + 4 + (4 * q if nn else 0)
    return b, 30 * F + 22 * N + (8 + 24) * q


def work(case):
    kind = case["kind"]
    b = f = 0
    if kind in ("batch", "form"):
        for grid, T, ms, _, _ in _sizes(case):
            b += 24 * (grid - 1) ** 2
            for m in ms:
                x = _frame_work(grid, int(m), int(m), case["mode"], False)
                b, f = b + x[0], f + x[1]
    elif kind == "clouds":
        T, N, M = case["T"], case["N"], case["M"]
        q = N + (M if case["mode"] == "eq1" else 0)
        # both clouds in, losses, neighbours and gradient out (the neighbours are an output)
        b = T * (12 * N + 12 * M + 4 * q + 12 * N + 4)
        f = T * (8 + 6) * q
    elif kind == "sample":
        T, N, V, F = case["T"], case["N"], case["grid"] ** 2, 2 * (case["grid"] - 1) ** 2
        b = 12 * F + (F if case["half"] else 0) + T * (12 * V + 12 * N + (12 + 12 + 4) * N)
        f = T * (30 * F + 22 * N)
    else:
        live = 1 if case.get("last") else case["T"]
        x = _frame_work(case["grid"], case["N"], case["M"], case["mode"], case.get("nn", False))
        # a frame of weight 0 only gets its zero gradient written
        b = 24 * (case["grid"] - 1) ** 2 + live * x[0] + \
            (case["T"] - live) * 12 * case["grid"] ** 2
        f = live * x[1]
    return {"bytes": float(b), "flops": float(f)}


# ---- the same in 64 bits ----------------------------------------------------------------------
def _exact_sample(verts, faces, draws, mask=None):
    """One frame in float64: points, faces and barycentric weights of the draws."""
    p = verts.double()[faces.long()]
    cdf = torch.cumsum(_areas(verts[None], faces, mask)[0], 0)
    r = draws.double()
    f = torch.searchsorted(cdf, r[:, 0] * cdf[-1], right=True).clamp(max=cdf.numel() - 1)
    sq = r[:, 1].sqrt()
    w = torch.stack([1 - sq, sq * (1 - r[:, 2]), sq * r[:, 2]], dim=1)
    return (w[:, :, None] * p[f]).sum(1), f, w


def _exact_nn(x, y, both):
    """Nearest neighbours of x in y (and of y in x), float64, by all pairs."""
    n, m = x.shape[0], y.shape[0]
    step = max(1, (1 << 27) // m)
    jab = []
    best = torch.full((m,), math.inf, dtype=torch.float64, device=x.device)
    jba = torch.zeros(m, dtype=torch.int64, device=x.device)
    for i in range(0, n, step):
        d = (x[i:i + step, None, 0] - y[None, :, 0]).square_()
        for k in (1, 2):
            d += (x[i:i + step, None, k] - y[None, :, k]).square_()
        jab.append(d.argmin(1))
        if both:
            v, j = d.min(0)
            jba = torch.where(v < best, j + i, jba)
            best = torch.minimum(best, v)
    return torch.cat(jab), jba


def _exact_cloud(x, y, mode):
    """Chamfer loss and its gradient with respect to x of one frame."""
    jab, jba = _exact_nn(x, y, mode == "eq1")
    dab = x - y[jab]
    if mode == "eq2":
        return dab.square().sum(), 2.0 * dab
    dba = x[jba] - y
    n, m = x.shape[0], y.shape[0]
    loss = dab.square().sum() / n + dba.square().sum() / m
    return loss, (2.0 / n * dab).index_add(0, jba, 2.0 / m * dba)


def _exact_frame(verts, faces, draws, targets, mode):
    x, f, w = _exact_sample(verts, faces, draws)
    loss, gx = _exact_cloud(x, targets.double(), mode)
    g = torch.zeros(verts.shape, dtype=torch.float64, device=verts.device)
    g.index_add_(0, faces.long()[f].reshape(-1), (w[:, :, None] * gx[:, None, :]).reshape(-1, 3))
    return loss, g


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "form"):
        pairs = sum(T * float(np.max(ms)) ** 2 for _, T, ms, _, _ in _sizes(case))
        if pairs > 2e11:
            return None
        losses, grads = [], []
        for t in _inputs(case, seed)["trajs"]:
            for k in range(t.T):
                a, b = int(t.n_off[k]), int(t.n_off[k + 1])
                x = _exact_frame(t.verts[k], t.faces, t.draws[a:b], t.targets[a:b], case["mode"])
                losses.append(x[0])
                grads.append(x[1].reshape(-1))
        losses = torch.stack(losses)
        return [losses.sum().reshape(1), losses, torch.cat(grads)]
    x = _inputs(case, seed)
    T = case["T"]
    if kind == "clouds":
        r = [_exact_cloud(x["a"][t].double(), x["b"][t].double(), case["mode"]) for t in range(T)]
        grad = torch.stack([q[1] for q in r]) * x["g"].double()[:, None, None]
        return [torch.stack([q[0] for q in r]), grad, None, None]
    if kind == "sample":
        r = [_exact_sample(x["verts"][t], x["faces"], x["draws"][t], x["mask"]) for t in range(T)]
        return [torch.stack([q[0] for q in r]), torch.stack([q[2] for q in r]), None]
    losses = torch.zeros(T, dtype=torch.float64, device=DEV)
    grad = torch.zeros(x["verts"].shape, dtype=torch.float64, device=DEV)
    for t in range(T - 1 if case.get("last") else 0, T):
        losses[t], grad[t] = _exact_frame(x["verts"][t], x["faces"], x["draws"][t],
                                          x["targets"][t], case["mode"])
    total = losses.sum()
    if kind == "call":
        return [total.reshape(1), losses, grad, None, None]
    if kind == "autograd":
        return [total, losses, grad]
    return [total.reshape(1), losses, grad]
