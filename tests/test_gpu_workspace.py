"""One workspace for several meshes: calls and plans on a workspace sized for a larger mesh, which
may be without the pruned search's regions (they are dropped where the faces outweigh the points)."""
import ctypes

import pytest
import torch

import oracle
import parity
import workloads as W
from paper_2204_03139_gb300 import _lib
from paper_2204_03139_gb300.batch import BatchedLoss, DeviceTrajectory

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
T, N, M = 57, 7008, 2689


def _ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


@pytest.fixture(scope="module")
def inputs():
    tr = W.lift_trajectory(77, 197, T, N, M, name="w")
    return DeviceTrajectory.from_host(tr, DEV)


@pytest.fixture(scope="module")
def small(inputs):
    """The workspace of a 200 x 200 mesh, too small for all regions of the 197 x 197 one."""
    nb = _lib.dc_workspace_size(T, 200 * 200, 2 * 199 * 199, N, M)
    assert nb < _lib.dc_workspace_size(T, 197 * 197, 2 * 196 * 196, N, M)
    return torch.empty(nb, dtype=torch.uint8, device=DEV)


def test_calls_on_the_workspace_of_a_larger_mesh(inputs, small):
    d = inputs
    draws, tgt = d.draws.view(T, N, 3), d.targets.view(T, M, 3)
    V, F = d.verts.shape[1], d.faces.shape[0]
    ref = _lib.dc_loss_traj(d.verts, d.faces, draws, tgt, check=True)
    o = {k: torch.empty_like(v) for k, v in ref.items()}
    L, st = _lib.lib(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    _lib._check(L.dc_loss_traj(_ptr(d.verts), _ptr(d.faces), None, _ptr(draws), _ptr(tgt), T, V, F,
                               N, M, 0, None, _ptr(o["loss_total"]), _ptr(o["loss_frames"]),
                               _ptr(o["grad_verts"]), _ptr(o["nn_ab"]), _ptr(o["nn_ba"]),
                               _ptr(small), small.numel(), st))
    _lib.check_ws(small)
    for k in ("loss_total", "loss_frames", "nn_ab", "nn_ba"):
        assert torch.equal(o[k], ref[k])
    assert parity.rel_l2(o["grad_verts"].cpu(), ref["grad_verts"].cpu()) < 1e-6
    one, g = torch.ones(1, device=DEV), torch.empty_like(ref["grad_verts"])
    _lib._check(L.dc_loss_traj_bwd(_ptr(d.verts), _ptr(d.faces), None, _ptr(draws), _ptr(tgt), T,
                                   V, F, N, M, 0, _ptr(ref["nn_ab"]), _ptr(ref["nn_ba"]), None,
                                   _ptr(one), None, _ptr(g), _ptr(small), small.numel(), st))
    _lib.check_ws(small)
    assert parity.rel_l2(g.cpu(), ref["grad_verts"].cpu()) < 2e-6


@pytest.mark.parametrize("staged", [False, True])
def test_plans_on_the_workspace_of_a_larger_mesh(inputs, small, staged):
    b = BatchedLoss([inputs])
    assert b.workspace_bytes > small.numel()
    total = b.run(check=True).clone()
    losses, grads = b.loss_frames[0].clone(), b.grad_verts[0].clone()
    b.loss_frames[0].zero_()
    b.grad_verts[0].zero_()
    L, st = _lib.lib(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    args = (b.frames, b.n_frames, 0, _ptr(small), small.numel())
    if staged:
        host = torch.empty(L.dc_batch_plan_bytes(b.frames, b.n_frames, 0), dtype=torch.uint8,
                           pin_memory=True)
        _lib._check(L.dc_batch_plan_async(*args, _ptr(host), host.numel(), st))
    else:
        _lib._check(L.dc_batch_plan(*args, st))
    out = torch.empty(1, device=DEV)
    _lib._check(L.dc_batch_run(_ptr(small), _ptr(out), st))
    _lib.check_ws(small)
    assert torch.equal(out, total) and torch.equal(b.loss_frames[0], losses)
    assert parity.rel_l2(b.grad_verts[0].cpu(), grads.cpu()) < 1e-6
    # without room for the other regions either it is refused as before
    assert L.dc_batch_plan(b.frames, b.n_frames, 0, _ptr(small), 1 << 20, st) == _lib.DC_ENOSPC


def test_server_admits_a_face_heavy_request_by_its_least_workspace():
    """A budget that holds the request without the pruned search's regions: it is served, and the
    running batch's bytes are given back."""
    from paper_2204_03139_gb300.serve import Server, _frames_of, request_bytes

    tr = parity.nudged(W.lift_trajectory(78, 197, T, N, M, name="r"))
    fr = _frames_of(tr)
    L = _lib.lib()
    least, full = (f(fr, tr.T) for f in (L.dc_batch_workspace_least, L.dc_batch_workspace_size))
    assert least < full
    need = request_bytes(tr)
    res = []
    for budget in (need + 1024, need + 2 * (full - least)):
        srv = Server(DEV, hbm_budget=budget)
        res.append(srv.submit(tr).result(timeout=120))
        srv.close()
        assert srv._used == 0 and srv._extra == 0
    ref = oracle.loss_traj(tr)
    for r in res:
        parity.check_loss(r.loss_frames, ref["loss_frames"])
        parity.check_grad(r.grad_verts, ref["grad_verts"])
    assert (res[0].loss_frames == res[1].loss_frames).all()


def test_the_engine_that_ran_is_told_and_tuning_records_no_other(inputs):
    """A problem whose faces outweigh its points keeps no regions of the pruned search: asked for, it
    runs the direct engine, which the workspace tells, and the tuner does not record it."""
    from paper_2204_03139_gb300 import autotune

    d = inputs
    v, y = d.verts, d.targets.view(T, M, 3)
    few = d.draws.view(T, N, 3)[:, :500].contiguous()
    with autotune.tuned(("pruned", 0)):
        _lib.dc_loss_traj(v, d.faces, few, y)
    assert _lib.ws_engine(_lib.workspace(1, DEV)) == _lib.ENGINE_DIRECT
    with autotune.tuned(("pruned", 0)):
        _lib.dc_chamfer_fwd(few[:1], y[:1])  # points only
    assert _lib.ws_engine(_lib.workspace(1, DEV)) == _lib.ENGINE_PRUNED
    shapes = (("pruned", 0), ("direct", 2))
    r = autotune.tune(v, d.faces, few, y, reps=1, save=False, shapes=shapes)
    assert r["best"] == ("direct", 2) and set(r["ms"]) == set(shapes)


@pytest.mark.parametrize("frames", [1, 32, 33, 57, 300])
def test_pruned_regions_are_kept_whatever_the_number_of_frames(frames):
    """Few points per frame, below the line of the default rule: asked for, the pruned search runs."""
    from paper_2204_03139_gb300 import autotune

    g = torch.Generator(device=DEV).manual_seed(frames)
    a, b = (torch.rand(frames, n, 3, generator=g, device=DEV) for n in (300, 411))
    out = []
    for shape, engine in ((("pruned", 0), _lib.ENGINE_PRUNED), (("direct", 0), _lib.ENGINE_DIRECT)):
        with autotune.tuned(shape):
            out.append(_lib.dc_chamfer_fwd(a, b, check=True))
        assert _lib.ws_engine(_lib.workspace(1, DEV)) == engine
    for x, y in zip(*out):
        assert torch.equal(x, y)
