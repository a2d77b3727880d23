"""The pruned search (sorted points, bounding boxes) against the oracle and the direct engine.

Neighbours are decided in the same float32 direct form with the lowest index among equal
distances, so they and the losses agree bit for bit; the sizes are the edges of its blocks (8,
64, 512 points), query tiles (32), cluster slices (from 1024 points per side) and counters (16 bit
up to 65 535 points)."""
import numpy as np
import pytest
import torch

import oracle
import parity
import workloads as W
from paper_2204_03139_gb300 import _lib, autotune

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PRUNED, DIRECT = ("pruned", 0), ("direct", 0)


def clouds(case, n, m):
    rng = np.random.default_rng(n * 7919 + m)
    a, b = rng.random((n, 3)), rng.random((m, 3))
    if case == "lattice":  # many exact ties
        a, b = np.round(a * 8) / 8, np.round(b * 8) / 8
    elif case == "one_point":
        a[:], b[:] = 0.5, 0.25
    elif case == "flat":
        a[:, 2] = b[:, 2] = 0.0
    elif case == "far":  # a few targets far away, and both clouds apart
        b[: max(1, m // 50)] *= 1e6
        a += 3.0
    elif case == "huge":
        a, b = a * 0.99e15, b * 0.99e15
    elif case == "tiny":
        a, b = a * 1e-18, b * 1e-18
    return a.astype(np.float32), b.astype(np.float32)


def nn(a, b, shape, mode):
    with autotune.tuned(shape):
        return _lib.dc_chamfer_fwd(torch.from_numpy(a[None]).to(DEV),
                                   torch.from_numpy(b[None]).to(DEV), mode=mode, check=True)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("n,m", [(1, 1), (1, 9), (7, 8), (31, 33), (63, 65), (511, 513),
                                 (1023, 1025), (2049, 4095), (4097, 1)])
def test_block_and_tile_edges_match_the_oracle(n, m, mode):
    a, b = clouds("cube", n, m)
    ref = oracle.nn_pair(a, b)
    loss, nab, nba = nn(a, b, PRUNED, mode)
    np.testing.assert_array_equal(nab[0].cpu().numpy(), ref["nn_ab"])
    if mode == 0:
        np.testing.assert_array_equal(nba[0].cpu().numpy(), ref["nn_ba"])
    parity.check_loss(loss.cpu().numpy()[:1], [oracle.chamfer(a, b, mode=mode)[0]])


@pytest.mark.parametrize("case", ["lattice", "one_point", "flat", "far", "huge", "tiny"])
def test_hard_clouds_match_the_oracle(case):
    a, b = clouds(case, 1500, 2100)
    ref = oracle.nn_pair(a, b)
    _, nab, nba = nn(a, b, PRUNED, 0)
    np.testing.assert_array_equal(nab[0].cpu().numpy(), ref["nn_ab"])
    np.testing.assert_array_equal(nba[0].cpu().numpy(), ref["nn_ba"])


@pytest.mark.parametrize("n,m", [(8193, 20000), (65535, 3000), (65536, 3000), (70001, 40003)])
def test_large_clouds_equal_the_direct_engine(n, m):
    a, b = clouds("cube", n, m)
    got, ref = nn(a, b, PRUNED, 0), nn(a, b, DIRECT, 0)
    for x, y in zip(got, ref):
        assert torch.equal(x, y)


@pytest.mark.parametrize("T", [1, 9, 19, 40])  # clusters of 8, 8, 4 and 2 CTAs
@pytest.mark.parametrize("mode", [0, 1])
def test_trajectories_equal_the_direct_engine(T, mode):
    tr = W.lift_trajectory(11 + T, 31, T, 8200, 5001, name="t")
    v, f = torch.from_numpy(tr.verts).to(DEV), torch.from_numpy(tr.faces).to(DEV)
    d, y = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
            for x in (tr.draws_tn3(), tr.targets_tm3()))
    w = torch.ones(T, device=DEV)
    w[T // 2] = 0.0 if T > 1 else 0.5
    mask = torch.from_numpy(W.upper_half_mask(31)).to(DEV) if T == 9 else None
    out = []
    for shape in (PRUNED, DIRECT):
        with autotune.tuned(shape):
            out.append(_lib.dc_loss_traj(v, f, d, y, mode=mode, frame_w=w, face_mask=mask,
                                         check=True))
    keys = ["loss_total", "loss_frames"]
    for k in keys:
        assert torch.equal(out[0][k], out[1][k])
    live = [t for t in range(T) if float(w[t]) != 0.0]  # a skipped frame has no neighbours
    for k in ["nn_ab"] + (["nn_ba"] if mode == 0 else []):
        assert torch.equal(out[0][k][live], out[1][k][live])
    assert parity.rel_l2(out[0]["grad_verts"].cpu(), out[1]["grad_verts"].cpu()) < 1e-6


def test_device_errors_reach_the_status():
    """A bad face index, a bad draw, a degenerate frame and a bad target, each in the last of
    three frames."""
    tr = W.lift_trajectory(5, 12, 3, 700, 600, name="e")
    for what, code in (("face", _lib.DC_EINVAL), ("draw", _lib.DC_EINVAL),
                       ("area", _lib.DC_EDEGENERATE), ("target", _lib.DC_EINVAL)):
        v, f = torch.from_numpy(tr.verts).clone(), torch.from_numpy(tr.faces).clone()
        d, y = (torch.from_numpy(np.ascontiguousarray(x)).clone()
                for x in (tr.draws_tn3(), tr.targets_tm3()))
        if what == "face":
            f[7, 1] = v.shape[1]
        elif what == "draw":
            d[2, 5, 0] = 1.5
        elif what == "area":
            v[2] = 0.25
        else:
            y[2, 9, 1] = float("nan")
        with autotune.tuned(PRUNED), pytest.raises(_lib.DCError) as e:
            _lib.dc_loss_traj(v.to(DEV), f.to(DEV), d.to(DEV), y.to(DEV), check=True)
        assert e.value.code == code


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("T,n,m", [(1, 1, 1), (1, 513, 255), (3, 1025, 257), (5, 2000, 3001),
                                   (2, 15745, 255), (2, 257, 15744), (103, 1025, 975)])
def test_recomputing_backward_equals_the_forward_gradient(T, n, m, mode):
    """dc_loss_traj_bwd with the neighbours of a forward call gives that call's gradient. Both sum
    the same float32 contributions in another order and grouping: a few roundings (6e-8) each."""
    tr = W.lift_trajectory(3, 13, T, n, m, name="b")
    v, f = torch.from_numpy(tr.verts).to(DEV), torch.from_numpy(tr.faces).to(DEV)
    d, y = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
            for x in (tr.draws_tn3(), tr.targets_tm3()))
    w = torch.linspace(0.0, 1.5, T, device=DEV) if T > 1 else None  # the first frame is skipped
    for shape in (PRUNED, DIRECT):
        with autotune.tuned(shape):
            r = _lib.dc_loss_traj(v, f, d, y, mode=mode, frame_w=w, check=True)
        g = _lib.dc_loss_traj_bwd(v, f, d, y, r["nn_ab"], r["nn_ba"], mode=mode, frame_w=w,
                                  grad_total=torch.ones(1, device=DEV), check=True)
        assert parity.rel_l2(g.cpu(), r["grad_verts"].cpu()) < 2e-6
    # a neighbour out of range is reported
    bad = r["nn_ab"].clone()
    bad[-1, -1] = m
    with pytest.raises(_lib.DCError) as e:
        _lib.dc_loss_traj_bwd(v, f, d, y, bad, r["nn_ba"], mode=mode, frame_w=w,
                              grad_total=torch.ones(1, device=DEV), check=True)
    assert e.value.code == _lib.DC_EINVAL


@pytest.mark.timeout(120)
def test_stall_test_runs_the_direct_engine_where_the_pruned_search_is_the_default():
    """The pruned search has no bounded waits to run out, so a pending stall test sends the call
    (or the run of a plan) that would take it to the direct engine, whose waits give up."""
    from paper_2204_03139_gb300.batch import BatchedLoss, DeviceTrajectory

    tr = W.lift_trajectory(6, 20, 40, 2000, 2100, name="s")
    v, f = torch.from_numpy(tr.verts).to(DEV), torch.from_numpy(tr.faces).to(DEV)
    d, y = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
            for x in (tr.draws_tn3(), tr.targets_tm3()))
    plan = BatchedLoss([DeviceTrajectory.from_host(tr, DEV)], shape=PRUNED)
    for run in (lambda: _lib.dc_loss_traj(v, f, d, y, check=True)["loss_frames"],
                lambda: (plan.run(check=True), plan.loss_frames[0])[1]):
        good = run().clone()
        _lib.test_inject_stall()
        with pytest.raises(_lib.DCError) as e:
            run()
        assert e.value.code == _lib.DC_ETIMEOUT
        assert torch.equal(run(), good)


@pytest.mark.parametrize("grid,engine", [(45, _lib.ENGINE_PRUNED), (182, _lib.ENGINE_DIRECT)])
def test_many_faces_per_point_leave_the_default_to_the_direct_engine(grid, engine):
    """16 frames of 4096 x 4096 points: with 1/2 face per point the pruned search is the default,
    with 8 its face records cost more than they save. The losses are the same either way."""
    tr = W.lift_trajectory(9, grid, 16, 4096, 4096, name="f")
    v, f = torch.from_numpy(tr.verts).to(DEV), torch.from_numpy(tr.faces).to(DEV)
    d, y = (torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
            for x in (tr.draws_tn3(), tr.targets_tm3()))
    ws = _lib.workspace(_lib.dc_workspace_size(16, v.shape[1], f.shape[0], 4096, 4096), DEV)
    r = _lib.dc_loss_traj(v, f, d, y, out={"ws": ws}, check=True)
    assert int(ws[52:56].cpu().view(torch.int32)[0]) == engine  # the header's engine word
    for shape in (PRUNED, DIRECT):
        with autotune.tuned(shape):
            ref = _lib.dc_loss_traj(v, f, d, y, check=True)
        for k in ("loss_frames", "loss_total", "nn_ab", "nn_ba"):
            assert torch.equal(r[k], ref[k])
        assert parity.rel_l2(r["grad_verts"].cpu(), ref["grad_verts"].cpu()) < 1e-6
