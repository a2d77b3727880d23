"""Clouds on which bounding boxes exclude little or nothing: the pruned search gives the direct
engine's neighbours and losses, in a time that stays within a factor of brute force.

Limit of the time: brute force in the pruned search's form evaluates the two directions separately
(the direct engine shares each distance between them) and at half the direct engine's rate or
more, with 1.5 for everything else: 6 times the direct engine."""
import numpy as np
import pytest
import torch

from paper_2204_03139_gb300 import _lib, autotune

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
PRUNED, DIRECT = ("pruned", 0), ("direct", 0)
T, N = 8, 10000


def clouds(case):
    rng = np.random.default_rng(3)
    a, b = rng.random((T, N, 3)), rng.random((T, N, 3))
    if case == "coincident":
        a[:], b[:] = 0.25, 0.25
    elif case == "mostly_coincident":  # as where clouds are padded with one point
        a[:, N // 10:], b[:, N // 10:] = 0.0, 0.0
    elif case == "tied":  # so far apart that all distances round to the same value
        a += 1e8
    elif case == "apart":
        a += 10.0
    elif case == "apart_along_x":
        a[..., 0] += 10.0
    elif case == "small_beside_large":
        a = 0.4 + 1e-3 * a
    elif case == "sphere_and_centre":  # equidistant, many of the distances exactly
        b -= 0.5
        b /= np.linalg.norm(b, axis=2, keepdims=True)
        a = 1e-4 * (a - 0.5)
    elif case == "sphere_and_inside":
        b -= 0.5
        b /= np.linalg.norm(b, axis=2, keepdims=True)
        a = 0.3 * (a - 0.5)
    elif case == "many_scales":  # around the origin, too dense there for the sort's cells
        a = 10 ** (-6 * rng.random((T, N, 1))) * (a - 0.5)
        b = 10 ** (-6 * rng.random((T, N, 1))) * (b - 0.5)
    elif case == "one_target":
        b[:] = 0.3
    elif case == "one_sim_point":
        a[:] = 0.3
    return (torch.from_numpy(x.astype(np.float32)).to(DEV) for x in (a, b))


def _time(fn):
    fn()
    best = float("inf")
    for _ in range(3):
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        start.record()
        fn()
        end.record()
        end.synchronize()
        best = min(best, start.elapsed_time(end))
    return best


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("case", ["coincident", "mostly_coincident", "tied", "apart", "apart_along_x",
                                  "small_beside_large", "one_target", "one_sim_point",
                                  "sphere_and_centre", "sphere_and_inside", "many_scales"])
def test_results_and_time_against_the_direct_engine(case, mode):
    a, b = clouds(case)
    out, ms = [], []
    for shape in (PRUNED, DIRECT):
        with autotune.tuned(shape):
            out.append(_lib.dc_chamfer_fwd(a, b, mode=mode, check=True))
            ms.append(_time(lambda: _lib.dc_chamfer_fwd(a, b, mode=mode)))
    for x, y in zip(*out):
        assert x is None and y is None or torch.equal(x, y)
    assert ms[0] < 6 * ms[1]


@pytest.mark.parametrize("n,m", [(2600, 2600), (2600, 33), (5000, 3001), (40, 9000)])
def test_walked_tiles_at_ragged_sizes(n, m):
    """Gradient too: equidistant clouds of sizes that leave ragged tiles and blocks."""
    rng = np.random.default_rng(n + m)
    x = rng.normal(size=(6, m, 3))
    y = torch.from_numpy((x / np.linalg.norm(x, axis=2, keepdims=True)).astype(np.float32)).to(DEV)
    v = torch.from_numpy((1e-3 * rng.normal(size=(6, 50, 3))).astype(np.float32)).to(DEV)
    f = torch.from_numpy(rng.permuted(np.tile(np.arange(50), (90, 1)), axis=1)[:, :3].astype(
        np.int32)).to(DEV)
    d = torch.from_numpy(rng.random((6, n, 3)).astype(np.float32)).to(DEV)
    out = []
    for shape in (PRUNED, DIRECT):
        with autotune.tuned(shape):
            out.append(_lib.dc_loss_traj(v, f, d, y, check=True))
    for k in ("loss_total", "loss_frames", "nn_ab", "nn_ba"):
        assert torch.equal(out[0][k], out[1][k])
    # The gradient in 64 bits, from the library's own samples and neighbours. Float32 sums of K terms
    # in any order are within K u sum |terms|: per vertex, K pairs reach it, each with a few roundings
    # of its own (difference, factor, weight).
    p, face, bary = (x.double() if x.is_floating_point() else x.long()
                     for x in _lib.dc_sample(v, f, d, check=True))
    nab, nba = out[0]["nn_ab"].long(), out[0]["nn_ba"].long()
    for t in range(v.shape[0]):
        yt, corners = y[t].double(), f.long()[face[t]].reshape(-1)
        ab, ba = 2.0 / n * (p[t] - yt[nab[t]]), 2.0 / m * (p[t][nba[t]] - yt)

        def at_vertices(x):  # [n, c] per point, with its weights
            w = (bary[t][:, :, None] * x[:, None, :]).reshape(-1, x.shape[1])
            return torch.zeros(v.shape[1], x.shape[1], dtype=torch.float64,
                               device=DEV).index_add_(0, corners, w)

        ref = at_vertices(ab.index_add(0, nba[t], ba))
        size = at_vertices(ab.abs().index_add(0, nba[t], ba.abs()))
        pairs = torch.ones(n, dtype=torch.float64, device=DEV).index_add_(
            0, nba[t], torch.ones(m, dtype=torch.float64, device=DEV))
        reach = torch.zeros(v.shape[1], dtype=torch.float64, device=DEV).index_add_(
            0, corners, pairs.repeat_interleave(3))
        for o in out:
            err = (o["grad_verts"][t].double() - ref).abs()
            assert bool((err <= 2.0 ** -24 * (reach[:, None] + 8) * size).all())
