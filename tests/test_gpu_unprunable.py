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
                                  "small_beside_large", "one_target", "one_sim_point"])
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
