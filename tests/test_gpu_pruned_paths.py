"""Sampled frames through every cluster size of the pruned search's preparation, with the area CDF in
shared memory and (over 56 000 faces) beyond it, against the direct engine; and the recomputing
backward on such a mesh. Every pruned call is checked to have run the pruned search."""
import numpy as np
import pytest
import torch

import parity
import workloads as W
from paper_2204_03139_gb300 import _lib, autotune

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def inputs(T, grid, n, m):
    tr = W.lift_trajectory(grid + n, grid, T, n, m, name="c")
    return (torch.from_numpy(np.ascontiguousarray(x)).to(DEV)
            for x in (tr.verts, tr.faces, tr.draws_tn3(), tr.targets_tm3()))


def check(T, grid, n, m):
    v, f, d, y = inputs(T, grid, n, m)
    out = []
    for shape, engine in ((("pruned", 0), _lib.ENGINE_PRUNED), (("direct", 0), _lib.ENGINE_DIRECT)):
        with autotune.tuned(shape):
            out.append(_lib.dc_loss_traj(v, f, d, y, check=True))
        assert _lib.ws_engine(_lib.workspace(1, DEV)) == engine
    for k in ("loss_total", "loss_frames", "nn_ab", "nn_ba"):
        assert torch.equal(out[0][k], out[1][k])
    # the same float32 terms in another order, a few per vertex: a few roundings (6e-8) each
    assert parity.rel_l2(out[0]["grad_verts"].cpu(), out[1]["grad_verts"].cpu()) < 2e-6


# clusters of 1, 2, 3, 4, 6 and 8 CTAs: 512 points of the larger side per CTA
@pytest.mark.parametrize("n,m", [(600, 700), (1100, 900), (1500, 1700), (2100, 2050), (3200, 1),
                                 (513, 4500)])
def test_cluster_sizes_by_the_points(n, m):
    check(2, 20, n, m)


# clusters of 8, 6, 4, 3, 2 and 1, by the number of frames; 60 552 faces, and enough pairs that the
# pruned search's regions are kept beside them
@pytest.mark.parametrize("T,n", [(15, 7301), (22, 6011), (30, 5207), (45, 4201), (60, 3607),
                                 (80, 3001)])
def test_cluster_sizes_with_the_cdf_in_global_memory(T, n):
    check(T, 175, n, n)


def test_recomputing_backward_with_the_cdf_in_global_memory():
    """From 16 000 points per frame on it has kernels of its own: five launches."""
    v, f, d, y = inputs(2, 175, 9000, 8000)
    with autotune.tuned(("direct", 0)):
        r = _lib.dc_loss_traj(v, f, d, y, check=True)
    before = _lib.lib().dc_launch_count()
    g = _lib.dc_loss_traj_bwd(v, f, d, y, r["nn_ab"], r["nn_ba"],
                              grad_total=torch.ones(1, device=DEV), check=True)
    assert _lib.lib().dc_launch_count() - before == 5
    assert parity.rel_l2(g.cpu(), r["grad_verts"].cpu()) < 2e-6
