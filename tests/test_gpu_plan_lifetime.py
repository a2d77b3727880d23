"""Asynchronous batch plans whose object is dropped while their upload is still queued."""
import gc

import numpy as np
import pytest
import torch

import workloads as W
from paper_2204_03139_gb300.batch import BatchedLoss, DeviceTrajectory

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_staging_is_not_reused_before_the_queued_upload_has_read_it():
    """Behind a busy stream: the pinned block of a dropped plan goes to no other allocation, and
    two plans of different batches, both dropped at once, each compute their own batch."""
    trajs = [DeviceTrajectory.from_host(W.lift_trajectory(k, 14 + k, 3, 700, 700, name="p"), DEV)
             for k in range(2)]
    want = []
    for t in trajs:
        b = BatchedLoss([t])
        b.run(check=True)
        want.append((b.loss_frames[0].clone(), b.grad_verts[0].clone()))
    outs = [[(torch.empty_like(lf), torch.empty_like(gv))] for lf, gv in want]
    stream = torch.cuda.Stream(DEV)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(1_000_000_000)  # about half a second
    b = BatchedLoss([trajs[0]], outputs=outs[0], async_plan=True, stream=stream)
    b.run()
    ptr, size = b._staging.data_ptr(), b._staging.numel()
    del b
    gc.collect()
    others = [torch.empty(size, dtype=torch.uint8, pin_memory=True) for _ in range(4)]
    assert not stream.query()  # the upload has not run yet
    assert ptr not in [o.data_ptr() for o in others]
    BatchedLoss([trajs[1]], outputs=outs[1], async_plan=True, stream=stream).run()
    stream.synchronize()
    for (lf, gv), out in zip(want, outs):
        assert torch.equal(out[0][0], lf)
        np.testing.assert_allclose(out[0][1].cpu().numpy(), gv.cpu().numpy(), rtol=1e-4,
                                   atol=1e-6 * float(gv.abs().max()))
