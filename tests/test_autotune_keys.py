"""The autotuner's keys (host logic, CPU)."""
from types import SimpleNamespace as NS

import numpy as np
import torch

from paper_2204_03139_gb300 import autotune


def test_keys_tell_meshes_apart_and_leave_older_entries(monkeypatch):
    """The winner depends on the faces per point, and an entry written before an engine existed is
    not found any more."""
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda device=None: "GPU")
    old = {"GPU|m0|T4|N12|M12": ["tensor", 0], "GPU|batch|m0|F4|N12|M12|P28": ["tensor", 0]}
    monkeypatch.setattr(autotune, "_cache", old)
    assert autotune.best(16, 4096, 4096, 0) is None
    assert autotune.best(16, 4096, 4096, 0, F=3872) is None
    coarse, fine = (autotune.bucket(16, 4096, 4096, 0, F=f) for f in (3872, 65522))
    assert coarse != fine

    def traj(faces):
        off = np.arange(17) * 4096
        return NS(T=16, n_off=off, m_off=off, faces=np.zeros((faces, 3)),
                  pairs=lambda: 16 * 4096 * 4096)

    assert autotune.best_batch([traj(3872)], 0) is None
    keys = {autotune.batch_bucket([traj(f)], 0) for f in (3872, 65522)}
    assert len(keys) == 2
    old[coarse] = ["pruned", 0]
    assert autotune.best(16, 4096, 4096, 0, F=3872) == ("pruned", 0)
    assert autotune.best(16, 4096, 4096, 0, F=65522) is None
