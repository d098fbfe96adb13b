"""A small call is as long as its host side: it asks the driver for a CUDA device
once, and still asks."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["evaluate", "evaluate_plain", "coordination"])
def test_one_device_check_per_call(vrp, monkeypatch, name):
    import torch
    w = workloads.make_instance(16, 2, 4, 4, "base", seed=0)
    inst = vrp.Instance.from_workload(w)
    ops, off = (torch.from_numpy(a).cuda() for a in workloads.precedence_candidates(16, 2, 64, seed=0))
    call = getattr(vrp, name)
    want = [t.cpu().numpy() for t in call(inst, ops, off)]
    asked = []
    real = vrp._torch                          # (torch.cuda.current_stream asks once more by itself)
    monkeypatch.setattr(vrp, "_torch", lambda: asked.append(1) or real())
    got = [t.cpu().numpy() for t in call(inst, ops, off)]
    assert len(asked) == 1
    assert all(np.array_equal(a, b) for a, b in zip(want, got))
    monkeypatch.setattr(torch.cuda, "is_available", lambda: False)
    with pytest.raises(RuntimeError):
        call(inst, ops, off)
