"""A batch created where the device has memory for its work arrays but not for its CG plans.

The plans are an acceleration: the batch must be created all the same and solve
matrix-free.  Tolerances: both ways converge every step to 1e-10 and the adjoints
to 1e-9; the step's conditioning (dt^2 H against M) loses two digits at most."""
import numpy as np
import pytest
import torch

import synth
from simhelp import dev, host
from test_gpu_batch_teams import _bodies

pytestmark = pytest.mark.gpu


def test_batch_without_memory_for_its_plans():
    from paper_2102_05791_gb300.api import Batch
    probs = _bodies([(24, 20)] * 512, 430)
    kw = dict(newton_rtol=1e-10, adjoint_rtol=1e-9, threads=256)
    rng = np.random.default_rng(431)
    x0 = np.concatenate([p.X for p in probs])
    args = [dev(x0), dev(0.1 * rng.standard_normal(x0.shape)),
            dev(rng.uniform(0.2, 0.8, size=(1, sum(p.T.shape[0] for p in probs)))),
            dev(rng.standard_normal(x0.shape)), dev(np.zeros_like(x0))]
    free0 = torch.cuda.mem_get_info()[0]
    batch = Batch(probs, **kw)
    need = free0 - torch.cuda.mem_get_info()[0]
    want = [host(t) for t in batch.rollout(*args)]
    batch.close()
    torch.cuda.empty_cache()
    # leave 16 MB less than the batch took: its last allocation, the plans' buffers, fails
    fill = torch.empty(torch.cuda.mem_get_info()[0] - need + (16 << 20), dtype=torch.uint8, device="cuda:0")
    batch = Batch(probs, **kw)
    del fill
    torch.cuda.empty_cache()
    got = [host(t) for t in batch.rollout(*args)]
    batch.close()
    assert (got[5][:, 0] == 0).all()
    for g, w in zip(got[:5], want):
        assert np.linalg.norm(g - w) <= 1e-7 * np.linalg.norm(w)
    assert not np.array_equal(got[0], want[0])  # it did run the other way
