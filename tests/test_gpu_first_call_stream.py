"""A handle's or a batch's first call on a stream of its own.

The first solve of a handle uploads the tables of its CG plan, the creation of
a batch all of its tables; a non-blocking stream (every torch side stream) does
not wait for the default stream, so the uploads must be complete, or on the
call's own stream, before its kernels read them.  All sums have a fixed order:
the results are the bits of a handle first used on the default stream."""
import numpy as np
import pytest
import torch

import synth
from simhelp import dev, host, make_sim
from test_gpu_batch_teams import _bodies

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(3, 2, 2), (13, 9, 8), (56, 31, 30)])
def test_first_solve_on_a_side_stream(dims):
    p = synth.make_small3d(*dims, split=6, seed=401)
    a = dev(p.a)
    b = dev(np.random.default_rng(402).standard_normal(p.X.shape))
    out = []
    for stream in (torch.cuda.Stream(), torch.cuda.current_stream()):
        sim = make_sim(p, "mixed")
        with torch.cuda.stream(stream):
            lam, _ = sim.adjoint(sim.X, a, b)
            stream.synchronize()
            out.append(host(lam))
        sim.close()
    assert np.array_equal(*out)


def test_first_rollout_on_a_side_stream():
    from paper_2102_05791_gb300.api import Batch
    probs = _bodies([(60, 35), (24, 13)] + [(2 + i % 4, 2) for i in range(40)], 410)
    rng = np.random.default_rng(411)
    x0 = np.concatenate([p.X for p in probs])
    n_elem = sum(p.T.shape[0] for p in probs)
    args = [dev(x0), dev(0.1 * rng.standard_normal(x0.shape)), dev(rng.uniform(0.2, 0.8, size=(2, n_elem))),
            dev(rng.standard_normal(x0.shape)), dev(np.zeros_like(x0))]
    torch.cuda.synchronize()
    out = []
    for stream in (torch.cuda.Stream(), torch.cuda.current_stream()):
        batch = Batch(probs)
        with torch.cuda.stream(stream):
            got = batch.rollout(*args)
            stream.synchronize()
            out.append([host(t) for t in got])
        batch.close()
    for s, d in zip(*out):
        assert np.array_equal(s, d)
