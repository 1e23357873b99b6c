"""Batches whose bodies go to thread-block clusters, to single CTAs, and (too
large for a plan) to the matrix-free iteration, against the oracle.

Tolerances as in test_gpu_batch: both sides converge to |g| <= 1e-8 |g0| per
step, adjoints to 1e-8."""
import numpy as np
import pytest
import torch

import synth
from simhelp import dev, host
from test_gpu_batch import _check_batch_against_oracle

pytestmark = pytest.mark.gpu


def _bodies(sizes, seed):
    out = []
    for i, s in enumerate(sizes):
        p = synth.make_small2d(*s, fix_bottom=False, seed=seed + i) if len(s) == 2 else \
            synth.make_small3d(*s, split=5 + i % 2, fix_bottom=False, seed=seed + i)
        p.k_contact, p.contact_power, p.dt = 1e6, 3, 1.0 / 30.0
        p.mu = 6e3 * (1 + i % 3)
        p.lam = 4.0 * p.mu
        out.append(p)
    return out


@pytest.mark.parametrize("sizes,threads", [
    ([(1, 1)], 512), ([(1, 1, 1)], 128),                             # fewer vertices than any team has threads
    ([(60, 35)], 512), ([(17, 8, 9)], 256),                          # one body: the largest team
    ([(31, 16), (1, 1), (31, 16)], 128),                             # slots just above 4 per thread; uneven team
    ([(40, 20)] + [(3 + i % 5, 2) for i in range(200)], 256),        # a large body among more small ones than SMs
    ([(9, 7, 6)] * 2 + [(2, 1, 1 + i % 3) for i in range(160)], 512),
    ([(135, 123)], 128),                                             # 16,864 vertices: above 8 per thread of 16 CTAs
])
def test_bodies_of_uneven_size(sizes, threads):
    _check_batch_against_oracle(_bodies(sizes, 300), 0.2, 0.8, seed=301, threads=threads)


def test_a_bodys_result_does_not_depend_on_its_neighbours_place():
    """Each body is summed in an order of its own: a second run gives the same bits, whichever team takes it."""
    from paper_2102_05791_gb300.api import Batch
    probs = _bodies([(24, 13), (5, 4), (17, 10)] + [(2 + i % 4, 2) for i in range(300)], 310)
    b = Batch(probs, threads=256)
    rng = np.random.default_rng(311)
    x0 = np.concatenate([p.X for p in probs])
    args = [dev(x0), dev(0.1 * rng.standard_normal(x0.shape)), dev(rng.uniform(0.2, 0.8, size=(2, b.E))),
            dev(rng.standard_normal(x0.shape)), dev(np.zeros_like(x0))]
    first = [host(t) for t in b.rollout(*args)]
    for _ in range(3):
        for r, f in zip(b.rollout(*args), first):
            assert np.array_equal(host(r), f)
    torch.cuda.synchronize()
    b.close()
