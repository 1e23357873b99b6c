"""The persistent CG solver over its variants, against the oracle.

Sizes reach one CTA, a thread-block cluster and a grid; edge slices stored by
rows in shared memory, by rows with steps left in L2, and by colours streamed
through the ring; both precisions, unused slots, random numbering.  The
adjoint is solved to adjoint_rtol = 1e-10, an FP64 residual the library
computes itself; the oracle's own FP64 residual of the returned lambda must
agree within rounding (its terms cancel to about 1e-6 of their size at most:
1e-16 / 1e-6), hence 2e-10."""
import numpy as np
import pytest

import oracle
import synth
from simhelp import deformed, dev, host, make_sim

pytestmark = pytest.mark.gpu


def _problem(dims, split, shuffle):
    if len(dims) == 2:
        p = synth.make_small2d(*dims, seed=201)
    else:
        p = synth.make_small3d(*dims, split=split, seed=202)
    if shuffle:
        rng = np.random.default_rng(203)
        to = rng.permutation(p.n_vert)
        at = np.argsort(to)
        p.X, p.fixed, p.T = p.X[at], p.fixed[at], to[p.T].astype(np.int32)
    return p


@pytest.mark.parametrize("dims,split,precision,shuffle", [
    ((1, 1), 0, "mixed", False), ((3, 3), 0, "mixed", False), ((3, 3), 0, "fp64", False), ((10, 2), 0, "fp64", False), ((20, 9), 0, "mixed", True),
    ((64, 41), 0, "mixed", False), ((64, 41), 0, "fp64", True), ((190, 121), 0, "mixed", False),
    ((1, 1, 1), 6, "mixed", False), ((1, 1, 1), 5, "fp64", False), ((7, 5, 3), 5, "mixed", False),
    ((13, 9, 8), 6, "mixed", True), ((12, 8, 9), 5, "fp64", False), ((24, 14, 13), 6, "mixed", False),
    ((24, 14, 13), 6, "fp64", True), ((56, 31, 30), 6, "mixed", True), ((80, 41, 40), 5, "mixed", False)])
def test_adjoint_residual(dims, split, precision, shuffle):
    p = _problem(dims, split, shuffle)
    m = oracle.make_model(p)
    x = deformed(p, min(0.01, 0.2 / dims[1]), seed=204)  # noise of 2 % of a cell: H stays positive definite
    b = np.random.default_rng(205).standard_normal(x.shape)
    sim = make_sim(p, precision, adjoint_rtol=1e-10)
    lam, st = sim.adjoint(dev(x), dev(p.a), dev(b))
    lam = host(lam)
    fx = p.fixed.astype(bool)
    b[fx] = 0.0
    assert (lam[fx] == 0.0).all()
    assert np.linalg.norm(m.hvp(x, p.a, lam) - b) <= 2e-10 * np.linalg.norm(b), st
    again, _ = sim.adjoint(dev(x), dev(p.a), dev(b))
    assert np.array_equal(host(again), lam)
    sim.close()


def test_extreme_right_hand_sides():
    """The solver scales b to unit norm: sums of squares outside FP32's range do no harm; b = 0 and NaN."""
    p = synth.make_small3d(4, 3, 3, split=6, seed=206)
    sim = make_sim(p, "mixed", adjoint_rtol=1e-10)
    x, a = dev(deformed(p, 0.01, seed=207)), dev(p.a)
    b = np.random.default_rng(208).standard_normal(p.X.shape)
    ref = host(sim.adjoint(x, a, dev(b))[0])
    # powers of two: the same bits, scaled (the last pass's FP32 corrections, 1e-10 of lambda, stay normal numbers)
    for s in (2.0 ** -40, 2.0 ** 40):
        assert np.array_equal(host(sim.adjoint(x, a, dev(s * b))[0]), s * ref)
    lam, st = sim.adjoint(x, a, dev(0.0 * b))
    assert st["status"] == 0 and st["cg_iters_total"] == 0 and not host(lam).any()
    _, st = sim.adjoint(x, a, dev(np.nan * b), check=False)
    assert st["status"] == -6
    sim.close()


def test_handles_of_different_sizes_side_by_side():
    """Two handles whose tiles and parts need different amounts of shared memory, used in turn."""
    sims = [make_sim(synth.make_small3d(*d, split=5, seed=s), "mixed") for d, s in (((9, 6, 5), 1), ((10, 6, 6), 2))]
    first = [host(s.solve(dev(np.full(s.n_elem, 0.4)))[0]) for s in sims]
    for s, f in zip(sims, first):
        assert np.array_equal(host(s.solve(dev(np.full(s.n_elem, 0.4)))[0]), f)
        s.close()
