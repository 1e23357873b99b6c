"""Energy and gradient in one pass, tiles split over clusters, and the line
search that takes the full step first, against the oracle.

Sizes: one tile on 8 CTAs, down to more tiles than half the SMs (no split);
ragged last tiles.  A gradient component sums about 24 corner terms of 230
operations each: 230 eps = 5e-14 of their absolute sum, 20 times that for
the cancellation of mu F against mu cof F inside an element: 1e-12.  The
energy likewise against its absolute sum."""
import numpy as np
import pytest

import oracle
import synth
from simhelp import deformed, dev, host, make_sim

pytestmark = pytest.mark.gpu


def _make(dims, **kw):
    return synth.make_small2d(*dims, seed=401, **kw) if len(dims) == 2 else \
        synth.make_small3d(*dims, split=6, seed=402, **kw)


@pytest.mark.parametrize("dims", [(1, 1), (16, 17), (41, 25), (67, 61), (150, 140),
                                  (1, 1, 1), (4, 4, 5), (11, 7, 9), (16, 13, 11), (20, 16, 15)])
def test_energy_and_gradient(dims):
    p = _make(dims)
    m = oracle.make_model(p)
    x = deformed(p, min(0.02, 0.2 / dims[1]), seed=403)
    sim = make_sim(p, "mixed")
    E, g = sim.energy_grad(dev(x), dev(p.a))
    Eo, So = m.energy(x, p.a, with_abs=True)
    go, gs = m.grad(x, p.a, with_scale=True)
    assert abs(float(E) - Eo) <= 1e-12 * So
    fx = p.fixed.astype(bool)
    assert (np.abs(host(g) - go)[~fx] <= 1e-12 * gs[~fx]).all()
    assert (host(g)[fx] == 0.0).all()
    E2, g2 = sim.energy_grad(dev(x), dev(p.a))
    assert float(E2) == float(E) and np.array_equal(host(g2), host(g))
    sim.close()


@pytest.mark.parametrize("dims,precision,stretch", [
    ((12, 7), "mixed", 3.0), ((12, 7), "fp64", 0.05), ((5, 4, 3), "mixed", 3.0), ((5, 4, 3), "fp64", 3.0)])
def test_rejected_full_steps(dims, precision, stretch):
    """From a far start full steps are rejected and undone; the solve then reaches |g| <= 1e-9 |g0|."""
    p = _make(dims)
    m = oracle.make_model(p)
    x0 = p.X.copy()
    y0 = p.X[:, 1].min()
    x0[:, 1] = np.where(p.fixed.astype(bool), p.X[:, 1], y0 + stretch * (p.X[:, 1] - y0))
    sim = make_sim(p, precision, newton_rtol=1e-9)
    x, st = sim.solve(dev(p.a), x_init=dev(x0), check=False)
    so = m.newton(p.a, x_init=x0, rtol=1e-9)[1]
    assert so["ls_halvings"] > 0 and st["ls_halvings"] > 0, (so, st)
    assert st["status"] == so["status"] == 0, (so, st)
    g0 = np.linalg.norm(m.grad(x0, p.a))
    assert np.linalg.norm(m.grad(host(x), p.a)) <= 1.01e-9 * g0
    assert abs(st["min_J"] - m.min_J(host(x))) <= 1e-12
    sim.close()


@pytest.mark.parametrize("dims,precision,muscle", [
    ((1, 1), "mixed", 0), ((33, 17), "fp64", 1), ((41, 25), "mixed", 1), ((300, 140), "mixed", 0),
    ((1, 1, 1), "fp64", 0), ((11, 7, 9), "mixed", 1), ((24, 21, 20), "mixed", 0), ((24, 21, 20), "fp64", 1)])
def test_hvp_from_the_callers_arrays(dims, precision, muscle):
    """One wave of tiles or less converts x and a in the tile kernel, more tiles in a pass before it.  Against the
    oracle: FP64 as the gradient above; FP32 inputs rounded to 6e-8, amplified by the same cancellation (a few hundred
    times at most in the norm): 2e-5.  Random element order."""
    p = _make(dims)
    p.muscle_model = muscle
    p.k_contact, p.contact_power = 1e5, 3
    order = np.random.default_rng(404).permutation(p.n_elem)
    p.T, p.fiber, p.a = p.T[order], p.fiber[order], np.random.default_rng(405).uniform(0.3, 0.9, p.n_elem)
    m = oracle.make_model(p)
    x = deformed(p, min(0.02, 0.2 / dims[1]), seed=406)
    v = np.random.default_rng(407).standard_normal(x.shape)
    v[p.fixed.astype(bool)] = 0.0
    sim = make_sim(p, precision, muscle_model=muscle)
    y = host(sim.hvp(dev(x), dev(p.a), dev(v, sim.vec_dtype)))
    ref = m.hvp(x, p.a, v)
    tol = 1e-12 if precision == "fp64" else 2e-5
    assert np.linalg.norm(y - ref) <= tol * np.linalg.norm(ref)
    sim.close()
