"""The inner products of the persistent CG solver.

After one CG iteration from zero the solution is lambda = alpha p0 with
alpha = r.z / p.Ap and r.z = p.b, so lambda.(b - A lambda) / lambda.b is the
relative error of alpha, formed here from lambda and the library's FP64 HVP.

Tolerances.  FP64: sums of at most 3e5 products and an HVP of its own rounding
(its terms cancel to 1e-3 at most): 1e-11.  Mixed: r.z, p.Ap and their quotient
carry about 48 bits and only alpha is rounded to FP32 (2^-24); the entries of
lambda and A p0 are FP32 too, their errors independent and averaged over a
thousand entries and more, for which half of that is added.  All material
constants are exact in FP32, so no common factor shifts A."""
import numpy as np
import pytest

import synth
from simhelp import dev, host, make_sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("dims", [(16, 9), (64, 41), (110, 110), (7, 6, 5), (13, 9, 8), (24, 14, 13), (40, 31, 30),
                                  (80, 41, 40)])
def test_first_step_length(dims, precision):
    if len(dims) == 2:
        p = synth.make_small2d(*dims, seed=421)
    else:
        p = synth.make_small3d(*dims, split=6, seed=422)
    p.mu, p.lam, p.k_muscle, p.k_contact = 4096.0, 16384.0, 0.0, 0.0
    sim = make_sim(p, precision, max_adjoint_cg=1, adjoint_rtol=1e-14)
    ref = make_sim(p, "fp64") if precision == "mixed" else sim
    x, a = sim.X, dev(p.a)
    free = p.fixed == 0
    rng = np.random.default_rng(423)
    worst = 0.0
    for _ in range(24):
        b = rng.standard_normal(p.X.shape) * free[:, None]
        lam, st = sim.adjoint(x, a, dev(b), check=False)
        assert st["cg_iters_total"] == 1, st
        al = host(ref.hvp(x, a, lam))
        lam = host(lam)
        worst = max(worst, abs(np.sum(lam * (b - al)) / np.sum(lam * b)))
    print(f"{dims} {precision}: {worst:.2e}")
    assert worst <= (1e-11 if precision == "fp64" else 1.5 * 2.0 ** -24)
    if ref is not sim:
        ref.close()
    sim.close()


@pytest.mark.parametrize("dims,bodies,threads", [((16, 9), 1, 256), ((90, 60), 1, 256), ((13, 9), 200, 256),
                                                 ((24, 21), 160, 128), ((31, 24), 160, 128), ((6, 5, 5), 160, 128)])
def test_first_step_length_of_a_batch(dims, bodies, threads):
    """The same in the batched solver: one step whose adjoint takes one iteration; xbar0 = M lambda."""
    from paper_2102_05791_gb300.api import Batch
    p = synth.make_small2d(*dims, fix_bottom=False, seed=424) if len(dims) == 2 else \
        synth.make_small3d(*dims, split=6, fix_bottom=False, seed=425)
    p.mu, p.lam, p.k_muscle, p.k_contact, p.gravity, p.dt = 4096.0, 16384.0, 0.0, 0.0, 0.0, 1.0 / 32.0
    d = p.X.shape[1]
    B = np.linalg.inv(np.swapaxes(p.X[p.T[:, 1:]] - p.X[p.T[:, :1]], 1, 2))
    vol = 1.0 / np.linalg.det(B) / (2.0 if d == 2 else 6.0)
    mass = np.zeros(len(p.X))
    np.add.at(mass, p.T, (p.density * vol / (d + 1))[:, None])
    batch = Batch([p] * bodies, threads=threads, max_adjoint_cg=1, adjoint_rtol=1e-14)
    sim = make_sim(p, "fp64", dt=0.0)
    x0 = dev(np.concatenate([p.X] * bodies))
    a = dev(np.tile(p.a, bodies)[None])
    rng = np.random.default_rng(426)
    worst = 0.0
    for _ in range(24 if bodies == 1 else 1):
        b = rng.standard_normal(x0.shape)
        sx, _, _, xb0, _, stats = batch.rollout(x0, dev(0.0 * b), a, dev(b), dev(0.0 * b))
        assert (host(stats)[:, 3] == 1).all()
        x1, ml = host(sx)[1].reshape(bodies, -1, d), host(xb0).reshape(bodies, -1, d)
        for k in range(0, bodies, max(1, bodies // 24)):
            lam, bk = ml[k] / mass[:, None], b.reshape(bodies, -1, d)[k]
            al = ml[k] + p.dt ** 2 * host(sim.hvp(dev(x1[k]), dev(p.a), dev(lam)))
            worst = max(worst, abs(np.sum(lam * (bk - al)) / np.sum(lam * bk)))
    print(f"{dims} x {bodies}: {worst:.2e}")
    assert worst <= 1.5 * 2.0 ** -24
    sim.close()
    batch.close()
