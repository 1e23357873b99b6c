"""The persistent CG solver's kernel variants that only larger meshes reach.

One size per variant (storage by rows or colours, slots a thread, slice resident
or streamed; see test_cg_capacity for which sizes reach which); the FP64 residual
of the adjoint, formed with an FP64 handle's HVP, agrees with adjoint_rtol within
the rounding of two FP64 sums whose terms cancel to 1e-6 at most, hence 2e-10."""
import numpy as np
import pytest

import synth
from simhelp import deformed, dev, host, make_sim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,precision", [
    ((110, 110), "mixed"),      # cluster, rows, 4 slots a thread
    ((400, 250), "mixed"),      # grid, rows, 4
    ((400, 250), "fp64"),       # grid, rows, 4
    ((640, 478), "mixed"),      # colours, resident, 4
    ((700, 460), "mixed"),      # colours, resident, 8
    ((900, 560), "mixed"),      # colours, streamed, 8
    ((70, 37, 36), "mixed"),    # grid, rows, 4
    ((100, 48, 47), "mixed"),   # colours, streamed, 4
    ((100, 72, 72), "mixed"),   # colours, streamed, 8
    ((66, 35, 34), "fp64"),     # grid, rows, 4
    ((72, 37, 36), "fp64"),     # colours, streamed, 2
    ((86, 44, 44), "fp64"),     # colours, streamed, 4
])
def test_adjoint_residual(dims, precision):
    if len(dims) == 2:
        p = synth.make_small2d(*dims, seed=441)
    else:
        p = synth.make_small3d(*dims, split=6, seed=442)
    x, a = dev(deformed(p, min(0.01, 0.2 / dims[1]), seed=443)), dev(p.a)
    b = np.random.default_rng(444).standard_normal(p.X.shape) * (p.fixed == 0)[:, None]
    sim = make_sim(p, precision, adjoint_rtol=1e-10, max_adjoint_cg=20000)
    n0 = sim.kernel_launches()
    lam, st = sim.adjoint(x, a, dev(b))
    assert sim.kernel_launches() - n0 < st["cg_iters_total"]  # one launch a solve, not several an iteration
    ref = make_sim(p, "fp64") if precision == "mixed" else sim
    r = host(ref.hvp(x, a, lam)) - b
    assert np.linalg.norm(r) <= 2e-10 * np.linalg.norm(b), st
    if ref is not sim:
        ref.close()
    sim.close()
