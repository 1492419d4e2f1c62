"""Ordered spreading (deterministic mode) against atomic spreading: the same force
summed in another order. The lattices have partial and one-cell tiles and wrapped
axes; the particles are dense enough that most cells receive several stencils."""
import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu

CASES = [("d2q9", (65, 17), (0, 1)), ("d2q9", (33, 40), (1, 0)), ("d2q9", (9, 9), (1, 1)),
         ("d3q19", (17, 9, 9), (1, 0, 1)), ("d3q15", (33, 8, 7), (0, 0, 0)),
         ("d3q19", (9, 25, 13), (0, 1, 0))]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("width,rebin,substeps", [(2, 1, 1), (4, 1, 1), (2, 4, 1), (4, 4, 1),
                                                  (4, 1, 3)])
@pytest.mark.parametrize("lattice,n,periodic", CASES)
def test_ordered_equals_atomic(lattice, n, periodic, width, rebin, substeps, precision):
    d = len(n)
    count = int(0.5 * np.prod(n))
    rng = np.random.default_rng(11)
    X = rng.uniform(0.15, np.array(n) - 0.15, (count, d))
    kw = dict(gravity=[0.0] * (d - 1) + [-1e-5], delta_width=width, precision=precision, kn=0.0,
              x0=X, u0=inputs.velocities(count, d, seed=2), diameter=np.full(count, 0.3),
              density_ratio=np.full(count, 2.0), rebin_every=rebin, substeps=substeps,
              overlap="off")
    out = []
    for det in (False, True, True):
        sim = Pibm(lattice, n, periodic, 0.8, deterministic=det, **kw)
        sim.step(6)
        assert sim.status() == 0
        out.append(sim.read("pop", "rho", "j", "x", "u"))
        sim.close()
    a, b, c = out
    for k in b:
        assert np.array_equal(b[k], c[k]), k  # run to run
    # each cell sums at most some tens of terms; six steps
    tol = 1e-12 if precision == "fp64" else 2e-5
    for k in ("j", "u"):
        assert np.abs(a[k] - b[k]).max() <= tol * np.abs(a[k]).max(), k
