"""Ordered spreading against atomic spreading where the stencil of the interpolation is not
that of the spreading: the 4-point Lagrange interpolant with either delta width, with and
without DEM sub-steps (which keep the spreading taps from the step's start)."""
import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("width", [2, 4])
@pytest.mark.parametrize("substeps", [1, 3])
@pytest.mark.parametrize("lattice,n,periodic", [("d2q9", (33, 20), (1, 0)),
                                                ("d3q19", (21, 13, 9), (1, 0, 1))])
def test_ordered_equals_atomic(lattice, n, periodic, substeps, width, precision):
    d = len(n)
    count = int(0.4 * np.prod(n))
    X = np.random.default_rng(7).uniform(0.2, np.array(n) - 0.2, (count, d))
    out = []
    for deterministic in (False, True):
        with Pibm(lattice, n, periodic, 0.8, deterministic=deterministic, precision=precision,
                  gravity=[0.0] * (d - 1) + [-1e-5], delta_width=width, interp="lagrange4",
                  kn=0.0, x0=X, u0=inputs.velocities(count, d, seed=2),
                  diameter=np.full(count, 0.3), density_ratio=np.full(count, 2.0),
                  substeps=substeps) as sim:
            sim.step(6)
            assert sim.status() == 0
            out.append(sim.read("j", "u"))
    # each cell sums at most some tens of terms; six steps
    tol = 1e-12 if precision == "fp64" else 2e-5
    for k in ("j", "u"):
        assert np.abs(out[0][k] - out[1][k]).max() <= tol * np.abs(out[0][k]).max(), k
