"""The gradient does not depend on how the run is cut into stretches: with few stretches
the steps are launched one by one, with four or more they are captured once and replayed,
for even and odd stretch lengths and a shorter last one. The 3D case has a periodic axis."""
import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import settling_gradient

pytestmark = pytest.mark.gpu

CASES = [("d2q9", (24, 20), (0, 0), 2, 60), ("d2q9", (24, 20), (1, 0), 4, 60),
         ("d3q19", (9, 10, 11), (0, 1, 0), 4, 80)]


@pytest.mark.parametrize("nsteps", [12, 13])
@pytest.mark.parametrize("lattice,n,periodic,width,count", CASES)
def test_stretch_length_does_not_matter(lattice, n, periodic, width, count, nsteps):
    X, dia, rr = inputs.sample_particles(n, count, 0.5, 2.0, (0.0, 1.0), 3)
    d = len(n)
    kw = dict(gravity=[0.0] * (d - 1) + [-1e-5], delta_width=width, x0=X, diameter=dia,
              density_ratio=rr, u0=inputs.velocities(count, d, seed=8, scale=1e-4))
    ref = settling_gradient(lattice, n, periodic, 0.8, nsteps, checkpoint_every=nsteps, **kw)
    for K in (1, 2, 3, 4, 5, 7, 20):
        got = settling_gradient(lattice, n, periodic, 0.8, nsteps, checkpoint_every=K, **kw)
        assert got["loss"] == ref["loss"], K  # the forward run repeats bit for bit
        for k in ("dtau", "drho", "dx0"):
            a, b = np.asarray(ref[k]), np.asarray(got[k])
            # the moment adjoints are added with atomics: rounding only
            assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max(), (K, k)
