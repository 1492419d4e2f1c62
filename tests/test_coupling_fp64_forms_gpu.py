"""The two forms of the particle coupling in 3D FP64 against one another: up to
FEW_PARTICLES a warp shares its particles' stencils, above it each particle keeps its own on
one lane. The larger set is the smaller one and a particle apart from it, too small to move
the fluid."""
import os
import re

import numpy as np
import pytest

from conftest import ROOT
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu


def few_particles():
    path = os.path.join(ROOT, "paper_1407_6704_gb300", "csrc", "pibm_internal.cuh")
    with open(path) as f:
        a, b, c = re.search(r"FEW_PARTICLES = (\d+)LL \* (\d+) \* (\d+);", f.read()).groups()
    return int(a) * int(b) * int(c)


@pytest.mark.parametrize("rebin", [1, 4])
@pytest.mark.parametrize("deterministic", [False, True])
@pytest.mark.parametrize("width,interp", [(2, "delta"), (4, "delta"), (2, "lagrange4"),
                                          (4, "lagrange4")])
@pytest.mark.parametrize("lattice,n,periodic", [("d3q19", (36, 38, 33), (1, 0, 0)),
                                                ("d3q15", (36, 38, 33), (0, 1, 0))])
def test_forms_agree(lattice, n, periodic, width, interp, deterministic, rebin):
    few = few_particles()
    rng = np.random.default_rng(9)
    X = rng.uniform(0.2, np.array(n) - [0.2, 0.2, 8.0], (few + 1, 3))
    X[few] = [18.3, 19.1, 31.2]
    dia, u0 = np.full(few + 1, 0.2), inputs.velocities(few + 1, 3, seed=4)
    dia[few] = 1e-7
    out = []
    for count in (few, few + 1):
        with Pibm(lattice, n, periodic, 0.8, gravity=[0.0, 0.0, -1e-5], delta_width=width,
                  interp=interp, kn=0.0, deterministic=deterministic, rebin_every=rebin,
                  x0=X[:count], u0=u0[:count], diameter=dia[:count],
                  density_ratio=np.full(count, 2.0)) as sim:
            sim.step(5)
            assert sim.status() == 0
            r = sim.read("pop", "x", "u")
            out.append({"pop": r["pop"], "x": r["x"][:few], "u": r["u"][:few]})
    # sums of at most 64 terms in two orders and five steps; the particle apart spreads
    # 1e-14 of what another one does
    for k in ("pop", "x", "u"):
        a, b = out[0][k], out[1][k]
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max(), k
