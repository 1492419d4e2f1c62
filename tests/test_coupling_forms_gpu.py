"""The forms of the particle coupling against one another: FP32 shares a particle's
stencil among lanes (a warp takes 32 particles, or 8 or 16 where there are few), FP64
keeps it on one lane except for few particles in 3D, and FP32 in 3D goes by tiles. Counts
around a warp and around the switch (4 * 152 * 32), one particle and a ragged tail."""
import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 31, 33, 4863, 4864, 4865])
@pytest.mark.parametrize("lattice,n,periodic,width,interp",
                         [("d2q9", (70, 66), (0, 1), 4, "delta"), ("d2q9", (70, 66), (1, 0), 2, "delta"),
                          ("d2q9", (70, 66), (0, 0), 2, "lagrange4"),
                          ("d3q19", (18, 19, 17), (1, 0, 0), 4, "delta"),
                          ("d3q19", (18, 19, 17), (0, 0, 1), 2, "lagrange4"),
                          ("d3q15", (18, 19, 17), (0, 1, 0), 4, "lagrange4"),
                          ("d3q15", (18, 19, 17), (0, 0, 0), 2, "delta")])
def test_fp32_forms_follow_fp64(lattice, n, periodic, width, interp, count):
    check_forms(lattice, n, periodic, width, interp, count)


@pytest.mark.parametrize("count", [19456, 19457])
@pytest.mark.parametrize("lattice,n,periodic,width,interp",
                         [("d2q9", (141, 133), (0, 1), 4, "delta"), ("d2q9", (141, 133), (0, 0), 2, "lagrange4"),
                          ("d3q19", (36, 38, 33), (1, 0, 0), 4, "delta"),
                          ("d3q15", (36, 38, 33), (0, 0, 1), 2, "lagrange4")])
def test_fp32_forms_at_the_switch(lattice, n, periodic, width, interp, count):
    check_forms(lattice, n, periodic, width, interp, count)


def check_forms(lattice, n, periodic, width, interp, count):
    d = len(n)
    rng = np.random.default_rng(count)
    X = rng.uniform(0.1, np.array(n) - 0.1, (count, d))
    kw = dict(gravity=[0.0] * (d - 1) + [-1e-5], delta_width=width, interp=interp, kn=0.0, x0=X,
              u0=inputs.velocities(count, d, seed=4), diameter=np.full(count, 0.2),
              density_ratio=np.full(count, 2.0))
    out = {}
    for prec in ("fp64", "fp32"):
        with Pibm(lattice, n, periodic, 0.8, precision=prec, **kw) as sim:
            sim.step(4)
            assert sim.status() == 0
            out[prec] = sim.read("j", "x", "u")
            out[prec]["f"] = sim.forces()[0]
    for k in ("j", "u", "f"):
        a, b = out["fp64"][k], out["fp32"][k]
        # FP32 moments and weights: a few rounding errors per tap over four steps
        assert np.abs(a - b).max() <= 1e-4 * np.abs(a).max(), k
