"""What overlap="auto" takes on 2D lattices of 2^20 cells (the contact search beside the
moments in FP32, the free tiles' collision beside the coupling in FP64, neither in FP32
with sub-cycling) against one stream, across rebuilds."""
import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,substeps,tol", [("fp32", 1, 2e-5), ("fp32", 2, 2e-5),
                                                    ("fp64", 1, 1e-9)])
@pytest.mark.parametrize("n", [(1024, 1024), (1027, 1025)])
def test_auto_follows_off(n, precision, substeps, tol):
    count = 3000
    rng = np.random.default_rng(5)
    # three rows one cell apart, jittered: some particles of diameter 0.8 touch
    i = np.arange(count)
    X = np.stack([10.0 + i % 1000, 5.0 + i // 1000], 1) + rng.uniform(-0.15, 0.15, (count, 2))
    out = {}
    for overlap in ("auto", "off"):
        with Pibm("d2q9", n, (1, 0), 0.8, precision=precision, gravity=[0.0, -1e-5], kn=1e-2,
                  x0=X, u0=inputs.velocities(count, 2, seed=4), diameter=np.full(count, 0.8),
                  density_ratio=np.full(count, 2.0), substeps=substeps,
                  rebin_every=5 if substeps == 1 else 1,
                  overlap=overlap) as sim:
            sim.step(12)
            assert sim.status() == 0
            out[overlap] = sim.read("j", "x", "u")
    # order of the atomic sums only: the bounds of the storage type
    for k in ("j", "x", "u"):
        a, b = out["auto"][k], out["off"][k]
        assert np.abs(a - b).max() <= tol * np.abs(b).max(), k
