"""Read-back of the state (rho, j, populations, X, U) against plain NumPy.

A simulation restarted from populations f0 and not stepped holds f0 itself up to
the storage rounding of f - w; rho and j are its moments. Lattices with one-cell
axes, odd extents and wrapped axes cover the wall and periodic pulls; the host
path stages planes in groups that depend on the storage type."""
import ctypes

import numpy as np
import pytest

from conftest import *  # noqa: F401,F403
from paper_1407_6704_gb300 import _lib, inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu

LATTICES = [("d2q9", (33, 7), (0, 1)), ("d2q9", (1, 40), (1, 0)), ("d2q9", (256, 2), (0, 0)),
            ("d3q15", (5, 4, 3), (1, 0, 1)), ("d3q19", (18, 9, 5), (0, 1, 0)),
            ("d3q19", (1, 1, 1), (0, 0, 0))]
# storage rounding: half an ulp of f - w (FP16 holds it scaled by 2^12, so its
# smallest step is 2^-24 / 2^12), plus FP64 rounding at the scale of f
REL = {"fp64": 0.0, "fp32": 2.0 ** -24, "fp16": 2.0 ** -11, "bf16": 2.0 ** -8}


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("lattice,n,periodic", LATTICES)
def test_fields_match_numpy(lattice, n, periodic, precision):
    import torch
    from oracle.oracle import lattice as velocity_set

    q = {"d2q9": 9, "d3q15": 15, "d3q19": 19}[lattice]
    d, e, w, _ = velocity_set(q)
    shape = tuple(reversed(n))
    f0 = inputs.populations(w, shape, seed=3, eps=1e-2)
    sim = Pibm(lattice, n, periodic, 0.8, precision=precision, f0=f0)
    r = sim.read("rho", "j", "pop")
    wb = w.reshape((-1,) + (1,) * d)
    assert np.all(np.abs(r["pop"] - f0) <= REL[precision] * np.abs(f0 - wb) + 2.0 ** -36 + 4e-16)
    # the read-back adds w to the stored value, widened exactly
    dev = f0 - wb
    stored = {"fp64": lambda: dev, "fp32": lambda: dev.astype(np.float32).astype(np.float64),
              "fp16": lambda: (dev.astype(np.float32) * np.float32(4096)).astype(np.float16)
              .astype(np.float64) / 4096,
              "bf16": lambda: torch.from_numpy(dev.astype(np.float32)).bfloat16().double().numpy()}
    assert np.array_equal(r["pop"], stored[precision]() + wb)
    # rho and j are sums of at most q FP64 terms of size at most max(f)
    tol = 2 * q * 2.0 ** -52
    assert np.abs(r["rho"] - r["pop"].sum(0)).max() <= tol
    j = np.tensordot(e[:, :d].T.astype(float), r["pop"], axes=1)
    assert np.abs(r["j"] - j).max() <= tol
    # each field on its own, and device destinations: the same bits
    for k in ("rho", "j", "pop"):
        assert np.array_equal(sim.read(k)[k], r[k])
    dev = {k: torch.full(r[k].shape, -1.0, dtype=torch.float64, device="cuda") for k in r}
    dst = (ctypes.c_void_p * _lib.NFIELDS)()
    for i, k in enumerate(("rho", "j", "pop")):
        dst[i] = dev[k].data_ptr()
    _lib.check(_lib.load().pibm_read_fields(sim._h, 7, dst, 1))
    for k in r:
        assert np.array_equal(dev[k].cpu().numpy(), r[k])
    sim.close()


@pytest.mark.parametrize("n,count", [((64, 64), 40), ((8, 8), 90)])
def test_particles_come_back_in_user_order(n, count):
    """After steps that sort the particles; the 8 x 8 lattice is too small to stage
    its particles on the device."""
    rng = np.random.default_rng(5)
    X = rng.uniform(0.5, np.array(n) - 0.5, (count, 2))
    U = inputs.velocities(count, 2, seed=6, scale=1e-6)
    kw = dict(x0=X, u0=U, diameter=np.full(count, 0.1), density_ratio=np.full(count, 2.0))
    sim = Pibm("d2q9", n, (0, 0), 0.8, kn=0.0, **kw)
    sim.step(3)
    r = sim.read("x", "u")
    assert np.abs(r["x"] - X).max() < 1e-4
    assert np.array_equal(sim.read("x")["x"], r["x"])
    assert np.array_equal(sim.read("u")["u"], r["u"])
    sim.close()


@pytest.mark.parametrize("n", [(120, 121), (300, 301)])
def test_large_host_arrays(n):
    """Arrays above a megabyte, which are mapped before the copy: new, in use, pinned, and
    not starting on a page."""
    import torch

    count = 40000 * (n[0] > 200) + 50
    rng = np.random.default_rng(2)
    sim = Pibm("d2q9", n, (1, 0), 0.8, kn=0.0, x0=rng.uniform(0.5, np.array(n) - 0.5, (count, 2)),
               u0=inputs.velocities(count, 2, seed=6, scale=1e-6), diameter=np.full(count, 0.1),
               density_ratio=np.full(count, 2.0))
    names = ("rho", "j", "pop", "x", "u")
    sim.step(3)
    r = sim.read(*names)
    shapes = {k: r[k].shape for k in names}
    pinned = {k: torch.full(shapes[k], -1.0, dtype=torch.float64, pin_memory=True).numpy()
              for k in names}
    shifted = {}
    for k in names:
        raw = np.full(r[k].size + 3, -1.0)
        shifted[k] = raw[1:-2].reshape(shapes[k])
    for out in (pinned, shifted):
        got = sim.read(*names, out=out)
        for k in names:
            assert np.array_equal(got[k], r[k]) and np.shares_memory(got[k], out[k])
    for k in names:
        raw = shifted[k].base if shifted[k].base.ndim == 1 else shifted[k].base.base
        assert raw[0] == -1.0 and (raw[-2:] == -1.0).all()
    sim.close()
