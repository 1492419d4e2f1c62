"""16-bit storage keeps the order of its sums: FP32 rounding that differs turns into other
stored values, and a run that repeats to the bit would give other results.

``golden/ordered16.txt`` holds particle velocities of ordered (deterministic) runs, from
the library as it was when one thread gathered and spread a particle's whole stencil, node
by node (written by ``python -m tests.test_storage16_order_gpu`` with that library)."""
import numpy as np
import pytest

from conftest import read_golden
from paper_1407_6704_gb300 import inputs
from paper_1407_6704_gb300.pibm import Pibm

pytestmark = pytest.mark.gpu

STEPS, EVERY = 40, 16  # every 16th particle is kept
RUNS = [("2d", "d2q9", (33, 26), (1, 0), dict(delta_width=4)),
        ("2d-lagrange", "d2q9", (33, 26), (0, 0), dict(delta_width=2, interp="lagrange4")),
        ("2d-sub", "d2q9", (33, 26), (0, 0), dict(delta_width=4, substeps=3)),
        ("3d", "d3q19", (21, 13, 9), (1, 0, 1), dict(delta_width=4)),
        ("3d-w2-kept", "d3q15", (21, 13, 9), (0, 1, 0), dict(delta_width=2, rebin_every=4)),
        ("3d-lagrange", "d3q19", (21, 13, 9), (0, 0, 0), dict(delta_width=2, interp="lagrange4")),
        ("3d-sub", "d3q19", (21, 13, 9), (0, 0, 1), dict(delta_width=4, substeps=2))]


def make(lattice, n, periodic, precision, deterministic=True, **kw):
    from oracle.oracle import lattice as velocity_set

    d, _, w, _ = velocity_set({"d2q9": 9, "d3q15": 15, "d3q19": 19}[lattice])
    count = int(0.3 * np.prod(n))
    X = np.random.default_rng(3).uniform(0.2, np.array(n) - 0.2, (count, d))
    return Pibm(lattice, n, periodic, 0.8, precision=precision, deterministic=deterministic,
                gravity=[0.0] * (d - 1) + [-1e-5], kn=0.0, x0=X,
                u0=inputs.velocities(count, d, seed=2), diameter=np.full(count, 0.4),
                density_ratio=np.full(count, 2.0),
                f0=inputs.populations(w, tuple(reversed(n)), seed=5, eps=1e-2), **kw)


def velocities(run, precision):
    name, lattice, n, periodic, kw = run
    with make(lattice, n, periodic, precision, **kw) as sim:
        sim.step(STEPS)
        assert sim.status() == 0
        return sim.read("u")["u"][::EVERY].ravel()


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("run", RUNS, ids=[r[0] for r in RUNS])
def test_ordered_runs_hold_their_values(run, precision):
    want = next(np.array(r[2:], dtype=float) for r in read_golden("ordered16.txt")
                if r[:2] == [run[0], precision])
    got = velocities(run, precision)
    # four FP32 roundings of the largest velocity (the FP64 update rounds elsewhere)
    assert np.abs(got - want).max() <= 4 * 2.0 ** -24 * np.abs(want).max()


@pytest.mark.parametrize("precision", ["fp16", "bf16"])
@pytest.mark.parametrize("width", [2, 4])
def test_gather_forms_agree_to_the_bit(width, precision):
    """The first step's velocities depend on the gather alone: the tile kernel (atomic
    spreading) and the direct one (ordered) add the same terms in the same order."""
    u = []
    for deterministic in (False, True):
        with make("d3q19", (21, 13, 9), (1, 0, 1), precision, deterministic,
                  delta_width=width) as sim:
            sim.step(1)
            assert sim.status() == 0
            u.append(sim.read("u")["u"])
    assert np.array_equal(u[0], u[1])


if __name__ == "__main__":
    for run in RUNS:
        for precision in ("fp16", "bf16"):
            print(run[0], precision, " ".join("%.9e" % v for v in velocities(run, precision)))
