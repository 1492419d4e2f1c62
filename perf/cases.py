"""The work a user of the library has it do, as cases that can be timed and checked.

A case is one of three things a program does with the public entry points:

  sim       a simulation (``Pibm``) advances by ``steps`` coupled steps, then its
            state is read back: to host arrays (``Pibm.read``) or to device memory
            (``pibm_read_fields`` with ``on_device``, for a program that keeps its
            frames on the GPU);
  ensemble  independent simulations advance together (``Ensemble``) and every
            member's state is read back to device memory;
  gradient  ``settling_gradient``: the settling velocity after ``steps`` steps and
            its derivatives, from host arrays to host arrays.

Sizes, counts and material values are those of the presets in
``paper_1407_6704_gb300/inputs.py``, of the benchmark's variants and of the tests
(a preset's particle density on another lattice where the preset itself is too
large), with ragged sizes and periodic axes as in the parity tests. Particles are
uniform random and do not overlap. Outputs come in the precision the populations
are stored in: FP64 as they are, 32- and 16-bit storage as FP32.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1407_6704_gb300 import _lib
from paper_1407_6704_gb300.pibm import Ensemble, Pibm, settling_gradient

KN, RESTITUTION = 1e-2, 0.9
YOUNG, POISSON = 0.1, 0.3


# --- the cases -------------------------------------------------------------------
def _sim(name, lattice, n, periodic, tau, width, precision, particles, dia, ratio, band, steps,
         gravity=1e-5, rebin=1, deterministic=False, interp="delta", contact="linear", substeps=1,
         implicit=True, restart=False, fields="rho,j,pop,x,u", host=False, kind="sim",
         checkpoint=0):
    n = tuple(n) + (1,) * (3 - len(n))
    periodic = tuple(periodic) + (True,) * (3 - len(periodic))
    case = {"name": name, "kind": kind, "lattice": lattice, "nx": n[0], "ny": n[1], "nz": n[2],
            "px": bool(periodic[0]), "py": bool(periodic[1]), "pz": bool(periodic[2]),
            "tau": tau, "width": width, "precision": precision, "particles": particles,
            "dlo": dia[0], "dhi": dia[1], "ratio": ratio, "band_lo": band[0], "band_hi": band[1],
            "gravity": gravity, "steps": steps, "rebin": rebin, "deterministic": deterministic,
            "interp": interp, "contact": contact, "substeps": substeps, "implicit": implicit,
            "restart": restart, "fields": fields, "host": host, "checkpoint": checkpoint}
    if name is None:
        del case["name"]
    return case


def _ensemble(name, members, sizes_seed, side, particles_hi, precision, rebin, steps):
    case = {"name": name, "kind": "ensemble", "members": members, "sizes_seed": sizes_seed,
            "side_lo": side[0], "side_hi": side[1], "particles_hi": particles_hi,
            "precision": precision, "rebin": rebin, "steps": steps}
    if name is None:
        del case["name"]
    return case


def listed():
    walls2, walls3 = (False, False), (False, False, False)
    return [
        # The paper's own validation: one particle settling in a 10 x 10 x 50 cavity
        # (D3Q15, Table 1's fluid at h/d = 2). The smallest simulation there is; what it
        # costs is launches and latency. Read back to the host, as a plot script does.
        _sim("column-one-particle", "d3q15", (10, 10, 50), walls3, 0.72, 4, "fp64", 1, (0.5, 0.5),
             1.01, (0.4, 0.6), 100, gravity=0.0527, host=True),
        # The 128^2 sedimentation preset (200 particles, 2-point kernel, FP64), every option
        # at its default.
        _sim("box-128", "d2q9", (128, 128), walls2, 0.8, 2, "fp64", 200, (0.5, 0.5), 2.0,
             (0.5, 1.0), 100, host=True),
        # An ordinary 2D run on a ragged lattice, periodic along the flow, restarted from a
        # moving state, FP32 storage, cell list rebuilt every step (the default).
        _sim("channel-2d", "d2q9", (509, 317), (True, False), 0.7, 4, "fp32", 6000, (0.3, 0.8),
             2.5, (0.0, 1.0), 50, restart=True),
        # The benchmark workload: 2048^2, 500,000 particles, FP32 storage, kept cell list.
        _sim("bed-2048-fp32", "d2q9", (2048, 2048), walls2, 0.6, 4, "fp32", 500_000, (0.3, 0.8),
             2.5, (0.4, 1.0), 20, rebin=10, fields="pop,x,u"),
        # The same in FP64, for runs whose error has to be below the model's.
        _sim("bed-2048-fp64", "d2q9", (2048, 2048), walls2, 0.6, 4, "fp64", 500_000, (0.3, 0.8),
             2.5, (0.4, 1.0), 10, rebin=10, fields="pop,x,u"),
        # Hertz contacts with 4 DEM sub-steps per fluid step (the benchmark's costliest
        # variant) on a quarter of that bed.
        _sim("bed-1024-hertz-4", "d2q9", (1024, 1024), walls2, 0.6, 4, "fp32", 125_000,
             (0.3, 0.8), 2.5, (0.4, 1.0), 10, contact="hertz", substeps=4),
        # The 3D workload with 16-bit storage: 256^3, 4,000,000 particles. The largest state.
        _sim("bed-256-fp16", "d3q19", (256, 256, 256), walls3, 0.55, 4, "fp16", 4_000_000,
             (0.6, 0.6), 2.0, (0.5, 1.0), 10, rebin=10, fields="pop,x,u"),
        # A mid-size ragged 3D channel in FP32 with the 4-point Lagrange interpolant of
        # Eq. (5), periodic sideways, kept cell list.
        _sim("channel-3d-lagrange", "d3q19", (110, 75, 97), (True, True, False), 0.6, 4, "fp32",
             90_000, (0.6, 0.6), 2.0, (0.5, 1.0), 20, rebin=10, interp="lagrange4"),
        # A reproducible 3D run: the 64^3 slice of the 3D workload, ordered spreading, FP64.
        _sim("slice-64-ordered", "d3q19", (64, 64, 64), walls3, 0.55, 4, "fp64", 62_500,
             (0.6, 0.6), 2.0, (0.5, 1.0), 10, deterministic=True),
        # A parameter study: 64 small simulations of uneven size advanced together.
        _ensemble("study-64", 64, 4, (64, 512), 20_000, "fp32", 10, 50),
        # Inverse problems, forward and reverse: the 96^3 differentiable configuration over a
        # shorter horizon, and a small 2D fit whose cost is latency.
        _sim("gradient-96", "d3q19", (96, 96, 96), walls3, 0.7, 4, "fp64", 20_000, (0.5, 0.5),
             2.0, (0.5, 1.0), 30, kind="gradient", checkpoint=10),
        _sim("gradient-2d", "d2q9", (72, 60), walls2, 0.8, 2, "fp64", 150, (0.5, 0.5), 2.0,
             (0.5, 1.0), 120, kind="gradient", checkpoint=20),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: lattices from a few thousand cells up to the listed
    largest of its kind, ragged sides, every storage type and option."""
    kind = rng.choice(("2d", "2d", "2d", "3d", "3d", "ensemble", "gradient"))
    tau = round(rng.uniform(0.55, 1.0), 3)
    ratio = round(rng.uniform(1.5, 3.0), 3)
    if kind == "ensemble":
        hi = int(_log_uniform(rng, 96, 512))
        return _ensemble(None, rng.randint(6, 48), rng.randrange(1000), (64, hi), 20_000,
                         rng.choice(("fp32", "fp32", "fp64")), rng.choice((1, 10)), 30)
    d = 3 if kind == "3d" or (kind == "gradient" and rng.random() < 0.5) else 2
    if kind == "gradient":
        cells = _log_uniform(rng, 2e3, 4e5)
    else:
        cells = _log_uniform(rng, 4e3, 4e6)
    side = cells ** (1.0 / d)
    n = [max(8, int(side * rng.uniform(0.7, 1.4))) for _ in range(d)]
    cells = math.prod(n)
    periodic = [rng.random() < 0.3 for _ in range(d - 1)] + [False]
    band = rng.choice(((0.5, 1.0), (0.4, 1.0), (0.0, 1.0)))
    dia = rng.choice(((0.5, 0.5), (0.6, 0.6), (0.3, 0.8)))
    inner = math.prod(n[:-1]) * (n[-1] * (band[1] - band[0]))
    particles = max(1, int(inner * _log_uniform(rng, 0.005, 0.3 if d == 2 else 0.4)))
    width = rng.choice((2, 4, 4))
    if kind == "gradient":
        return _sim(None, "d2q9" if d == 2 else rng.choice(("d3q15", "d3q19")), n, periodic, tau,
                    width, "fp64", min(particles, 40_000), dia, ratio, band, rng.randint(15, 30),
                    kind="gradient", checkpoint=rng.choice((5, 10)))
    lattice = "d2q9" if d == 2 else rng.choice(("d3q15", "d3q19", "d3q19"))
    precision = rng.choice(("fp64", "fp32", "fp32", "fp16", "bf16"))
    option = rng.choice(("plain", "plain", "plain", "lagrange4", "hertz", "substeps", "ordered",
                         "explicit"))
    kw = {}
    if option == "lagrange4":
        kw["interp"] = "lagrange4"
    elif option == "hertz":
        kw["contact"] = "hertz"
    elif option == "substeps":
        kw["substeps"] = rng.randint(2, 5)
    elif option == "ordered":
        kw["deterministic"] = True
    elif option == "explicit" and d == 2:  # diverges for the light particles of 3D
        kw["implicit"] = False
    # a kept cell list belongs to large runs
    if cells >= 2 ** 18 and option != "substeps" and rng.random() < 0.7:
        kw["rebin"] = 10
    return _sim(None, lattice, n, periodic, tau, width, precision, particles, dia, ratio, band,
                max(10, min(50, int(1e7 / cells))), restart=cells <= 2 ** 18 and rng.random() < 0.5,
                fields="rho,j,pop,x,u" if precision in ("fp64", "fp32") else "pop,x,u",
                host=precision == "fp64" and cells < 2 ** 17, **kw)


# --- inputs ----------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _adjacent(cq, cp, n, periodic):
    """Candidate pairs (i, j): item j of the cells cp lies in the cell of item i of the cells
    cq or in a neighbour of it, one neighbour offset at a time."""
    d = cq.shape[1]

    def flat(c):
        v = c[:, d - 1]
        for k in range(d - 2, -1, -1):
            v = v * n[k] + c[:, k]
        return v

    key, order = torch.sort(flat(cp), stable=True)
    for off in np.ndindex(*([3] * d)):
        c, ok = [], torch.ones(len(cq), dtype=torch.bool, device=cq.device)
        for k in range(d):
            v = cq[:, k] + (off[k] - 1)
            if periodic[k]:
                v = v % n[k]
            else:
                ok = ok & (v >= 0) & (v < n[k])
            c.append(v)
        want = torch.where(ok, flat(torch.stack(c, 1)), torch.full_like(c[0], -1))
        lo = torch.searchsorted(key, want)
        cnt = torch.searchsorted(key, want, right=True) - lo
        cnt = torch.where(ok, cnt, torch.zeros_like(cnt))
        i = torch.repeat_interleave(torch.arange(len(cq), device=cq.device), cnt)
        first = torch.cumsum(cnt, 0) - cnt
        j = order[lo[i] + torch.arange(len(i), device=cq.device) - first[i]]
        yield i, j


def _cells(X, n):
    top = torch.tensor(n[:X.shape[1]], device=X.device) - 1
    return torch.minimum(torch.floor(X).long().clamp(min=0), top)


def _separation(s, n, periodic):
    """Minimum-image separation, per axis."""
    out = []
    for k in range(s.shape[1]):
        v = s[:, k]
        if periodic[k]:
            v = torch.where(v > 0.5 * n[k], v - n[k], v)
            v = torch.where(v < -0.5 * n[k], v + n[k], v)
        out.append(v)
    return torch.stack(out, 1)


def _cloud(gen, n, d, periodic, dia, band):
    """Uniform random, pairwise non-overlapping particles of the given diameters, at least half
    the largest away from every face and inside the band of the last axis: every round draws
    the particles not yet placed; one that overlaps a placed particle, or one of the round with
    a lower index, is drawn again."""
    dev = _device()
    count = len(dia)
    dmax = float(dia.max())
    lo = np.full(d, 0.5 * dmax)
    hi = np.array(n[:d], dtype=np.float64) - 0.5 * dmax
    lo[-1] = max(lo[-1], band[0] * n[d - 1])
    hi[-1] = min(hi[-1], band[1] * n[d - 1])
    rad = torch.from_numpy(0.5 * dia).to(dev)
    X = torch.zeros((count, d), dtype=torch.float64, device=dev)
    placed = torch.zeros(count, dtype=torch.bool, device=dev)
    todo = torch.arange(count, device=dev)
    for _ in range(400):
        if not len(todo):
            return X.cpu().numpy()
        X[todo] = torch.from_numpy(lo + (hi - lo) * gen.random((len(todo), d))).to(dev)
        live = torch.nonzero(placed).squeeze(1)
        live = torch.cat([live, todo])
        ok = torch.ones(len(todo), dtype=torch.bool, device=dev)
        for i, j in _adjacent(_cells(X[todo], n), _cells(X[live], n), n, periodic):
            a, b = todo[i], live[j]
            s = _separation(X[a] - X[b], n, periodic)
            near = (s * s).sum(1) < (rad[a] + rad[b]) ** 2
            clash = near & (placed[b] | (b < a))
            ok[i[clash]] = False
        placed[todo[ok]] = True
        todo = todo[~ok]
    raise RuntimeError("no room for the particles")


def _dims(case):
    d = 2 if case["lattice"] == "d2q9" else 3
    return d, (case["nx"], case["ny"], case["nz"]), (case["px"], case["py"], case["pz"])


def _inputs(case, seed):
    """Host arrays of one simulation: x0, u0, diameter, density_ratio, f0 (u0 and f0 are None
    for a run that starts at rest)."""
    d, n, per = _dims(case)
    gen = np.random.Generator(np.random.PCG64(seed))
    count = case["particles"]
    dia = gen.uniform(case["dlo"], case["dhi"], count)
    ratio = np.full(count, float(case["ratio"]))
    X = _cloud(gen, n, d, per, dia, (case["band_lo"], case["band_hi"]))
    u0 = f0 = None
    if case["restart"]:
        q, _, w = velocity_set(case["lattice"])
        u0 = 1e-3 * gen.uniform(-1.0, 1.0, (count, d))
        f0 = w[:, None] * (1.0 + 1e-3 * gen.uniform(-1.0, 1.0, (q, n[0] * n[1] * n[2])))
    return {"x0": X, "u0": u0, "diameter": dia, "density_ratio": ratio, "f0": f0}


def _members(case):
    """The members of an ensemble as sim cases: square boxes of log-uniform side, particles in
    the top half, at most 30 % of its area."""
    gen = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    out = []
    for _ in range(case["members"]):
        side = int(round(math.exp(gen.uniform(math.log(case["side_lo"]),
                                              math.log(case["side_hi"])))))
        count = int(round(math.exp(gen.uniform(math.log(100), math.log(case["particles_hi"])))))
        count = min(count, int(0.3 * side * side / 2.0 / (math.pi * 0.25 / 4.0)))
        out.append(_sim("member", "d2q9", (side, side), (False, False),
                        float(gen.uniform(0.55, 1.0)), 2, case["precision"], count, (0.5, 0.5),
                        float(gen.uniform(1.5, 3.0)), (0.5, 1.0), case["steps"],
                        rebin=case["rebin"], fields="pop,x,u"))
    return out


def _member_seed(seed, k):
    return seed * 1000 + k


def _gravity(case):
    d = _dims(case)[0]
    return [0.0] * (d - 1) + [-case["gravity"]]


def _open(case, seed):
    d, n, per = _dims(case)
    return Pibm(case["lattice"], n[:d], per[:d], case["tau"], gravity=_gravity(case),
                delta_width=case["width"], implicit=case["implicit"],
                precision=case["precision"], deterministic=case["deterministic"], kn=KN,
                restitution=RESTITUTION, interp=case["interp"], contact=case["contact"],
                young=YOUNG, poisson=POISSON, substeps=case["substeps"],
                rebin_every=case["rebin"], **_inputs(case, seed))


def _shapes(case):
    d, n, _ = _dims(case)
    q = velocity_set(case["lattice"])[0]
    grid = (n[1], n[0]) if d == 2 else (n[2], n[1], n[0])
    parts = (case["particles"], d)
    return {"rho": grid, "j": (d,) + grid, "pop": (q,) + grid, "x": parts, "u": parts}


def prepare(case, seed):
    """What the program holds before the call: the simulations and the arrays their frames go
    to, or the host arrays of a gradient call."""
    state = {"case": case}
    if case["kind"] == "gradient":
        state["inputs"] = _inputs(case, seed)
    elif case["kind"] == "sim":
        state["sim"] = _open(case, seed)
        if not case["host"]:
            shapes = _shapes(case)
            state["frame"] = {k: torch.zeros(shapes[k], dtype=torch.float64, device="cuda")
                              for k in case["fields"].split(",")}
    else:
        members = _members(case)
        state["sims"] = [_open(m, _member_seed(seed, k)) for k, m in enumerate(members)]
        state["ensemble"] = Ensemble(state["sims"])
        # one array per field; every member fills its own stretch of it
        state["frames"], state["frame"] = [], {}
        names = ("pop", "x", "u")
        sizes = [{k: math.prod(_shapes(m)[k]) for k in names} for m in members]
        for k in names:
            state["frame"][k] = torch.zeros(sum(s[k] for s in sizes), dtype=torch.float64,
                                            device="cuda")
        at = dict.fromkeys(names, 0)
        for s in sizes:
            state["frames"].append({k: state["frame"][k][at[k]:at[k] + s[k]] for k in names})
            for k in names:
                at[k] += s[k]
    return state


# --- one pass --------------------------------------------------------------------
_FIELD = {"rho": 0, "j": 1, "pop": 2, "x": 3, "u": 4}


def _read_on_device(sim, frame):
    """pibm_read_fields into device memory."""
    dst = (ctypes.c_void_p * _lib.NFIELDS)()
    mask = 0
    for k, t in frame.items():
        dst[_FIELD[k]] = t.data_ptr()
        mask |= 1 << _FIELD[k]
    _lib.check(_lib.load().pibm_read_fields(sim._h, mask, dst, 1), "pibm_read_fields")


def _stored(case, frame):
    if case["precision"] == "fp64":
        return frame
    return {k: v.float() for k, v in frame.items()}


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        d, n, per = _dims(case)
        return settling_gradient(case["lattice"], n[:d], per[:d], case["tau"], case["steps"],
                                 checkpoint_every=case["checkpoint"], gravity=_gravity(case),
                                 delta_width=case["width"], kn=KN, restitution=RESTITUTION,
                                 **state["inputs"])
    if case["kind"] == "sim":
        state["sim"].step(case["steps"])
        if case["host"]:
            return state["sim"].read(*case["fields"].split(","))
        _read_on_device(state["sim"], state["frame"])
        return _stored(case, state["frame"])
    state["ensemble"].step(case["steps"])
    _lib.check(state["ensemble"].status(), "ensemble")
    for sim, frame in zip(state["sims"], state["frames"]):
        _read_on_device(sim, frame)
    return _stored(case, state["frame"])


# --- the work it cannot do without -------------------------------------------------
def _step_work(case):
    """(bytes, flops) of one step: every stored population read and written once, every
    particle's X, U and diameter read and X, U written in FP64; the arithmetic of the
    collision and of the particles' stencils."""
    d, n, _ = _dims(case)
    cells = n[0] * n[1] * n[2]
    q = velocity_set(case["lattice"])[0]
    size = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["precision"]]
    taps_i = (4 if case["interp"] == "lagrange4" else case["width"]) ** d
    taps_s = case["width"] ** d
    flops = cells * 15.0 * q + case["particles"] * (taps_i * 2.0 * (d + 1) + taps_s * 2.0 * d
                                                    + 40.0 * case["substeps"])
    return cells * 2.0 * q * size + case["particles"] * (4.0 * d + 1.0) * 8.0, flops


def work(case):
    if case["kind"] == "ensemble":
        each = [work(m) for m in _members(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    d, n, _ = _dims(case)
    cells = n[0] * n[1] * n[2]
    q = velocity_set(case["lattice"])[0]
    by, fl = _step_work(case)
    if case["kind"] == "gradient":
        # forward, then the reverse step: the populations and their adjoint read, the
        # adjoint written; about three times the arithmetic
        return {"bytes": case["steps"] * (by * 2.5), "flops": case["steps"] * 4.0 * fl}
    # the read-back: the populations once, every field written once in FP64
    size = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}[case["precision"]]
    out = sum(math.prod(_shapes(case)[k]) for k in case["fields"].split(","))
    return {"bytes": case["steps"] * by + cells * q * size + 8.0 * out, "flops": case["steps"] * fl}


# --- the same in 64 bits with plain torch ------------------------------------------
def velocity_set(lattice):
    """(q, velocities, weights) in the order of include/pibm.h."""
    axes2 = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0)]
    axes3 = axes2 + [(0, 0, 1), (0, 0, -1)]
    if lattice == "d2q9":
        e = [(0, 0, 0)] + axes2 + [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    elif lattice == "d3q15":
        e = [(0, 0, 0)] + axes3 + [(1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1),
                                   (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]
        w = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8
    else:
        e = [(0, 0, 0)] + axes3 + [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1),
                                   (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
                                   (0, 1, -1), (0, -1, 1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    return len(e), np.array(e), np.array(w)


class _Exact:
    """The coupled step in FP64 torch operations, on populations minus their rest values."""

    def __init__(self, case, inputs, dev):
        self.case, self.dev = case, dev
        self.d, self.n, self.per = _dims(case)
        self.q, self.e, self.w = velocity_set(case["lattice"])
        self.opp = [0] + [a + 1 if a % 2 else a - 1 for a in range(1, self.q)]
        self.shape = (self.n[2], self.n[1], self.n[0])
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.X = t(inputs["x0"])
        self.U = torch.zeros_like(self.X) if inputs["u0"] is None else t(inputs["u0"])
        self.dia, self.ratio = t(inputs["diameter"]), t(inputs["density_ratio"])
        self.tau = t(case["tau"])
        self.grav = t(_gravity(case))
        if inputs["f0"] is None:
            self.f = torch.zeros((self.q,) + self.shape, dtype=torch.float64, device=dev)
        else:
            self.f = t(inputs["f0"] - self.w[:, None]).reshape((self.q,) + self.shape)
        lne = math.log(RESTITUTION)
        self.beta = -lne / math.sqrt(math.pi ** 2 + lne ** 2)

    def taps(self, X, lagrange):
        """Per axis: (node indices, weights), each (particles, W)."""
        W = 4 if lagrange else self.case["width"]
        out = []
        for k in range(self.d):
            x, n = X[:, k], self.n[k]
            first = torch.floor(x.detach() - 0.5) - (W // 2 - 1)
            if lagrange and not self.per[k]:
                first = first.clamp(0, n - 4)
            node = first[:, None] + torch.arange(W, device=self.dev)
            if lagrange:
                t = x - (first + 0.5)
                w = torch.stack([-(t - 1) * (t - 2) * (t - 3) / 6, t * (t - 2) * (t - 3) / 2,
                                 -t * (t - 1) * (t - 3) / 2, t * (t - 1) * (t - 2) / 6], 1)
            else:
                r = node + 0.5 - x[:, None]
                w = 1 - r.abs() if W == 2 else 0.25 * (1 + torch.cos(0.5 * math.pi * r))
            idx = node.long()
            if self.per[k]:
                idx = idx % n
            elif not lagrange:
                inside = (idx >= 0) & (idx < n)
                w = torch.where(inside, w, torch.zeros_like(w))
                w = w / w.sum(1, keepdim=True)
                idx = idx.clamp(0, n - 1)
            out.append((idx, w))
        return out

    def each_tap(self, taps):
        W = taps[0][0].shape[1]
        for t in np.ndindex(*([W] * self.d)):
            cell = torch.zeros_like(taps[0][0][:, 0])
            weight = None
            for k in range(self.d - 1, -1, -1):
                cell = cell * self.n[k] + taps[k][0][:, t[k]]
                v = taps[k][1][:, t[k]]
                weight = v if weight is None else weight * v
            yield cell, weight

    def law(self, delta, vn, meff, R):
        if self.case["contact"] == "hertz":
            E = YOUNG / (2 * (1 - POISSON ** 2))
            S = 2 * E * torch.sqrt(R * delta)
            return 4 / 3 * E * torch.sqrt(R) * delta ** 1.5 \
                - 2 * math.sqrt(5 / 6) * self.beta * torch.sqrt(S * meff) * vn
        return KN * delta - 2 * self.beta * torch.sqrt(meff * KN) * vn

    def contacts(self, X, U, rad, m):
        F = torch.zeros_like(X)
        Xd, cell = X.detach(), _cells(X.detach(), self.n)
        a, b = [], []
        for i, j in _adjacent(cell, cell, self.n, self.per):
            half = i < j
            i, j = i[half], j[half]
            s = _separation(Xd[i] - Xd[j], self.n, self.per)
            touch = (s * s).sum(1) < (rad[i] + rad[j]) ** 2
            a.append(i[touch])
            b.append(j[touch])
        i, j = torch.cat(a), torch.cat(b)
        if len(i):
            s = _separation(X[i] - X[j], self.n, self.per)
            dist = torch.sqrt((s * s).sum(1))
            normal = s / dist[:, None]
            vn = ((U[i] - U[j]) * normal).sum(1)
            f = self.law(rad[i] + rad[j] - dist, vn, m[i] * m[j] / (m[i] + m[j]),
                         rad[i] * rad[j] / (rad[i] + rad[j]))[:, None] * normal
            F = F.index_add(0, i, f).index_add(0, j, -f)
        cols = []
        for k in range(self.d):
            col = F[:, k]
            if not self.per[k]:
                # against a wall a body at rest of the same material: R* = R, m_eff = m
                for low, delta in ((1.0, rad - X[:, k]), (-1.0, rad - (self.n[k] - X[:, k]))):
                    hit = torch.nonzero(delta.detach() > 0).squeeze(1)
                    if len(hit):
                        col = col.index_add(0, hit, low * self.law(delta[hit], low * U[hit, k],
                                                                   m[hit], rad[hit]))
            cols.append(col)
        return torch.stack(cols, 1)

    def step(self, f, X, U, tau, ratio):
        d, q, e = self.d, self.q, self.e
        sub = self.case["substeps"]
        rad, Ap = 0.5 * self.dia, math.pi * self.dia ** 2 / 4
        vol = math.pi * self.dia ** 2 / 4 if d == 2 else math.pi * self.dia ** 3 / 6
        m = ratio * vol
        body = (m * (1 - 1 / ratio))[:, None] * self.grav
        dens = f.sum(0)
        mom = [sum(int(e[a][k]) * f[a] for a in range(q) if e[a][k]) for k in range(d)]
        field = torch.stack([dens] + mom, -1).reshape(-1, d + 1)
        at = 0.0
        for cell, weight in self.each_tap(self.taps(X, self.case["interp"] == "lagrange4")):
            at = at + weight[:, None] * field.index_select(0, cell)
        rho_l, j_l = 1 + at[:, :1], at[:, 1:]
        X0, h, total = X, 1.0 / sub, 0.0
        A, M = Ap[:, None], m[:, None]
        for _ in range(sub):
            Fc = self.contacts(X, U, rad, m)
            if self.case["implicit"]:
                V = (M * U + h * (2 * A * j_l + body + Fc)) / (M + h * 2 * A * rho_l)
                Ub = V
            else:
                V = U + h * (body + Fc - 2 * A * (rho_l * U - j_l)) / M
                Ub = U
            total = total + 2 * (rho_l * Ub - j_l)
            cols = []
            for k in range(d):
                x = X[:, k] + h * V[:, k]
                cols.append(x - self.n[k] * torch.floor(x.detach() / self.n[k]) if self.per[k] else x)
            X, U = torch.stack(cols, 1), V
        amp = A * total * h
        force = torch.zeros((len(field), d), dtype=torch.float64, device=self.dev)
        for cell, weight in self.each_tap(self.taps(X0, False)):
            force = force.index_add(0, cell, weight[:, None] * amp)
        F = [force[:, k].reshape(self.shape) for k in range(d)]
        # Eqs. (2), (3), (8)
        om = 1 / tau
        cF = 1 - 0.5 * om
        rho = 1 + dens
        u = [(mom[k] + 0.5 * F[k]) / rho for k in range(d)]
        uu = sum(v * v for v in u)
        uF = sum(u[k] * F[k] for k in range(d))
        post = []
        for a in range(q):
            axes = [k for k in range(d) if e[a][k]]
            eu = sum(int(e[a][k]) * u[k] for k in axes) if axes else 0.0
            eF = sum(int(e[a][k]) * F[k] for k in axes) if axes else 0.0
            eq = self.w[a] * (dens + rho * (3 * eu + 4.5 * eu * eu - 1.5 * uu))
            post.append(f[a] + om * (eq - f[a])
                        + cF * self.w[a] * (3 * (eF - uF) + 9 * eu * eF))
        # pull, bouncing back where the link comes from beyond a wall
        new = []
        for a in range(q):
            v = torch.roll(post[a], tuple(int(e[a][k]) for k in range(3)), (2, 1, 0))
            wall = None
            for k in range(d):
                if e[a][k] and not self.per[k]:
                    face = torch.zeros(self.n[k], dtype=torch.bool, device=self.dev)
                    face[0 if e[a][k] > 0 else self.n[k] - 1] = True
                    face = face.reshape([-1 if ax == 2 - k else 1 for ax in range(3)])
                    wall = face if wall is None else wall | face
            new.append(v if wall is None else torch.where(wall, post[self.opp[a]], v))
        return torch.stack(new), X, U

    def outputs(self, names):
        w = torch.tensor(self.w, device=self.dev).reshape(-1, 1, 1, 1)
        grid = self.shape[1:] if self.d == 2 else self.shape
        out = {}
        for k in names:
            if k == "rho":
                out[k] = 1 + self.f.sum(0).reshape(grid)
            elif k == "j":
                out[k] = torch.stack([sum(int(self.e[a][c]) * self.f[a] for a in range(self.q)
                                          if self.e[a][c]) for c in range(self.d)])
                out[k] = out[k].reshape((self.d,) + grid)
            elif k == "pop":
                out[k] = (self.f + w).reshape((self.q,) + grid)
            else:
                out[k] = self.X if k == "x" else self.U
        return out


def exact(case, seed):
    dev = _device()
    if case["kind"] == "ensemble":
        parts = []
        for k, m in enumerate(_members(case)):
            parts.append(exact(m, _member_seed(seed, k)))
        return {k: torch.cat([p[k].reshape(-1) for p in parts]) for k in ("pop", "x", "u")}
    sim = _Exact(case, _inputs(case, seed), dev)
    if case["kind"] == "sim":
        with torch.no_grad():
            for _ in range(case["steps"]):
                sim.f, sim.X, sim.U = sim.step(sim.f, sim.X, sim.U, sim.tau, sim.ratio)
            return sim.outputs(case["fields"].split(","))
    from torch.utils.checkpoint import checkpoint

    given = [sim.tau.requires_grad_(), sim.ratio.requires_grad_(), sim.X.requires_grad_()]
    f, X, U = sim.f, sim.X, sim.U
    for _ in range(case["steps"]):
        f, X, U = checkpoint(sim.step, f, X, U, sim.tau, sim.ratio, use_reentrant=False)
    loss = U[:, sim.d - 1].mean()
    dtau, drho, dx0 = torch.autograd.grad(loss, given)
    return {"loss": float(loss.detach()), "dtau": float(dtau), "drho": drho, "dx0": dx0}
