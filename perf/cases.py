"""What the framework is timed on: cavity runs, media, batches and gradients.

Every pass goes through the public API (``Simulation``, ``Batch``,
``ProbeEnergyProblem``): a run on a handle that a program keeps advances it by
``steps`` time steps and reads the physical fields (and the probe series)
back; a gradient pass evaluates the objective and its gradient for the
permittivity in hand.  ``exact`` computes the same outputs in FP64 with plain
torch operations (Thomas sweeps over whole planes, dense matrices for the
fourth-order operator, autograd for the gradient).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2011_14043_gb300 import Batch, Simulation
from paper_2011_14043_gb300.adjoint import ProbeEnergyProblem

C0 = 299792458.0
MU0 = 1.25663706212e-6
EPS0 = 1.0 / (MU0 * C0 * C0)
E = ("ex", "ey", "ez")
COMPS = E + ("hx", "hy", "hz")
# (E, H, axis of the lines as a dimension of [k][j][i], sign) of the two split operators
PAIRS = {"A": (("ex", "hz", 1, 1.0), ("ey", "hx", 0, 1.0), ("ez", "hy", 2, 1.0)),
         "B": (("ex", "hy", 0, -1.0), ("ey", "hz", 2, -1.0), ("ez", "hx", 1, -1.0))}


def _case(name, kind="run", nx=64, ny=64, nz=64, scheme="fadi", precision="f32", cfl=4.0, steps=20, media="vacuum",
          source=False, probes=0, order=2, **more):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "scheme": scheme, "precision": precision, "cfl": cfl,
         "steps": steps, "media": media, "source": source, "probes": probes, "order": order, **more}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the 2-D TM pulse of the first workload recipe with its field probe: 4096 cells, all launches and latency
        _case("tm2d_64_f64", nx=64, ny=64, nz=1, precision="f64", cfl=5.0, steps=200, probes=1),
        # a small resonator, as parameter sweeps step by the hundred
        _case("cavity_32_f32", nx=32, ny=32, nz=32, steps=100),
        # the cavity-mode recipe at its own size: the whole state fits the L2 cache
        _case("cavity_128_f32", nx=128, ny=128, nz=128, steps=50),
        # the headline benchmark's grid: the state is several times the L2 cache
        _case("cavity_256_f32", nx=256, ny=256, nz=256, steps=20),
        # a homogeneous lossy filling in a box of odd sides, second-order LOD
        _case("lossy_219_f32", nx=219, ny=101, nz=75, scheme="flod2", steps=30, media="lossy"),
        # the FP64 form on a box of uneven sides, the reference that FP32 runs are held against
        _case("cavity_200_f64", nx=200, ny=184, nz=216, precision="f64", steps=6),
        # dielectric blocks and a dipole at the recipe's full size, first-order LOD
        _case("blocks_256_f32", nx=256, ny=256, nz=256, scheme="flod", cfl=8.0, steps=12, media="blocks", source=True),
        # the same medium on an odd grid, split-step, watched by probes at every step
        _case("blocks_150_f32", nx=150, ny=117, nz=203, scheme="fss", cfl=8.0, steps=20, media="blocks", source=True,
              probes=3),
        # cavities of uneven sizes and CFL numbers stepped as one batch
        _case("batch_10_f32", kind="batch", count=10, sizes=4, steps=20, media="blocks"),
        # one design iteration: objective and gradient with respect to every cell's permittivity
        _case("gradient_96_f32", kind="gradient", nx=96, ny=96, nz=96, steps=50, every=25, media="region", source=True),
        # fourth-order differences
        _case("order4_192_f32", nx=192, ny=192, nz=192, steps=10, order=4),
        # magnetic and dielectric blocks (the general-media form) with a probe
        _case("magnetic_120_f32", nx=120, ny=96, nz=144, steps=20, media="magnetic", probes=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 6 + ["batch", "gradient"])
    if kind == "batch":
        return _case(None, kind="batch", count=rng.randint(2, 10), sizes=rng.randint(10, 10 ** 6),
                     steps=rng.randint(5, 20), media="blocks", precision=rng.choice(["f32", "f32", "f64"]),
                     scheme=rng.choice(["fadi", "fadi", "flod", "fss"]))
    nx, ny, nz = (_log(rng, 20, 256) for _ in range(3))
    cfl = round(rng.uniform(2.0, 10.0), 3)
    precision = rng.choice(["f32", "f32", "f32", "f64"])
    if kind == "gradient":
        nx, ny, nz = (_log(rng, 20, 96) for _ in range(3))
        return _case(None, kind="gradient", nx=nx, ny=ny, nz=nz, cfl=cfl, precision=precision,
                     steps=rng.randint(10, 50), every=rng.randint(4, 25), media="region", source=True)
    form = rng.choice(["plane", "vacuum", "vacuum", "lossy", "blocks", "blocks", "magnetic", "order4", "long"])
    scheme = rng.choice(["fadi", "fadi", "flod", "fss", "flod2"])
    if form == "plane":
        return _case(None, nx=_log(rng, 24, 400), ny=_log(rng, 24, 400), nz=1, precision=precision, cfl=cfl,
                     steps=rng.randint(50, 200), probes=rng.randint(0, 2))
    if form == "long":  # a waveguide: one side up to four times the rest of the range
        side = [_log(rng, 20, 64), _log(rng, 20, 64), _log(rng, 260, 1000)]
        rng.shuffle(side)
        return _case(None, nx=side[0], ny=side[1], nz=side[2], scheme=scheme, precision=precision, cfl=cfl,
                     steps=rng.randint(5, 20), media=rng.choice(["vacuum", "blocks"]))
    if form == "order4":
        return _case(None, nx=nx, ny=ny, nz=nz, scheme=scheme, precision="f32", cfl=cfl, steps=rng.randint(4, 10),
                     order=4)
    return _case(None, nx=nx, ny=ny, nz=nz, scheme=scheme, precision=precision, cfl=cfl, steps=rng.randint(5, 12),
                 media=form, source=rng.random() < 0.5, probes=rng.choice([0, 0, 1, 3]))


# -- inputs -------------------------------------------------------------------

D = 1e-3  # cell size [m]


def _dt(case):
    s = 2.0 if case["nz"] == 1 else 3.0
    return case["cfl"] * D / (C0 * math.sqrt(s))


def _shape(c, n):
    nx, ny, nz = n
    return {"ex": (nz + 1, ny + 1, nx), "ey": (nz + 1, ny, nx + 1), "ez": (nz, ny + 1, nx + 1),
            "hx": (nz, ny, nx + 1), "hy": (nz, ny + 1, nx), "hz": (nz + 1, ny, nx)}[c]


def _rng(seed, what):
    return np.random.default_rng([*np.atleast_1d(seed), what])


def _fields(n, seed, precision):
    """Eight cavity modes of random indices, amplitudes and divergence-free
    polarisations of E, and as many of H (a 2-D grid: a Gaussian pulse of Ez),
    as the GPU tensors a program sets."""
    g = _rng(seed, 0)
    nx, ny, nz = n
    dev = torch.device("cuda")
    f = {c: torch.zeros(_shape(c, n), dtype=torch.float64, device=dev) for c in COMPS}
    if nz == 1:
        ic, jc = (g.integers(m // 5, m - m // 5 + 1) for m in (nx, ny))
        x, y = (torch.arange(m + 1, dtype=torch.float64, device=dev) for m in (nx, ny))
        f["ez"][0] = torch.exp(-((x[None] - ic) ** 2 + (y[:, None] - jc) ** 2) / 72.0)
    else:
        for k in range(16):
            cut, comps, amp = (torch.cos, E, 1.0) if k < 8 else (torch.sin, COMPS[3:], 1.0 / 376.73)
            m = [int(g.integers(1, min(16, w - 1) + 1)) for w in n]
            kp = np.array([math.sin(m[a] * math.pi / n[a] / 2) for a in range(3)])
            p = g.standard_normal(3)
            p = p - kp * (p @ kp) / (kp @ kp)
            p *= amp * g.standard_normal() / np.linalg.norm(p)
            other = torch.sin if cut is torch.cos else torch.cos
            for a, c in enumerate(comps):
                t = []  # E: cosine along its own axis, sines across (zero on the walls); H the other way round
                for q in range(3):
                    half = 0.5 if (q == a) == (k < 8) else 0.0
                    at = torch.arange(_shape(c, n)[2 - q], dtype=torch.float64, device=dev) + half
                    t.append((cut if q == a else other)(at * (m[q] * math.pi / n[q])))
                f[c] += float(p[a]) * t[2][:, None, None] * t[1][None, :, None] * t[0][None, None, :]
    for c in E:
        f[c] *= _interior(c, n, dev)
    return {c: v.to(torch.float64 if precision == "f64" else torch.float32) for c, v in f.items()}


def _interior(c, n, dev):
    """1 on the unknown E samples, 0 on the walls."""
    m = torch.ones(_shape(c, n), dtype=torch.float64, device=dev)
    for dim in range(3):
        if 2 - dim != E.index(c):  # tangential to the walls normal to this dimension
            m.narrow(dim, 0, 1).zero_()
            m.narrow(dim, m.shape[dim] - 1, 1).zero_()
    return m


def _blocks(g, n, lo, hi, base=1.0):
    a = np.full((n[2], n[1], n[0]), base)
    for _ in range(16):
        s = [slice(None)] * 3
        for q, m in enumerate(n):
            w = int(g.integers(max(1, m // 16), max(1, m // 4) + 1))
            o = int(g.integers(0, m - w + 1))
            s[2 - q] = slice(o, o + w)
        a[tuple(s)] = g.uniform(lo, hi)
    return a


def _media(case, n, seed):
    """(eps_r, mu_r, sigma) per cell, None where uniformly 1, 1, 0."""
    g = _rng(seed, 1)
    shape = (n[2], n[1], n[0])
    kind = case["media"]
    if kind == "lossy":
        return np.full(shape, 2.2), None, np.full(shape, 1e-3)
    if kind == "blocks":
        return _blocks(g, n, 1.0, 4.0 if case["kind"] == "batch" else 10.0), None, None
    if kind == "magnetic":
        return _blocks(g, n, 1.0, 6.0), _blocks(g, n, 1.0, 3.0), None
    if kind == "region":  # the design region: the middle third of every axis
        a = np.ones(shape)
        s = tuple(slice(m // 3, max(m // 3 + 1, 2 * m // 3)) for m in shape)
        a[s] = g.uniform(1.0, 6.0, a[s].shape)
        return a, None, None
    return None, None, None


def _current(case, seed):
    """Modulated-Gaussian dipole current, one value per step."""
    g = _rng(seed, 2)
    t = (np.arange(case["steps"]) + 0.5) / case["steps"]
    return g.uniform(0.5, 2.0) * np.exp(-((t - 0.5) / 0.2) ** 2) * np.sin(2 * math.pi * 3.0 * t)


def _spot(n):
    return tuple(m // 2 for m in n)


def _probe(n, k):
    return (E[2 - k] if n[2] > 1 else "ez",) + tuple((m * (k + 1)) // 4 for m in n)


def _batch_grids(case):
    g = np.random.default_rng(case["sizes"])
    return [((int(g.integers(32, 161)), int(g.integers(32, 97)), int(g.integers(32, 129))),
             float(g.uniform(2.0, 10.0))) for _ in range(case["count"])]


def _n(case):
    return case["nx"], case["ny"], case["nz"]


def _block(n):
    """The probe block of the objective: a few cells past the design region."""
    out = []
    for m in n:
        lo = (3 * m) // 4
        out += [lo, lo + max(1, m // 48)]
    return tuple(out)


def _simulation(case, n, cfl, seed):
    sim = Simulation(*n, D, scheme=case["scheme"], precision=case["precision"], cfl=cfl)
    if case["order"] == 4:
        sim.set_order(4)
    media = _media(case, n, seed)
    if any(a is not None for a in media):
        sim.set_material(*media)
    sim.set_fields(_fields(n, seed, case["precision"]))
    if case["source"]:
        sim.set_source("ez", *_spot(n), _current(case, seed))
    return sim


def prepare(case, seed):
    if case["kind"] == "gradient":
        n = _n(case)
        prob = ProbeEnergyProblem(*n, D, steps=case["steps"], probe_block=_block(n), cfl=case["cfl"],
                                  precision=case["precision"], checkpoint_every=case["every"],
                                  source=("ez",) + _spot(n) + (_current(case, seed),))
        eps = torch.from_numpy(_media(case, n, seed)[0]).cuda().requires_grad_(True)
        return {"problem": prob, "eps": eps}
    if case["kind"] == "batch":
        sims = [_simulation(case, n, cfl, [seed, q]) for q, (n, cfl) in enumerate(_batch_grids(case))]
        return {"sims": sims, "batch": Batch(sims), "steps": case["steps"]}
    sim = _simulation(case, _n(case), case["cfl"], seed)
    pids = [sim.add_probe(*_probe(_n(case), k)) for k in range(case["probes"])]
    return {"sim": sim, "probes": pids, "steps": case["steps"]}


def run(state):
    if "problem" in state:
        eps = state["eps"]
        eps.grad = None
        J = state["problem"].objective(eps)
        J.backward()
        return {"objective": J.detach(), "gradient": eps.grad}
    if "batch" in state:
        state["batch"].step(state["steps"])
        return [s.get_fields(device=True) for s in state["sims"]]
    sim = state["sim"]
    sim.step(state["steps"])
    # a probe keeps its whole series: the first ``steps`` values are those of the handle's first pass
    return {"fields": sim.get_fields(device=True),
            "probes": [sim.get_probe(p, state["steps"]) for p in state["probes"]]}


# -- work ----------------------------------------------------------------------

def work(case):
    """Each procedure of a step reads and writes the six components once and
    reads the media it needs once (8 bytes per cell and array, as they are
    given); 42 right-hand-side and explicit operations and 30 of the
    tridiagonal solves per cell and step of two procedures.  A gradient takes
    the forward steps and as many transposed ones."""
    size = 8 if case["precision"] == "f64" else 4
    procedures = 3 if case["scheme"] == "fss" else 2
    grids = [n for n, _ in _batch_grids(case)] if case["kind"] == "batch" else [_n(case)]
    cells = float(sum(a * b * c for a, b, c in grids))
    media = {"vacuum": 0, "lossy": 0, "blocks": 1, "region": 1, "magnetic": 2}[case["media"]]
    passes = case["steps"] * procedures * (2 if case["kind"] == "gradient" else 1)
    per = 4 if case["nz"] == 1 else 12  # a plane has Ez and one H component per procedure
    out = 8.0 if case["kind"] == "gradient" else 6.0 * size
    return {"bytes": cells * (passes * (per * size + 8 * media) + out), "flops": cells * passes * 36.0}


# -- the same outputs in 64 bits ------------------------------------------------

def _edges(cell, c, n):
    """Mean of a per-cell array over the cells that share each E edge (or H face)."""
    s = _shape(c, n)
    dims = [d for d in range(3) if s[d] == cell.shape[d] + 1]  # the sample lies on a grid plane of these

    def widen(a, d):
        z = torch.zeros_like(a.narrow(d, 0, 1))
        return torch.cat([z, a], d) + torch.cat([a, z], d)
    tot, cnt = cell, torch.ones_like(cell)
    for d in dims:
        tot, cnt = widen(tot, d), widen(cnt, d)
    return tot / cnt


class _Exact:
    """The fundamental schemes on one grid in FP64 torch tensors."""

    def __init__(self, case, n, cfl, media, current=None):
        self.n, self.scheme, self.order = n, case["scheme"], case["order"]
        self.dt = _dt({"cfl": cfl, "nz": n[2]})
        self.dev = torch.device("cuda")
        one = torch.ones((n[2], n[1], n[0]), dtype=torch.float64, device=self.dev)
        eps, mu, sig = (one * (1.0 if k < 2 else 0.0) if a is None else
                        (a if isinstance(a, torch.Tensor) else torch.from_numpy(a).to(self.dev))
                        for k, a in enumerate(media))
        self.eps = {c: EPS0 * _edges(eps, c, n) for c in E}
        self.sig = {c: _edges(sig, c, n) for c in E}
        self.mu = {c: MU0 * _edges(mu, c, n) for c in COMPS[3:]}
        self.lossy = bool((sig > 0).any())
        self.mask = {c: _interior(c, n, self.dev) for c in E}
        self.current = current
        self.at = _spot(n)[::-1]
        self.dense = {}

    def f(self, k):
        """f_E of step k at the source sample (0 outside the table)."""
        if self.current is None or not 0 <= k < len(self.current):
            return 0.0
        return -float(self.current[k]) / (D * D) / self.eps["ez"][self.at]

    def add(self, u, v):
        if isinstance(v, float) and v == 0.0:
            return u
        spot = torch.zeros_like(u["ez"])
        spot[self.at] = 1.0
        return {**u, "ez": u["ez"] + v * spot}

    # first differences along a dimension, with the images of the walls at order 4
    def _matrix(self, N):
        if N not in self.dense:
            m = torch.zeros(N, N + 1, dtype=torch.float64, device=self.dev)  # faces x nodes
            for f in range(N):
                for o, w in ((1, 9 / 8), (0, -9 / 8), (2, -1 / 24), (-1, 1 / 24)):
                    j, s = f + o, 1.0
                    if j < 0:
                        j, s = -j, -1.0
                    if j > N:
                        j, s = 2 * N - j, -1.0
                    if 0 < j < N:
                        m[f, j] += s * w / D
            self.dense[N] = m
        return self.dense[N]

    def d_e(self, w):  # nodes (dimension 0) to faces
        if self.order == 4:
            return torch.tensordot(self._matrix(w.shape[0] - 1), w, 1)
        return (w[1:] - w[:-1]) / D

    def d_h(self, h):  # faces (dimension 0) to nodes, zero on the two walls
        if self.order == 4:
            return -torch.tensordot(self._matrix(h.shape[0]).T, h, 1)
        z = torch.zeros_like(h[:1])
        return torch.cat([z, (h[1:] - h[:-1]) / D, z], 0)

    def solve(self, r, b, d, loss):
        """(1/2 + loss b sigma/4) w - (b/2) D(d D w) = r on the interior nodes (dimension 0), w = 0 on the walls."""
        N = r.shape[0] - 1
        if self.order == 4:  # homogeneous media
            key = (N, float(b.reshape(-1)[0]), float(d.reshape(-1)[0]))
            if key not in self.dense:
                m = self._matrix(N)[:, 1:N]
                self.dense[key] = torch.linalg.inv(0.5 * torch.eye(N - 1, dtype=torch.float64, device=self.dev) +
                                                   0.5 * key[1] * key[2] * m.T @ m)
            w = torch.tensordot(self.dense[key], r[1:N], 1)
            z = torch.zeros_like(r[:1])
            return torch.cat([z, w, z], 0)
        z = torch.zeros_like(r[0])
        dn = d / (D * D)
        low, up = -0.5 * b[1:N] * dn[:-1], -0.5 * b[1:N] * dn[1:]
        diag = 0.5 - low - up + loss
        c, y = [], []
        for j in range(N - 1):
            inv = 1.0 / (diag[j] - low[j] * c[-1]) if j else 1.0 / diag[j]
            y.append((r[j + 1] - low[j] * y[-1]) * inv if j else r[j + 1] * inv)
            c.append(up[j] * inv)
        w = [z]
        for j in range(N - 2, -1, -1):
            w.append(y[j] - c[j] * w[-1])
        return torch.stack([z] + w[1:][::-1] + [z])

    def procedure(self, op, h, u, loss=1.0, alpha=1.0, beta=-1.0, kd=1.0, keep=None):
        """One updating procedure of length h; E = alpha w + beta E."""
        out = dict(u)
        for e, hc, axis, s in PAIRS[op]:
            mv = lambda a: a.movedim(axis, 0)  # noqa: E731
            if u[e].shape[axis] < 3:
                continue
            b, d = mv(abs(h) / (2 * self.eps[e])), mv(abs(h) / (2 * self.mu[hc]))
            sg = s * (1.0 if h > 0 else -1.0)
            m = mv(self.mask[e])
            r = (mv(u[e]) + sg * b * self.d_h(mv(u[hc]))) * m
            N = r.shape[0] - 1
            w = self.solve(r.contiguous(), b.contiguous(), d.contiguous(),
                           loss * (b * mv(self.sig[e]) / 4)[1:N] if self.lossy else 0.0) * m
            out[e] = (alpha * w + beta * mv(u[e])).movedim(0, axis)
            out[hc] = (mv(u[hc]) + kd * sg * d * self.d_e(w)).movedim(0, axis)
            if keep is not None:
                keep[e] = w.movedim(0, axis)
        return out

    def start(self, u):
        if self.scheme == "flod2":
            s = 0.125 * self.dt * self.f(0)
            return self.add(self.procedure("B", self.dt / 2, self.add(u, s)), s)
        if self.scheme != "fadi":
            return u
        tau, v = self.dt / 2, dict(u)  # v = (I + tau B) u + tau f
        for e, hc, axis, s in PAIRS["B"]:
            if u[e].shape[axis] < 3:
                continue
            ue, uh = u[e].movedim(axis, 0), u[hc].movedim(axis, 0)
            m = self.mask[e].movedim(axis, 0)
            ve = ue + s * tau / self.eps[e].movedim(axis, 0) * self.d_h(uh) * m
            if self.lossy:
                ve = ve - tau * (self.sig[e] / (2 * self.eps[e])).movedim(axis, 0) * ue
            v[e] = ve.movedim(0, axis)
            v[hc] = (uh + s * tau / self.mu[hc].movedim(axis, 0) * self.d_e(ue)).movedim(0, axis)
        return self.add(v, tau * self.f(0))

    def step(self, u, k):
        """One step; also the FADI output E of this step (before the source added after it)."""
        dt, f, w = self.dt, self.f(k), {}
        if self.scheme == "fadi":
            u = self.add(self.procedure("A", dt, u), 0.5 * dt * f)
            u = self.procedure("B", dt, u, keep=w)
            return self.add(u, 0.5 * dt * self.f(k + 1)), w

        def sourced(op, h, u, s):
            return self.add(self.procedure(op, h, self.add(u, s)), s)
        if self.scheme == "fss":
            for op, h, c in (("A", dt / 2, 0.125), ("B", dt, 0.25), ("A", dt / 2, 0.125)):
                u = sourced(op, h, u, c * dt * f)
            return u, w
        u = sourced("A", dt, u, 0.25 * dt * f)
        s = 0.25 * dt * f if self.scheme == "flod" else 0.125 * dt * (f + self.f(k + 1))
        return sourced("B", dt, u, s), w

    def output(self, u, k):
        """The physical field, k steps taken."""
        dt = self.dt
        if self.scheme == "fadi":
            return self.procedure("B", -dt, self.add(u, -0.5 * dt * self.f(k)), loss=-1.0, alpha=0.5, beta=0.0, kd=0.5)
        if self.scheme == "flod2":
            s = -0.125 * dt * self.f(k)
            return self.add(self.procedure("B", -dt / 2, self.add(u, s), loss=-1.0), s)
        return u


def _exact_run(case, n, cfl, seed):
    x = _Exact(case, n, cfl, _media(case, n, seed), _current(case, seed) if case["source"] else None)
    u = x.start({c: v.double() for c, v in _fields(n, seed, case["precision"]).items()})
    series = [[] for _ in range(case["probes"])]
    for k in range(case["steps"]):
        u, _ = x.step(u, k)
        if series:
            o = x.output(u, k + 1)
            for q, s in enumerate(series):
                c, i, j, l = _probe(n, q)
                s.append(o[c][l, j, i])
    return x.output(u, case["steps"]), [torch.stack(s) for s in series]


def exact(case, seed):
    if case["kind"] == "gradient":
        n = _n(case)
        eps = torch.from_numpy(_media(case, n, seed)[0]).cuda().requires_grad_(True)
        x = _Exact(case, n, case["cfl"], (eps, None, None), _current(case, seed))
        zero = {c: torch.zeros(_shape(c, n), dtype=torch.float64, device="cuda") for c in COMPS}
        u, J = x.start(zero), 0.0
        b = _block(n)
        s = (slice(b[4], b[5]), slice(b[2], b[3]), slice(b[0], b[1]))
        for k in range(case["steps"]):
            u, w = x.step(u, k)
            J = J + sum((0.25 * w[c][s] ** 2).sum() for c in E)
        J.backward()
        return {"objective": J.detach(), "gradient": eps.grad}
    with torch.no_grad():
        if case["kind"] == "batch":
            return [_exact_run(case, n, cfl, [seed, q])[0] for q, (n, cfl) in enumerate(_batch_grids(case))]
        fields, probes = _exact_run(case, _n(case), case["cfl"], seed)
        return {"fields": fields, "probes": probes}
