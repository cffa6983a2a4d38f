"""The work that a user of this library has it do, as cases to be timed.

A radiation step of a simulation is: the particles have moved, so the neighbour search runs
again; the radiation is sub-cycled on the new set; the total energy is read.  The cases cover
that step from the smallest set to a few million particles, the calls beside it (one plain
step, individual time bins, the drift correction, the differentiable step, the search alone),
both precisions, both Riemann solvers and every kind of sink.  Particle sets and radiation
fields are those of ``paper_2302_12727_gb300/workloads.py`` (jittered lattice, sine density,
lognormal density; weak background, point sources, collimated beam), drawn on the GPU.

``exact`` evaluates the same equations in 64 bits with plain torch (Ivkovic 2023, arXiv
2302.12727, Part II "The Neighbor Search", Part III "One RT Time Step").
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2302_12727_gb300 import SubcycleFunction, Transport

DEV = "cuda:0"
ETA = 1.2348
KAPPA = 1.825742          # support radius over smoothing length
SIGMA = 16.0 / math.pi    # normalisation of the cubic spline
C_RED = 1.0


# ---------------------------------------------------------------------------------------
# the cases
def _case(name, kind, layout, n, groups, sources, n_sub, precision="fp32", riemann="glf", sink="none", sigma=0.0):
    c = {"kind": kind, "layout": layout, "n": n, "groups": groups, "sources": sources, "n_sub": n_sub,
         "precision": precision, "riemann": riemann, "sink": sink, "sigma": sigma}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the small test problem everybody starts with: one source in a 16^3 box, ten sub-cycles;
        # bound by launches and latency
        _case("point-source-4k", "hydro", "lattice", 16 ** 3, 1, 1, 10),
        # the benchmark: sine density with a beam and a source, three groups, grey gas, 50 sub-cycles
        _case("beam-262k", "hydro", "sine", 64 ** 3, 3, 1, 50, sink="grey"),
        # a production-sized cosmological step: clustered gas, four groups, 64 sources
        _case("lognormal-2m", "hydro", "lognormal", 128 ** 3, 4, 64, 32, sigma=1.0),
        # photo-ionisation with five groups (more than one pass of the pair kernels takes) on an odd
        # number of particles that do not move between calls
        _case("photo-100k-g5", "subcycle", "sine", 99991, 5, 4, 16, sink="photo"),
        # the less diffusive Riemann solver
        _case("hll-131k", "subcycle", "sine", 131071, 3, 1, 20, riemann="hll", sink="grey"),
        # a code that sub-cycles itself: one plain step of a large one-group set per call
        _case("step-1m-g1", "step", "lognormal", 1000003, 1, 16, 1, sink="grey", sigma=1.0),
        # the double-precision path, for validation runs
        _case("double-33k", "hydro", "lattice", 32 ** 3, 2, 8, 16, precision="fp64"),
        # gradients of a loss with respect to the initial field and the luminosities, in double: in
        # float they hang on which side of the limiter's kinks the rounding falls, so that no two
        # roundings of the forward pass give the same ones
        _case("adjoint-33k", "adjoint", "lattice", 32 ** 3, 2, 8, 16, precision="fp64"),
        # the same on a small odd set, as gradient checks use it
        _case("adjoint-9k", "adjoint", "lattice", 21 ** 3, 1, 4, 8, precision="fp64"),
        # individual time steps on clustered gas: one hydro step of eight smallest steps
        _case("bins-262k", "bins", "lognormal", 64 ** 3, 4, 8, 3, sigma=1.0),
        # moving gas: drift correction, neighbour search at the new positions, few sub-cycles
        _case("moving-500k", "moving", "sine", 500009, 2, 4, 4, sink="grey"),
        # the neighbour search alone on strongly clustered gas, and the geometry read back
        _case("search-clustered-1m", "search", "lognormal", 1000000, 1, 0, 0, sigma=2.0),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1

    kind = rng.choice(["hydro", "hydro", "hydro", "subcycle", "subcycle", "step", "double", "adjoint", "bins", "moving",
                       "search"])
    groups = rng.randint(1, 5)
    sources = rng.choice([1, 2, 5, 16, 64])
    layout = rng.choice(["lattice", "sine", "lognormal"])
    sigma = round(rng.uniform(0.6, 1.0), 2) if layout == "lognormal" else 0.0
    sink = rng.choice(["none", "grey", "photo"])
    if kind in ("double", "adjoint"):
        n = rng.randint(13, 30) ** 3
        return _case("", "hydro" if kind == "double" else kind, "lattice", n, rng.randint(1, 3), rng.choice([1, 3, 8]),
                     rng.randint(4, 16), precision="fp64", sink="none" if kind == "adjoint" else sink)
    hi = 1500000 if kind in ("step", "search", "moving") else 1000000
    n = rng.randint(16, 80) ** 3 if layout == "lattice" else size(30000 if sigma else 8000, hi)
    if kind == "search":
        return _case("", kind, "lognormal", size(200000, hi), 1, 0, 0, sigma=round(rng.uniform(1.0, 2.0), 2))
    if kind == "step":
        return _case("", kind, layout, n, groups, sources, 1, sink=sink, sigma=sigma)
    if kind == "bins":
        return _case("", kind, "lognormal", size(30000, 300000), groups, sources, rng.randint(1, 3),
                     sigma=round(rng.uniform(0.7, 1.0), 2))
    if kind == "moving":
        return _case("", kind, layout, n, groups, sources, rng.randint(1, 8), sink=sink, sigma=sigma)
    n_sub = rng.randint(2, 50)
    while n * (groups + 1) * n_sub > 150e6:
        n_sub -= 1
    riemann = rng.choice(["glf", "glf", "glf", "hll"])
    return _case("", kind, layout, n, groups, sources, max(n_sub, 2), riemann=riemann, sink=sink, sigma=sigma)


# unordered pairs per particle of the three layouts
_PAIRS = {"lattice": 23.8, "sine": 23.2, "lognormal": 23.6}


def work(case):
    """Bytes: the positions, the state in and out, the absorption (or the fields read back).
    Flops: counted on the pair arithmetic (flux geometry 77 and 193 a group, gradient 35 and 28
    a group for each of the two directions, 8 a group to accumulate; per pair)."""
    n, G = case["n"], case["groups"]
    ts = 8 if case["precision"] == "fp64" else 4
    P = n * (24.7 if case["sigma"] > 1.5 else _PAIRS[case["layout"]])
    search = P * 2 * 60.0
    step = P * (77.0 + 193.0 * G + 2 * (35.0 + 28.0 * G) + 8.0 * G + (120.0 * G if case["riemann"] == "hll" else 0.0))
    state = 2.0 * 4 * G * n * ts + 8.0 * n * {"none": 0, "grey": 1, "photo": 2}[case["sink"]]
    k = case["kind"]
    if k == "search":
        return {"bytes": 24.0 * n + 8.0 * n * 13, "flops": search}
    if k == "adjoint":   # forward, forward again from the checkpoints, and the reverse of each step
        return {"bytes": state + 2.0 * 4 * G * n * ts, "flops": 4.0 * case["n_sub"] * step}
    if k == "bins":      # the shares of the bins 0..B as many steps of 2^B as they take
        return {"bytes": state + 24.0 * n + 4.0 * n, "flops": search + step * (2.0 ** (case["n_sub"] + 1) - 1) / (case["n_sub"] + 1)}
    if k == "step":
        return {"bytes": state, "flops": step}
    if k == "subcycle":
        return {"bytes": state, "flops": case["n_sub"] * step}
    extra = 24.0 * n if k == "moving" else 0.0
    return {"bytes": state + 24.0 * n + extra, "flops": search + case["n_sub"] * step}


# ---------------------------------------------------------------------------------------
# inputs
def _cross_sections(G):
    return np.geomspace(4.0, 0.25, G)[:, None] * np.array([[1.0, 0.5]])


def _inputs(case, seed):
    """Everything a run needs, drawn from the seed: plain tensors on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + 12727)
    n, G, S = case["n"], case["groups"], case["sources"]

    def uni(*shape):
        return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)

    if case["layout"] == "lattice":
        side = round(n ** (1 / 3))
        i = (torch.arange(side, device=DEV, dtype=torch.float64) + 0.5) / side
        x = torch.stack([a.reshape(-1) for a in torch.meshgrid(i, i, i, indexing="ij")])
        x = x + 0.2 / side * (2 * uni(3, n) - 1)
        rho = torch.ones(n, device=DEV, dtype=torch.float64)
    elif case["layout"] == "sine":
        def dens(p):
            return 1 + 0.5 * torch.sin(2 * math.pi * p).prod(0)
        cand = uni(3, int(1.6 * n) + 4096)
        keep = 1.5 * uni(cand.shape[1]) < dens(cand)
        x = cand[:, keep][:, :n].contiguous()
        assert x.shape[1] == n
        rho = dens(x)
    else:
        mesh = min(256, max(32, 1 << round(math.log2(n ** (1 / 3)) + 1)))
        f = torch.fft.fftfreq(mesh, 1.0 / mesh, device=DEV, dtype=torch.float64)
        fz = torch.fft.rfftfreq(mesh, 1.0 / mesh, device=DEV, dtype=torch.float64)
        k2 = f[:, None, None] ** 2 + f[None, :, None] ** 2 + fz[None, None, :] ** 2
        amp = torch.where(k2 > 0, k2.clamp(min=0.25).rsqrt(), torch.zeros_like(k2))
        noise = torch.complex(normal(*k2.shape), normal(*k2.shape))
        delta = torch.fft.irfftn(noise * amp, s=(mesh, mesh, mesh))
        delta = delta * (case["sigma"] / delta.std())
        field = torch.exp(delta - 0.5 * case["sigma"] ** 2).reshape(-1)
        weight = torch.round(field * (2.0 ** 30 / float(field.max()))).to(torch.int64)   # whole: the sums are exact
        cum = torch.cumsum(weight, 0)
        cell = torch.searchsorted(cum, (uni(n) * float(cum[-1])).to(torch.int64), right=True).clamp(max=mesh ** 3 - 1)
        x = torch.stack([cell // (mesh * mesh), cell // mesh % mesh, cell % mesh]).to(torch.float64)
        x = (x + uni(3, n)) / mesh
        rho = field[cell] / field.mean()
    x = x - torch.floor(x)
    x = torch.where(x >= 1.0, torch.zeros_like(x), x)
    # the same particles a little later (or earlier): a smooth flow and some random motion
    spacing = n ** (-1 / 3)
    v = 0.1 * spacing * (torch.sin(2 * math.pi * (x.roll(1, 0) + uni(3, 1))) + 0.5 * normal(3, n))
    moved = x + v
    moved = moved - torch.floor(moved)
    moved = torch.where(moved >= 1.0, torch.zeros_like(moved), moved)
    xsrc = uni(3, S)
    L = torch.exp(normal(S, G))
    ts = torch.float64 if case["precision"] == "fp64" else torch.float32
    U = torch.zeros(G, 4, n, device=DEV, dtype=torch.float64)
    E = 1e-10 * (1 + 0.1 * (2 * uni(G, n) - 1))
    dirs = normal(G, 3, n)
    dirs = dirs / dirs.norm(dim=1, keepdim=True)
    U[:, 0] = E
    U[:, 1:] = 0.05 * C_RED * E[:, None] * dirs
    if case["layout"] == "sine":   # a collimated beam along x
        yz = torch.hypot(x[1] - 0.5, x[2] - 0.5)
        beam = (yz < 0.05) & (x[0] >= 0.1) & (x[0] <= 0.2)
        U[:, 0, beam] = 1.0
        U[:, 1, beam] = C_RED
        U[:, 2:, beam] = 0.0
    elif case["kind"] in ("step", "moving", "adjoint"):   # radiation everywhere, as in the midst of a run
        wave = 1 + 0.5 * torch.sin(2 * math.pi * (x[:1] + 2 * x[1:2] + uni(G, 1)))
        U[:, 0] = wave
        U[:, 1:] = 0.3 * C_RED * wave[:, None] * dirs[:, :, :1]
    # a Courant step, from the density that the particles were drawn from.  The densest places of
    # a random sample have half the cell size that it gives, and the explicit scheme, second order
    # in space, needs a third of a cell there (a fifth on clustered gas) to stay stable for long
    dx = 0.62 * (n * rho) ** (-1 / 3)
    dt = (0.5 if case["layout"] == "lattice" else 0.14) * float(dx.min()) / C_RED
    bins = torch.floor(torch.log2(dx / float(dx.min()))).clamp(0, max(case["n_sub"], 0)).to(torch.int32)
    out = {"x": moved.contiguous(), "x_before": x.contiguous(), "v": v.contiguous(), "xsrc": xsrc.contiguous(),
           "L": L.contiguous() if S else None, "U0": U.to(ts).contiguous(), "dt": dt, "bins": bins,
           "alpha": None, "species": None, "sigma": None}
    if case["sink"] == "grey":
        out["alpha"] = (0.1 * rho).contiguous()
    elif case["sink"] == "photo":
        neutral = rho * (0.2 + 0.8 * uni(n))
        out["species"] = torch.stack([neutral, 0.1 * rho]).contiguous()
        out["sigma"] = _cross_sections(G)
    if case["kind"] == "adjoint":   # the loss is the energy in the middle of the box
        inside = (out["x"] - 0.5).norm(dim=0) < 0.15
        w = torch.zeros(G, 4, n, device=DEV, dtype=ts)
        w[:, 0] = inside.to(ts)
        out["weight"] = w
    return out


def prepare(case, seed):
    s = _inputs(case, seed)
    moves = case["kind"] in ("hydro", "moving", "search", "bins")
    first = s["x_before"] if moves else s["x"]
    t = Transport(first, None, s["xsrc"] if case["sources"] else None, n_groups=case["groups"], c_red=C_RED,
                  eta_res=ETA, precision=case["precision"], riemann=case["riemann"])
    if s["species"] is not None:
        t.set_absorbers(s["species"], s["sigma"])
    s["transport"], s["kind"], s["n_sub"], s["pass"] = t, case["kind"], case["n_sub"], 0
    # where the particles are at each pass: they go to and fro, as the next call always finds them moved
    s["where"] = [s["x"], s["x_before"]]
    if case["kind"] == "adjoint":
        s["U0"].requires_grad_(True)
        s["L"].requires_grad_(True)
    return s


def run(s):
    t, k = s["transport"], s["kind"]
    x = s["where"][s["pass"] & 1]
    s["pass"] += 1
    if k == "search":
        t.rebuild(x)
        f = t.fields()
        return {"h": f["h"], "omega": f["omega"], "V": f["V"], "B": f["B"], "pairs": t.diagnostics()["n_pairs"]}
    if k == "adjoint":
        U = SubcycleFunction.apply(s["U0"], s["L"], t, s["n_sub"], s["dt"], None, 4)
        dU0, dL = torch.autograd.grad(U, (s["U0"], s["L"]), s["weight"])
        return {"U": U.detach(), "dU0": dU0, "dL": dL}
    U = s["U0"].clone()
    if k == "step":
        return {"U": t.step(U, s["dt"], s["L"], s["alpha"])}
    if k == "subcycle":
        return {"U": t.subcycle(U, s["n_sub"], s["dt"], s["L"], s["alpha"])}
    if k == "moving":
        t.drift(U, s["v"] if x is s["x"] else -s["v"], 1.0)
    t.rebuild(x)
    if k == "bins":
        t.set_time_bins(s["bins"], dt_min=s["dt"], max_bin=s["n_sub"])
        t.step_bins(U, s["L"], s["alpha"])
        return {"U": U}
    if s["species"] is not None:
        t.set_absorbers(s["species"], s["sigma"])
    t.subcycle(U, s["n_sub"], s["dt"], s["L"], s["alpha"])
    return {"U": U, "energy": t.energy(U)}


# ---------------------------------------------------------------------------------------
# the same in 64 bits
def _w(q):
    return (1 - q).clamp(min=0) ** 3 - 4 * (0.5 - q).clamp(min=0) ** 3


def _dw(q):
    return -3 * (1 - q).clamp(min=0) ** 2 + 12 * (0.5 - q).clamp(min=0) ** 2


def _wrap(d):
    return d - torch.round(d)


def _within(x, centre, R, most=60_000_000):
    """All (i, j) with |x_j - centre_i| < R_i in the periodic unit box, and the separations."""
    got = []
    octave = torch.floor(torch.log2(R / float(R.min())) * 1.0).to(torch.int64)
    for o in torch.unique(octave).tolist():
        ask = torch.nonzero(octave == o)[:, 0]
        nc = int(1.0 / float(R[ask].max()))
        nc = 1 if nc < 3 else min(nc, 512)
        c = (x * nc).to(torch.int64).clamp(max=nc - 1)
        key = (c[2] * nc + c[1]) * nc + c[0]
        order = torch.argsort(key, stable=True)
        count = torch.bincount(key, minlength=nc ** 3)
        start = torch.cumsum(count, 0) - count
        q = (centre[:, ask] * nc).to(torch.int64).clamp(max=nc - 1)
        span = range(-1, 2) if nc > 1 else range(1)
        for dz in span:
            for dy in span:
                for dx in span:
                    cell = (((q[2] + dz) % nc) * nc + (q[1] + dy) % nc) * nc + (q[0] + dx) % nc
                    m = count[cell]
                    upto = torch.cumsum(m, 0)
                    total = int(upto[-1])
                    cuts = [0]
                    while cuts[-1] < len(ask):
                        done = int(upto[cuts[-1] - 1]) if cuts[-1] else 0
                        nxt = len(ask) if total - done <= most else int(torch.searchsorted(upto, done + most))
                        cuts.append(max(nxt, cuts[-1] + 1))
                    for a, b in zip(cuts[:-1], cuts[1:]):
                        mm = m[a:b]
                        i = torch.repeat_interleave(torch.arange(a, b, device=x.device), mm)
                        if not i.numel():
                            continue
                        off = torch.arange(i.numel(), device=x.device) - torch.repeat_interleave(torch.cumsum(mm, 0) - mm, mm)
                        j = order[start[cell[i]] + off]
                        i = ask[i]
                        d = _wrap(x[:, j] - centre[:, i])
                        keep = d.square().sum(0) < R[i].square()
                        got.append((i[keep], j[keep], d[:, keep]))
    return torch.cat([a for a, _, _ in got]), torch.cat([b for _, b, _ in got]), torch.cat([c for _, _, c in got], 1)


def _solve_h(x, centre, h):
    """h = eta omega(h)^(-1/3) by safeguarded Newton steps, and omega (centre may be x itself)."""
    n = centre.shape[1]
    lo, hi = torch.zeros_like(h), torch.full_like(h, math.inf)
    lists = None
    for it in range(80):
        if lists is None or bool((h > reach).any()):
            reach = h * (1.3 if it == 0 else 1.05)
            i, _, d = _within(x, centre, KAPPA * reach)
            lists = (i, d.square().sum(0).sqrt())
        i, r = lists
        q = r / (KAPPA * h[i])
        w = _w(q)
        sw = torch.zeros_like(h).index_add_(0, i, w)
        sd = torch.zeros_like(h).index_add_(0, i, 3 * w + q * _dw(q))
        iH = 1 / (KAPPA * h)
        om = SIGMA * iH ** 3 * sw
        cb = om.clamp(min=1e-300) ** (1 / 3)
        f = torch.where(sw > 0, h - ETA / cb, torch.full_like(h, -math.inf))
        fp = 1 + (ETA / 3) / (cb * om.clamp(min=1e-300)) * (-KAPPA * SIGMA * iH ** 4 * sd)
        lo, hi = torch.where(f < 0, h, lo), torch.where(f < 0, hi, h)
        new = h - f / fp
        bad = ~((new > lo) & (new < hi) & (fp > 0))
        new = torch.where(bad, torch.where(torch.isinf(hi), 1.5 * h, 0.5 * (lo + hi)), new)
        if it > 3 and bool(((f / fp).abs() < 1e-15 * h).logical_or((hi - lo) < 1e-15 * h).all()) or it == 79:
            return h, om
        h = new.clamp(min=0.5 * h, max=2 * h) if it < 8 else new
    return h, om


def _first_h(x, n):
    """A first guess from the counts in nested meshes: the finest where 27 cells hold 40 particles."""
    h = torch.full((n,), ETA * (1.0 / n) ** (1 / 3) * 4, device=x.device, dtype=torch.float64)
    nc = 4
    while nc <= 512:
        c = (x * nc).to(torch.int64).clamp(max=nc - 1)
        count = torch.bincount((c[2] * nc + c[1]) * nc + c[0], minlength=nc ** 3).reshape(nc, nc, nc)
        for a in range(3):
            count = count + count.roll(1, a) + count.roll(-1, a)
        m = count.reshape(-1)[(c[2] * nc + c[1]) * nc + c[0]]
        h = torch.where(m >= 40, ETA * (27.0 / nc ** 3 / m) ** (1 / 3), h)
        nc *= 2
    return h


class _Set:
    """Geometry and pairs of one particle configuration."""

    def __init__(self, x, xsrc, eager=True):
        n = x.shape[1]
        self.n = n
        self.h, self.om = _solve_h(x, x, _first_h(x, n))
        H = KAPPA * self.h
        i, j, _ = _within(x, x, H)
        keep = i != j
        i, j = i[keep], j[keep]
        pair = torch.unique(torch.minimum(i, j) * n + torch.maximum(i, j))
        self.k, self.l = pair // n, pair % n
        self.d = _wrap(x[:, self.l] - x[:, self.k])
        self.r = self.d.square().sum(0).sqrt()
        self.V = 1 / self.om
        self.wk, self.wl = _w(self.r / H[self.k]), _w(self.r / H[self.l])
        fac = SIGMA / H ** 3 * self.V
        dd = (self.d[:, None] * self.d[None]).reshape(9, -1)
        E = torch.zeros(n, 9, device=x.device, dtype=torch.float64)
        E.index_add_(0, self.k, (dd * (fac[self.k] * self.wk)).T.contiguous())
        E.index_add_(0, self.l, (dd * (fac[self.l] * self.wl)).T.contiguous())
        self.B = torch.linalg.inv(E.reshape(n, 3, 3))
        self.fac = fac
        self.d = self.d.T.contiguous()
        psi_k = torch.bmm(self.B[self.k], self.d[:, :, None])[:, :, 0] * (self.V * fac)[self.k, None] * self.wk[:, None]
        psi_l = torch.bmm(self.B[self.l], self.d[:, :, None])[:, :, 0] * (self.V * fac)[self.l, None] * self.wl[:, None]
        self.A = psi_k + psi_l          # V_k psit_l(x_k) - V_l psit_k(x_l), the latter along -d
        self.An = self.A.square().sum(1).sqrt()
        self.ak = (self.h[self.k] / (self.h[self.k] + self.h[self.l]))[:, None]
        self.src = None
        if xsrc is not None and xsrc.shape[1]:
            S = xsrc.shape[1]
            hs, oms = _solve_h(x, xsrc, torch.full((S,), ETA * (1.0 / n) ** (1 / 3), device=x.device, dtype=torch.float64))
            s, g, d = _within(x, xsrc, KAPPA * hs)
            psi = SIGMA / (KAPPA * hs[s]) ** 3 / oms[s] * _w(d.square().sum(0).sqrt() / (KAPPA * hs[s]))
            octant = (d[0] < 0).long() + 2 * (d[1] < 0).long() + 4 * (d[2] < 0).long()
            w8 = torch.zeros(S * 8, device=x.device, dtype=torch.float64).index_add_(0, 8 * s + octant, psi)
            share = w8.reshape(S, 8).sum(1) / (w8.reshape(S, 8) > 0).sum(1)
            self.src = (s, g, psi * share[s] / w8[8 * s + octant] / self.V[g])

    def inject(self, E, L, dt):
        """E [n] of one group, L [S]."""
        if self.src is None or L is None:
            return E
        s, g, xi = self.src
        return E.index_add(0, g, xi * L[s] * dt)

    def gradient(self, U):
        """U [n, 4] -> [n, 4, 3]"""
        dU = U[self.l] - U[self.k]
        acc = torch.zeros(self.n, 12, device=U.device, dtype=U.dtype)
        acc = acc.index_add(0, self.k, (dU[:, :, None] * (self.wk[:, None] * self.d)[:, None]).reshape(-1, 12))
        acc = acc.index_add(0, self.l, (dU[:, :, None] * (self.wl[:, None] * self.d)[:, None]).reshape(-1, 12))
        return torch.bmm(acc.reshape(-1, 4, 3), self.B * self.fac[:, None, None])

    def flux(self, U, grad, table=None):
        """The pair fluxes Phi [P, 4] from the limited face states."""
        a = torch.bmm(grad[self.k], self.d[:, :, None])[:, :, 0]
        b = torch.bmm(grad[self.l], self.d[:, :, None])[:, :, 0]
        zero = torch.zeros((), device=U.device, dtype=U.dtype)
        s = torch.where(torch.sign(a) * torch.sign(b) > 0, torch.where(a.abs() < b.abs(), a, b), zero)
        left, right = U[self.k] + self.ak * s, U[self.l] - (1 - self.ak) * s
        fl, fr = _m1(left, self.A), _m1(right, self.A)
        if table is None:
            return 0.5 * (fl + fr) - 0.5 * C_RED * self.An[:, None] * (right - left)
        xl, nl = _speeds(left, self.A, table)
        xr, nr = _speeds(right, self.A, table)
        lp, lm = torch.maximum(xl, xr).clamp(min=0)[:, None], torch.minimum(nl, nr).clamp(max=0)[:, None]
        span = lp - lm
        hll = (lp * fl - lm * fr + lp * lm * self.An[:, None] * (right - left)) / torch.where(span > 0, span, torch.ones_like(span))
        return torch.where(span > 0, hll, 0.5 * (fl + fr))

    def gathered(self, phi):
        out = torch.zeros(self.n, 4, device=phi.device, dtype=phi.dtype).index_add(0, self.k, phi)
        return out.index_add(0, self.l, -phi)

    def step(self, U, dt, L=None, alpha=None, table=None):
        if L is not None and self.src is not None:
            U = torch.cat([self.inject(U[:, 0], L, dt)[:, None], U[:, 1:]], 1)
        U = U - (dt / self.V)[:, None] * self.gathered(self.flux(U, self.gradient(U), table))
        return U if alpha is None else U * (1 - C_RED * dt * alpha).clamp(min=0)[:, None]


def _m1(U, A):
    """The M1 flux contracted with A; chi = (3 + 4 f^2) / (5 + 2 sqrt(4 - 3 f^2)), f <= 1."""
    E, F = U[:, 0], U[:, 1:]
    FA, F2 = (F * A).sum(1), F.square().sum(1)
    cE = C_RED * E.clamp(min=0)
    q = torch.maximum(F2, cE.square())
    iq = torch.where(q > 0, 1 / torch.where(q > 0, q, torch.ones_like(q)), torch.zeros_like(q))
    u = F2 * iq
    s = torch.sqrt(4 - 3 * u)
    iso = (1 + s - 2 * u) / (5 + 2 * s)
    along = 3 * iq / (2 + s) * FA
    return torch.cat([FA[:, None], (C_RED * cE)[:, None] * (iso[:, None] * A + along[:, None] * F)], 1)


_TABLE = []


def _wave_table():
    """Extreme eigenvalues of the M1 flux Jacobian along n over (f, theta), 101 x 101."""
    if not _TABLE:
        f = np.linspace(0, 1, 101)[:, None] * np.ones((1, 101))
        th = np.linspace(0, np.pi, 101)[None] * np.ones((101, 1))
        base = np.stack([np.ones_like(f), f * np.cos(th), f * np.sin(th), 0 * f], -1)
        J = np.empty(f.shape + (4, 4))
        for b in range(4):   # complex steps along each variable
            u = base.astype(complex)
            u[..., b] += 1e-30j
            f2 = (u[..., 1:] ** 2).sum(-1) / u[..., 0] ** 2
            chi = (3 + 4 * f2) / (5 + 2 * np.sqrt(4 - 3 * f2))
            safe = np.where(np.abs(f2) > 1e-40, f2, 1)
            along = np.where(np.abs(f2) > 1e-40, (3 * chi - 1) / 2 / safe, 0.75) * u[..., 1] / u[..., 0]
            J[..., 0, b] = u[..., 1].imag / 1e-30
            for a in range(3):
                J[..., a + 1, b] = ((u[..., 0] * (1 - chi) / 2 if a == 0 else 0) + along * u[..., 1 + a]).imag / 1e-30
        ev = np.linalg.eigvals(J).real
        hi, lo = ev.max(-1), ev.min(-1)
        hi[100], lo[100] = np.cos(th[100]), np.cos(th[100])   # free streaming: a fourfold root
        _TABLE.append(torch.from_numpy(np.stack([hi, lo], -1)).to(DEV).reshape(-1, 2))
    return _TABLE[0]


def _speeds(U, A, table):
    E, F = U[:, 0], U[:, 1:]
    Fn = F.square().sum(1).sqrt()
    pos = E > 0
    f = torch.where(pos, Fn / (C_RED * torch.where(pos, E, torch.ones_like(E))), torch.zeros_like(E)).clamp(max=1)
    th = torch.atan2(torch.linalg.cross(F, A).square().sum(1).sqrt(), (F * A).sum(1))
    x, y = f * 100, th / math.pi * 100
    i, j = x.to(torch.int64).clamp(max=99), y.to(torch.int64).clamp(max=99)
    t, s = (x - i)[:, None], (y - j)[:, None]
    at = i * 101 + j
    v = (1 - t) * (1 - s) * table[at] + t * (1 - s) * table[at + 101] + (1 - t) * s * table[at + 1] + t * s * table[at + 102]
    v = torch.where(pos[:, None], C_RED * v, torch.tensor([C_RED, -C_RED], device=U.device, dtype=U.dtype))
    return v[:, 0], v[:, 1]


def _bin_steps(ps, U, bins, dt_min, B, L):
    """One hydro step with individual time bins (one group)."""
    b = bins.to(torch.int64)
    while True:   # interacting particles differ by two bins at most
        m = b.clone()
        m.scatter_reduce_(0, ps.k, b[ps.l] + 2, "amin")
        m.scatter_reduce_(0, ps.l, b[ps.k] + 2, "amin")
        if torch.equal(m, b):
            break
        b = m
    top = int(b.max())
    span = 2 ** b
    grad = torch.zeros(ps.n, 4, 3, device=U.device, dtype=U.dtype)
    acc = torch.zeros(ps.n, 4, device=U.device, dtype=U.dtype)
    both = torch.minimum(span[ps.k], span[ps.l]).to(U.dtype)
    for s in range(2 ** top):
        starts = s % span == 0
        if ps.src is not None and L is not None:
            src, g, xi = ps.src
            add = torch.zeros_like(U[:, 0]).index_add(0, g, xi * L[src] * dt_min)
            U = torch.cat([(U[:, 0] + torch.where(starts, add * span, torch.zeros_like(add)))[:, None], U[:, 1:]], 1)
        grad = torch.where(starts[:, None, None], ps.gradient(U), grad)
        on = (starts[ps.k] | starts[ps.l]).to(U.dtype)
        acc = acc + ps.gathered(ps.flux(U, grad) * (both * on)[:, None])
        ends = (s + 1) % span == 0
        U = torch.where(ends[:, None], U - (dt_min / ps.V)[:, None] * acc, U)
        acc = torch.where(ends[:, None], torch.zeros_like(acc), acc)
    return U


def exact(case, seed):
    s = _inputs(case, seed)
    k, G, dt = case["kind"], case["groups"], s["dt"]
    xsrc = s["xsrc"] if case["sources"] else None
    U0 = s["U0"].to(torch.float64)
    if k == "moving":
        before = _Set(s["x_before"], None)
        U0 = torch.stack([(U0[g].T + torch.bmm(before.gradient(U0[g].T.contiguous()), s["v"].T[:, :, None])[:, :, 0]).T for g in range(G)])
        del before
    ps = _Set(s["x"], xsrc)
    if k == "search":
        return {"h": ps.h, "omega": ps.om, "V": ps.V, "B": ps.B, "pairs": int(ps.k.numel())}
    table = _wave_table() if case["riemann"] == "hll" else None
    L, out = s["L"], []
    if k == "adjoint":
        U0.requires_grad_(True)
        L = L.clone().requires_grad_(True)
    for g in range(G):
        U = U0[g].T.contiguous()
        Lg = None if L is None else L[:, g]
        alpha = s["alpha"]
        if s["species"] is not None:
            alpha = (torch.from_numpy(s["sigma"][g]).to(DEV)[:, None] * s["species"]).sum(0)
        if k == "bins":
            out.append(_bin_steps(ps, U, s["bins"].clamp(0, case["n_sub"]), dt, case["n_sub"], Lg).T)
            continue
        for _ in range(case["n_sub"]):
            U = ps.step(U, dt, Lg, alpha, table)
        out.append(U.T)
    U = torch.stack(out)
    if k == "adjoint":
        dU0, dL = torch.autograd.grad(U, (U0, L), s["weight"].to(torch.float64))
        return {"U": U.detach(), "dU0": dU0, "dL": dL}
    if k in ("hydro", "moving"):
        return {"U": U, "energy": [float((ps.V * U[g, 0]).sum()) for g in range(G)]}
    return {"U": U}
