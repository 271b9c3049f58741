"""The work that users of this library have it do, as cases that can be timed.

A case is one call chain of a simulation in progress: whole time steps of a
domain (lbm_step), of several domains on streams of their own, or of a batch
(lbm_batch_step); a small study job from host arrays to host arrays; or the
readings that a study takes between its chunks of steps.  Sizes and parameters
are those of the benchmark workloads, the studies, the served job mix and the
tests of this repository, and draw() spreads over the same ranges.

Step cases return the populations themselves: the domain's device buffers come
from torch tensors (the allocator hook of lbm_params), and after an even number
of steps the population buffer is in canonical order [i, z, y, x].

exact() restates the method in plain torch float64.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

from paper_2201_12404_gb300 import lbm

EOS = dict(a=0.003, b=0.095, R=1.0, acentric=0.344)
WIDTH = 5.0                 # interface width of the initial profiles
PRECISION = {"fp64": lbm.LBM_FP64, "fp32": lbm.LBM_FP32, "fp16dev": lbm.LBM_FP16DEV}
STORED = {"fp64": torch.float64, "fp32": torch.float32, "fp16dev": torch.float16}
BYTES = {"fp64": 8, "fp32": 4, "fp16dev": 2}
# floating-point operations of one update of a node (moments, force stencil,
# equilibria, split, entropic sums, relaxation), counted from the formulas
FLOPS = {2: 400.0, 3: 1400.0}


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def _case(name, kind, D, nx, ny, nz, precision, steps, T=0.59, kappa=0.01, nu=0.005, nu_ratio=1.0, radius=0.0,
          film=0.0, speed=0.0, walls=True, **more):
    return dict(name=name, kind=kind, D=D, nx=nx, ny=ny, nz=nz, precision=precision, steps=steps, T=T, kappa=kappa,
                nu=nu, nu_ratio=nu_ratio, radius=radius, film=film, speed=speed, walls=walls, **more)


def listed():
    return [
        # the smallest domain: the benchmark's periodic static drop (spurious currents,
        # Laplace's law), where the latency of a step counts
        _case("static2d_128x128_fp32", "steps", 2, 128, 128, 1, "fp32", 100, T=0.8, kappa=0.002, nu=0.01, radius=25.0,
              walls=False),
        # the coexistence study's column in the reference precision, as a study job: fields
        # from host arrays, steps, fields back to host arrays
        _case("coexist2d_800x10_fp64", "study", 2, 800, 10, 1, "fp64", 100, T=0.7, kappa=0.005, nu=0.1, walls=False),
        # the benchmark's 2-D drop impact
        _case("impact2d_2048x1024_fp32", "steps", 2, 2048, 1024, 1, "fp32", 20, nu=0.0064, nu_ratio=21.0, radius=128.0,
              film=25.6, speed=0.05),
        # the stability study's impact box with half-precision storage
        _case("impact2d_1200x600_fp16dev", "steps", 2, 1200, 600, 1, "fp16dev", 20, T=0.7, nu=0.02, radius=50.0,
              film=50.0, speed=0.03),
        # the coexistence sweep: 16 uneven 2-D jobs in one batch
        _case("batch2d_16jobs_fp32", "batch", 2, 64, 256, 1, "fp32", 20, T=0.6, kappa=0.005, nu=0.1, walls=False, jobs=16),
        # a small served 3-D job, odd sides
        _case("impact3d_67x67x67_fp32", "steps", 3, 67, 67, 67, "fp32", 40, T=0.75, nu=0.03, radius=13.0, film=13.0,
              speed=0.02),
        # the resident 3-D jobs of the server: cubes of several sizes, a stream each
        _case("serve3d_4jobs_fp32", "streams", 3, 64, 64, 64, "fp32", 10, T=0.7, nu=0.02, radius=12.0, film=12.0,
              speed=0.03, jobs=4),
        # a medium 3-D impact with ragged sides
        _case("impact3d_203x187x149_fp32", "steps", 3, 203, 187, 149, "fp32", 10, nu=0.01, nu_ratio=15.0, radius=30.0,
              film=13.0, speed=0.04),
        # the headline workload: drop impact on a thin film at full size
        _case("impact3d_512x512x256_fp32", "steps", 3, 512, 512, 256, "fp32", 4, nu_ratio=21.0, radius=64.0, film=12.8,
              speed=0.04),
        # the same at half the resolution, half-precision storage
        _case("impact3d_256x256x128_fp16dev", "steps", 3, 256, 256, 128, "fp16dev", 10, nu_ratio=21.0, radius=32.0,
              film=6.4, speed=0.04),
        # the reference precision in 3-D
        _case("impact3d_128x128x64_fp64", "steps", 3, 128, 128, 64, "fp64", 4, T=0.7, nu=0.02, radius=16.0, film=8.0,
              speed=0.03),
        # what a study reads after each chunk of steps: totals, largest speed, interface
        # width, crown radius
        _case("readings3d_256x256x128_fp32", "readings", 3, 256, 256, 128, "fp32", 0, nu_ratio=21.0, radius=32.0,
              film=12.0, speed=0.04),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choices(["steps2", "steps3", "batch", "streams", "study", "readings"], [4, 5, 1, 1, 1, 1])[0]
    T, kappa = rng.uniform(0.68, 0.85), rng.choice([0.005, 0.01])
    nu, ratio, speed = math.exp(rng.uniform(math.log(0.015), math.log(0.08))), rng.choice([1.0, 1.0, 8.0]), rng.uniform(0.0, 0.04)
    more = dict(T=round(T, 3), kappa=kappa, nu=round(nu, 4), nu_ratio=ratio, speed=round(speed, 4), walls=rng.random() < 0.7)
    if kind in ("steps2", "study"):
        D, nz = 2, 1
        nx, ny = (_log(rng, 60, 2048), _log(rng, 60, 1024)) if kind == "steps2" else (_log(rng, 100, 800), _log(rng, 8, 200))
        precision = rng.choices(["fp32", "fp16dev", "fp64"], [6, 2, 2])[0] if kind == "steps2" else "fp64"
    elif kind == "batch":
        D, nx, ny, nz, precision = 2, _log(rng, 40, 80), _log(rng, 100, 300), 1, "fp32"
        more.update(jobs=rng.randint(3, 20))
    else:
        D, hi = 3, 100 if kind == "streams" else 300
        nx, ny, nz = (_log(rng, 40, hi) for _ in range(3))
        precision = rng.choices(["fp32", "fp16dev", "fp64"], [7, 2, 1])[0] if kind == "steps3" else "fp32"
        if kind == "streams":
            more.update(jobs=rng.randint(2, 6))
        if precision == "fp64":
            nx, ny, nz = min(nx, 120), min(ny, 120), min(nz, 80)
    shortest = min(v for v in (nx, ny, nz) if v > 1)
    more.update(radius=round(rng.uniform(0.12, 0.22) * shortest, 1), film=round(rng.uniform(0.1, 0.2) * (ny if D == 2 else nz), 1) if more["walls"] else 0.0)
    shape = dict(kind=kind, D=D, nx=nx, ny=ny, nz=nz, **more)
    budget = (3e6 if D == 2 else 2e6) if precision == "fp64" else 4e7 if D == 2 else 6e7
    steps = 0 if kind == "readings" else 2 * max(1, min(50, int(budget / sum(m[0] * m[1] * m[2] for m in _members(shape)) / 2)))
    c = _case("", {"steps2": "steps", "steps3": "steps"}.get(kind, kind), D, nx, ny, nz, precision, steps, **more)
    del c["name"]
    return c


def _members(case):
    """The domains of a case: (nx, ny, nz, T) each.  A batch grows its jobs' sides in
    four steps and spreads their temperatures as the coexistence sweep does; the served
    cubes grow by a third each."""
    jobs = case.get("jobs", 1)
    if case["kind"] == "batch":
        return [((1 + k % 4) * case["nx"], (1 + k % 4) * case["ny"], 1, case["T"] + (0.9 - case["T"]) * k / max(1, jobs - 1))
                for k in range(jobs)]
    return [tuple(int(round(case[s] * (1 + k / 3.0))) for s in ("nx", "ny", "nz")) + (case["T"],) if case["D"] == 3
            else (case["nx"], case["ny"], 1, case["T"]) for k in range(jobs)]


def work(case):
    Q, nodes = (9 if case["D"] == 2 else 27), float(sum(m[0] * m[1] * m[2] for m in _members(case)))
    fields = 8.0 * (1 + case["D"]) * nodes
    if case["kind"] == "readings":  # the populations once, for the totals and the density and velocity fields alike
        return {"bytes": nodes * Q * BYTES[case["precision"]], "flops": nodes * 150.0}
    w = {"bytes": case["steps"] * nodes * 2 * Q * BYTES[case["precision"]], "flops": case["steps"] * nodes * FLOPS[case["D"]]}
    if case["kind"] == "study":
        w["bytes"] += 2 * fields
    return w


# ---------------------------------------------------------------------------
# Preparation and the pass
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _coexistence(T):
    """Densities of vapour and liquid (Maxwell equal areas) of the Peng-Robinson fluid, float64."""
    P = lambda r: _pressure(r, T)  # noqa: E731
    r = np.linspace(1e-4, 0.97 / EOS["b"], 400001)
    dp = np.diff(P(r))
    spin = r[np.flatnonzero(np.diff(np.sign(dp)))]
    lo, hi = float(spin[0]), float(spin[-1])  # the spinodals

    def root(p, a, b, rising):
        for _ in range(200):
            m = 0.5 * (a + b)
            a, b = (m, b) if (P(m) < p) == rising else (a, m)
        return 0.5 * (a + b)

    x, w = np.polynomial.legendre.leggauss(400)

    def area(p):
        """Integral of (P - p)/rho^2 between the phases, over nodes even in log rho."""
        v, l = root(p, 1e-12, lo, True), root(p, hi, 0.99 / EOS["b"], True)
        half = 0.5 * math.log(l / v)
        s = v * np.exp(half * (x + 1.0))
        return float(np.sum(w * (P(s) - p) / s)) * half, v, l

    a, b = max(float(P(hi)), 1e-12), float(P(lo))
    for _ in range(100):
        m = 0.5 * (a + b)
        if area(m)[0] > 0:
            a = m
        else:
            b = m
    _, v, l = area(0.5 * (a + b))
    return v, l


def _alpha_T(T):
    Tc = 0.0778 * EOS["a"] / (0.45724 * EOS["b"] * EOS["R"])
    m = 0.37464 + 1.54226 * EOS["acentric"] - 0.26992 * EOS["acentric"] ** 2
    return EOS["R"] * T * Tc, EOS["a"] * (1.0 + m * (1.0 - math.sqrt(T))) ** 2


def _pressure(rho, T):
    RT, aalpha = _alpha_T(T)
    b = EOS["b"]
    return rho * RT / (1.0 - b * rho) - aalpha * rho * rho / (1.0 + 2.0 * b * rho - b * b * rho * rho)


def _geometry(case, seed, k, nx, ny, nz):
    """Initial geometry of domain k, varied by the seed: drop radius, film, gap, speed, width."""
    r = random.Random(1000003 * int(seed) + k)
    tall = nz if case["D"] == 3 else ny
    scale = nx / case["nx"]
    g = dict(radius=case["radius"] * scale * r.uniform(0.97, 1.03), film=case["film"] * scale, speed=case["speed"] * r.uniform(0.9, 1.0),
             width=WIDTH * r.uniform(0.98, 1.02))
    # over a film: two widths above it; otherwise centred
    g["gap"] = 2.0 * g["width"] if g["film"] > 0 else 0.5 * (tall - 1) - g["radius"] + r.uniform(-0.4, 0.4)
    return g


def _slab(case, seed, k, nx, ny):
    """Flat liquid layer over the middle half of the longer side: (density, velocity) on the host."""
    r = np.random.default_rng([int(seed), k])
    rv, rl = _coexistence(_members(case)[k][3])
    along = np.arange(max(nx, ny), dtype=np.float64)
    lo = len(along) * 0.25 + r.uniform(-0.5, 0.5)
    d = np.maximum(lo - along, along - (lo + 0.5 * len(along)))
    rho = 0.5 * (rl + rv) - 0.5 * (rl - rv) * np.tanh(2.0 * d / WIDTH)
    rho = rho[None, :] if nx >= ny else rho[:, None]
    rho = np.broadcast_to(rho, (ny, nx)) * (1.0 + r.uniform(-1e-6, 1e-6, (ny, nx)))
    return np.ascontiguousarray(rho)[None], np.zeros((2, 1, ny, nx))


class _Buffers:
    """Device memory of a domain from torch tensors, through the allocator hook."""

    def __init__(self):
        self.tensors, self.first = {}, None
        self.alloc, self.free = lbm.DEV_ALLOC(self._alloc), lbm.DEV_FREE(self._free)

    def _alloc(self, nbytes, ctx):
        try:
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
        except RuntimeError:
            return None
        self.tensors[t.data_ptr()] = t
        if self.first is None:
            self.first = t  # the populations are a domain's first buffer
        return t.data_ptr()

    def _free(self, ptr, ctx):
        self.tensors.pop(int(ptr), None)


@functools.lru_cache(maxsize=None)
def _stream():
    """The stream the program steps its domains on."""
    return torch.cuda.Stream()


def _params(case, k):
    nx, ny, nz, T = _members(case)[k]
    rv, rl = _coexistence(T)
    bc = [0] * 6
    if case["walls"]:
        bc[2 * case["D"] - 2] = bc[2 * case["D"] - 1] = 1
    return lbm.lbm_default_params(
        lattice=lbm.LBM_D3Q27 if case["D"] == 3 else lbm.LBM_D2Q9, precision=PRECISION[case["precision"]], nx=nx, ny=ny,
        nz=nz, T_over_Tc=T, kappa=case["kappa"], nu_liquid=case["nu"], nu_vapour=case["nu"] * case["nu_ratio"],
        rho_liquid=rl, rho_vapour=rv, bc=bc,
        # the served domains run side by side, each on a stream that the library makes
        stream=None if case["kind"] == "streams" else _stream().cuda_stream, **EOS)


def prepare(case, seed):
    doms, pops = [], []
    for k, (nx, ny, nz, _) in enumerate(_members(case)):
        p, mem = _params(case, k), _Buffers()
        p.dev_alloc, p.dev_free = mem.alloc, mem.free
        dom = lbm.Domain(p)
        if case["kind"] == "batch":
            dom.lbm_init_fields(*_slab(case, seed, k, nx, ny))
        elif case["kind"] != "study":
            dom.lbm_init_drop_on_film(**_geometry(case, seed, k, nx, ny, nz))
        doms.append(dom)
        Q = 9 if case["D"] == 2 else 27
        pops.append(mem.first.view(STORED[case["precision"]])[: Q * nx * ny * nz].view(Q, nz, ny, nx))
    s = dict(case=case, domains=doms, populations=pops)
    if case["kind"] == "batch":
        s["batch"] = lbm.Batch(doms)
    if case["kind"] == "study":
        s["fields"] = _slab(case, seed, 0, case["nx"], case["ny"])
    return s


def run(state):
    case, doms = state["case"], state["domains"]
    if case["kind"] == "study":
        doms[0].lbm_init_fields(*state["fields"])
        doms[0].lbm_step(case["steps"])
        return list(doms[0].lbm_read_macroscopic())
    if case["kind"] == "readings":
        totals = doms[0].lbm_read_diag()
        width, grad = doms[0].lbm_interface_width()
        return dict(mass=totals["mass"], momentum=totals["momentum"], max_u=totals["max_u"], speed=doms[0].lbm_max_speed(),
                    width=width, grad=grad, crown=doms[0].lbm_crown_radius(_layer(case)))
    if case["kind"] == "batch":
        state["batch"].lbm_batch_step(case["steps"])
    else:
        for d in doms:
            d.lbm_step(case["steps"])
    return list(state["populations"])


def _layer(case):
    """The layer two nodes above the film, where the crown is sampled."""
    return int(case["film"]) + 2


# ---------------------------------------------------------------------------
# The method in float64
# ---------------------------------------------------------------------------

class _Reference:
    """One domain of the two-phase entropic lattice Boltzmann method in torch float64:
    arrays [.., z, y, x], populations indexed (cx+1) + 3 (cy+1) + 9 (cz+1)."""

    def __init__(self, case, k):
        self.nx, self.ny, self.nz, self.T = _members(case)[k]
        self.D, self.case = case["D"], case
        self.rv, self.rl = _coexistence(self.T)
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.c = [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1 if self.D == 3 else 0) for i in range(9 if self.D == 2 else 27)]
        w1 = {0: 2 / 3, 1: 1 / 6, -1: 1 / 6}
        self.w = [w1[c[0]] * w1[c[1]] * (w1[c[2]] if self.D == 3 else 1.0) for c in self.c]
        self.wall = [case["walls"] and a == self.D - 1 for a in range(3)]

    def at(self, field, shift, odd=False):
        """field(r + shift): periodic, or mirrored across half-way walls (odd: negated there)."""
        for a, s in enumerate(shift):
            if s == 0:
                continue
            dim = field.dim() - 1 - a
            n = field.shape[dim]
            if not self.wall[a]:
                field = torch.roll(field, -s, dim)
                continue
            i = torch.arange(n, device=field.device) + s
            out = (i < 0) | (i >= n)
            i = torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i))
            field = field.index_select(dim, i)
            if odd:
                shape = [1] * field.dim()
                shape[dim] = n
                field = field * torch.where(out, -1.0, 1.0).to(field.dtype).view(shape)
        return field

    def psi(self, rho):
        d = _pressure(rho, self.T) - rho / 3.0
        return d.abs().sqrt(), torch.where(d > 0, 1.0, -1.0).to(rho.dtype)

    def force(self, rho):
        psi, s = self.psi(rho)
        G3, G4 = ([torch.zeros_like(rho) for _ in range(self.D)] for _ in range(2))
        for c, w in zip(self.c, self.w):
            if any(c):
                far = tuple(2 * v for v in c)
                t3 = 2.0 * self.at(rho, c) - self.at(rho, far)
                t4 = (4.0 / 3.0) * self.at(psi, c) - self.at(psi, far) / 6.0
                for a in range(self.D):
                    if c[a]:
                        G3[a] += 3.0 * w * c[a] * t3
                        G4[a] += 3.0 * w * c[a] * t4
        return [-(2.0 * s * psi * G4[a] + self.case["kappa"] * rho * G3[a]) for a in range(self.D)]

    @staticmethod
    def factors(xi, zeta):
        """The one-dimensional factors for c = -1, 0, +1."""
        return (0.5 * (zeta - xi), 1.0 - zeta, 0.5 * (zeta + xi))

    def product(self, i, F):
        p = F[0][self.c[i][0] + 1] * F[1][self.c[i][1] + 1]
        return p * F[2][self.c[i][2] + 1] if self.D == 3 else p

    def moments(self, f):
        rho = f.sum(0)
        j = [sum(c[a] * f[i] for i, c in enumerate(self.c) if c[a]) for a in range(self.D)]
        return rho, j

    def equilibrium(self, rho, u):
        E = [self.factors(v, 1.0 / 3.0 + v * v) for v in u]
        return torch.stack([rho * self.product(i, E) for i in range(len(self.c))])

    def rest(self, rho, u):
        """The state whose reported velocity is u."""
        F = self.force(rho)
        return self.equilibrium(rho, [u[a] - F[a] / (2.0 * rho) for a in range(self.D)])

    def step(self, f):
        D, Q = self.D, len(self.c)
        rho, j = self.moments(f)
        phi = ((rho - self.rv) / (self.rl - self.rv)).clamp(0.0, 1.0)
        nu_v = self.case["nu"] * self.case["nu_ratio"]
        om = 1.0 / (3.0 * (nu_v + phi * (self.case["nu"] - nu_v)) + 0.5)
        u = [v / rho for v in j]
        F = self.force(rho)
        E, S, D1 = [], [], []
        for a in range(D):
            q = rho * ((j[a] + 0.5 * F[a]) / rho) ** 3
            e = tuple(1 if b == a else 0 for b in range(3))
            m = tuple(-v for v in e)
            Phi = (1.0 - 0.5 * om) * 0.5 * (self.at(q, m, odd=True) - self.at(q, e, odd=True))
            xs = u[a] + F[a] / rho
            E.append(self.factors(u[a], 1.0 / 3.0 + u[a] * u[a]))
            S.append(self.factors(xs, 1.0 / 3.0 + xs * xs + Phi / rho))
            D1.append((u[a] - 0.5, -2.0 * u[a], u[a] + 0.5))
        # second-order central moments: off-diagonal and deviatoric parts are the shear
        Pi = lambda a, b: sum(c[a] * c[b] * f[i] for i, c in enumerate(self.c) if c[a] * c[b])  # noqa: E731
        off = {(a, b): Pi(a, b) - rho * u[a] * u[b] for a in range(D) for b in range(a + 1, D)}
        dia = [Pi(a, a) - rho * u[a] * u[a] - rho / 3.0 for a in range(D)]
        tr = sum(dia) / D
        d2 = (0.5, -1.0, 0.5)

        def shear(i):
            k = [self.c[i][a] + 1 for a in range(D)]
            s = torch.zeros_like(rho)
            for (a, b), m in off.items():
                t = m * D1[a][k[a]] * D1[b][k[b]]
                for e in range(D):
                    if e not in (a, b):
                        t = t * E[e][k[e]]
                s += t
            for a in range(D):
                t = (dia[a] - tr) * d2[k[a]]
                for e in range(D):
                    if e != a:
                        t = t * E[e][k[e]]
                s += t
            return s

        A, B, least = torch.zeros_like(rho), torch.zeros_like(rho), torch.full_like(rho, math.inf)
        for i in range(Q):
            s, feq, fst = shear(i), rho * self.product(i, E), rho * self.product(i, S)
            h = f[i] - feq - s
            A += s * h / fst
            B += h * h / fst
            least = torch.minimum(least, fst)
        ratio = torch.where(B > 1e-300, A / B, torch.zeros_like(A))
        gamma = torch.where(least > 0, 2.0 / om - (2.0 - 2.0 / om) * ratio, torch.full_like(A, 2.0))
        out = torch.empty_like(f)
        for i in range(Q):
            s, feq, fst = shear(i), rho * self.product(i, E), rho * self.product(i, S)
            post = f[i] - om * s - 0.5 * om * gamma * (f[i] - feq - s) + fst - feq
            self.stream(out, i, post)
        return out

    def stream(self, out, i, post):
        c, a = self.c[i], self.D - 1
        dim = post.dim() - 1 - a
        n, way = post.shape[dim], c[a] if self.wall[a] else 0
        moved = torch.roll(post, tuple(v for v in c[: self.D]), tuple(post.dim() - 1 - b for b in range(self.D)))
        if way == 0:
            out[i].copy_(moved)
            return
        # what crosses the wall comes back reversed at its own node
        edge = n - 1 if way > 0 else 0
        inner = slice(1, n) if way > 0 else slice(0, n - 1)
        pick = [slice(None)] * post.dim()
        pick[dim] = inner
        out[i][tuple(pick)] = moved[tuple(pick)]
        pick[dim] = slice(edge, edge + 1)
        out[len(self.c) - 1 - i][tuple(pick)] = post[tuple(pick)]

    def drop(self, radius, film, gap, speed, width):
        g = dict(dtype=torch.float64, device=self.dev)
        z, y, x = torch.meshgrid(torch.arange(self.nz, **g), torch.arange(self.ny, **g), torch.arange(self.nx, **g), indexing="ij")
        tall = z if self.D == 3 else y
        r2 = (x - 0.5 * (self.nx - 1)) ** 2 + (tall - (film + radius + gap)) ** 2
        if self.D == 3:
            r2 = r2 + (y - 0.5 * (self.ny - 1)) ** 2
        d_drop = r2.sqrt() - radius
        dist = torch.minimum(d_drop, tall - (film - 0.5)) if film > 0 else d_drop
        rho = 0.5 * (self.rl + self.rv) - 0.5 * (self.rl - self.rv) * torch.tanh(2.0 * dist / width)
        u = [torch.zeros_like(rho) for _ in range(self.D)]
        u[-1] = -speed * (0.5 - 0.5 * torch.tanh(2.0 * d_drop / width))
        return rho, u

    def deviations(self, f, rho_before):
        """The stored form of half precision: f_i/(w_i rho_w) - 1, rho_w the density that the
        node a population came from had before its collision."""
        scale = torch.empty_like(f)
        for i, w in enumerate(self.w):
            self.stream(scale, i, w * rho_before)
        return f / scale - 1.0


def exact(case, seed):
    outs = []
    for k, (nx, ny, nz, _) in enumerate(_members(case)):
        m = _Reference(case, k)
        if case["kind"] in ("batch", "study"):
            rho, u = (torch.from_numpy(v).to(m.dev) for v in _slab(case, seed, k, nx, ny))
            u = list(u)
        else:
            rho, u = m.drop(**_geometry(case, seed, k, nx, ny, nz))
        f = m.rest(rho, u)
        for _ in range(case["steps"]):
            before = f
            f = m.step(f)
        if case["precision"] == "fp16dev":
            f = m.deviations(f, before.sum(0))
        if case["kind"] == "study":
            rho, j = m.moments(f)
            F = m.force(rho)
            return [rho.cpu().numpy(), torch.stack([(j[a] + 0.5 * F[a]) / rho for a in range(m.D)]).cpu().numpy()]
        if case["kind"] == "readings":
            return _exact_readings(case, m, f)
        outs.append(f)
    return outs


def _exact_readings(case, m, f):
    rho, j = m.moments(f)
    F = m.force(rho)
    length = lambda v: float(sum(t * t for t in v).sqrt().max())  # noqa: E731
    e = lambda a, s: tuple(s if b == a else 0 for b in range(3))  # noqa: E731
    grad = length([0.5 * (m.at(rho, e(a, 1)) - m.at(rho, e(a, -1))) for a in range(m.D)])
    layer = rho[_layer(case)] if m.D == 3 else rho[0, _layer(case)][None]
    y, x = torch.nonzero(layer > 0.5 * (m.rl + m.rv), as_tuple=True)
    dx, dy = x - 0.5 * (m.nx - 1), (y - 0.5 * (m.ny - 1)) if m.D == 3 else 0.0 * x
    crown = float((dx * dx + dy * dy).sqrt().max()) if len(x) else 0.0
    mom = np.zeros(3)
    mom[: m.D] = [float(v.sum()) for v in j]
    return dict(mass=float(rho.sum()), momentum=mom, max_u=length([v / rho for v in j]),
                speed=length([(j[a] + 0.5 * F[a]) / rho for a in range(m.D)]), width=(m.rl - m.rv) / grad, grad=grad, crown=crown)
