"""The work a program gives this library, as cases that can be timed.

One case is one radiation step (or a group of them) through the public entry
points: fld_step on a resident context, fld_step_host on host buffers,
fld_step_batched over a handful of requests, the opacity update between
steps, and a multigroup step with its group fields and rates.  The grids run
from the smallest request of the serving stream (16^3) to the benchmark's
512^3 box; shapes that are not powers of two, every boundary kind, both
limiters, both time discretisations and both precisions are among them.

A pass of a device-buffer case starts from the same E^n: the program's other
operators (advection, here a copy) hand E over before each radiation step.
"""
import math

import numpy as np
import torch

from paper_1306_0645_gb300 import fld, synth

KPC, YEAR, HNU, C, SIGMA, NDOT = synth.KPC, synth.YEAR, synth.HNU_HI, synth.C_LIGHT, synth.SIGMA_HI, synth.NDOT
BOX, DT = synth.BOX, synth.DT
COLD = 1e-30            # erg/cm^3, the initial E of the paper's tests

# Lower edges of 2 to 5 frequency groups, in units of nu_HI: the helium
# thresholds and splits above them; the spectrum ends at 1000.
EDGES = {2: (1.0, 4.0), 3: (1.0, 24.6 / 13.6, 4.0), 4: (1.0, 24.6 / 13.6, 4.0, 10.0),
         5: (1.0, 24.6 / 13.6, 4.0, 6.0, 10.0)}


def _case(name, kind, n, **more):
    c = {"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "precision": "mixed", "bc": "closed",
         "theta": 1.0, "limiter": "paper", "medium": "uniform", "mean": 1e-3, "sigma_ln": 0.0, "sources": 1,
         "state": "cold", "box_kpc": 6.6, "persistent": 0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest request of the serving stream, with the server's
        # persistent inner solves: latency of one small call
        _case("request_16", "step", (16, 16, 16), sources=24, persistent=8192),
        # a small ragged subvolume cut from a larger box: x extents that are
        # multiples of 4 but not 8 and then of 2 only, a periodic axis, an
        # outflow face, trapezoidal rule
        _case("ragged_44x36x28", "step", (44, 36, 28), bc="ragged", theta=0.5, medium="clumps", sigma_ln=1.0,
              sources=40, state="lit"),
        # the single-source verification problem in plain FP64 (config 1)
        _case("single_source_32_fp64", "step", (32, 32, 32), precision="fp64", limiter="lp"),
        # a middle request of the serving stream
        _case("request_64", "step", (64, 64, 64), sources=33),
        # eight requests that arrived together, stepped in one call
        _case("batch_8", "batch", (64, 64, 64), sizes="16,48,32,64,16,32,64,48", sources=17, persistent=8192),
        # two merging HII regions (Sec. 4.1): a long box with outflow faces
        _case("two_sources_128x64x64", "step", (128, 64, 64), bc="outflow", theta=0.5, sources=2, state="lit",
              box_kpc=20.0),
        # the cosmological box in plain FP64 (config 2): periodic, ionised
        # around the sources
        _case("cosmological_128_fp64", "step", (128, 128, 128), precision="fp64", bc="periodic", medium="ionised",
              mean=2e-4, sigma_ln=1.0, sources=256, state="lit"),
        # four frequency groups stepped together: group fields, the step of
        # every group, the photoionisation and heating rates
        _case("multigroup_128", "groups", (128, 128, 128), groups=4, medium="clumps", sigma_ln=1.0, sources=512,
              state="lit"),
        # a periodic box whose extents are not powers of two
        _case("periodic_192x160x224", "step", (192, 160, 224), bc="periodic", medium="ionised", mean=2e-4,
              sigma_ln=1.0, sources=512, state="lit"),
        # the uniform medium with many sources and the opacity update that
        # follows each of its successive steps (config 3)
        _case("evolve_256", "evolve", (256, 256, 256), sources=4096, state="lit"),
        # fields that live in host memory: transfer and step in one call
        _case("host_256", "host", (256, 256, 256), medium="clumps", sigma_ln=1.5, sources=8192, state="lit"),
        # the benchmark's box: optically thick clumps, 65536 sources (config 4)
        _case("clumps_512", "step", (512, 512, 512), medium="clumps", sigma_ln=1.5, sources=65536, state="lit"),
    ]


def _shape(rng, lo, hi):
    """Extents (3 .. 9) 2^k of a grid with about lo .. hi cells."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    k = max(1, round(math.log2(want ** (1 / 3) / 5.5)))
    while True:
        n = tuple(rng.randint(3, 9) << k for _ in range(3))
        if lo <= n[0] * n[1] * n[2] <= hi:
            return n


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "fp64", "batch", "groups", "evolve", "host"])
    more = {"bc": rng.choice(["closed", "closed", "periodic", "outflow", "ragged"]),
            "theta": rng.choice([1.0, 1.0, 0.5]), "state": rng.choice(["cold", "lit"]),
            "limiter": rng.choice(["paper", "paper", "lp"])}
    more["medium"] = rng.choice(["uniform", "clumps", "ionised"])
    more["sigma_ln"] = 0.0 if more["medium"] == "uniform" else round(rng.uniform(0.5, 1.5), 2)
    more["mean"] = round(10.0 ** rng.uniform(-4, -3), 6)
    if kind == "batch":
        sizes = [16 * rng.randint(1, 4) for _ in range(rng.randint(3, 12))]
        return _drawn("batch", (max(sizes),) * 3, rng, sizes=",".join(map(str, sizes)), persistent=8192)
    if kind == "fp64":
        return _drawn("step", _shape(rng, 4096, 128 ** 3), rng, precision="fp64", **more)
    if kind == "groups":
        more.update(state="lit", limiter="paper")
        return _drawn("groups", _shape(rng, 32768, 128 ** 3), rng, groups=rng.randint(2, 5), **more)
    if kind == "host":
        more["bc"] = rng.choice(["closed", "outflow"])
        return _drawn("host", _shape(rng, 64 ** 3, 256 ** 3), rng, **more)
    n = _shape(rng, 4096, 320 ** 3)
    small = n[0] * n[1] * n[2] <= 8192
    return _drawn(kind, n, rng, persistent=8192 if small and rng.random() < 0.5 else 0, **more)


def _drawn(kind, n, rng, **more):
    c = _case("", kind, n, **more)
    del c["name"]
    c["sources"] = rng.randint(1, 64) if kind == "batch" else max(1, n[0] * n[1] * n[2] // rng.choice([512, 2048, 8192]))
    return c


# ------------------------------------------------------------------- inputs

def _flags(bc):
    """(periodic, dirichlet) flags per axis and per side."""
    if bc == "periodic":
        return (True,) * 3, (False,) * 6
    if bc == "outflow":
        return (False,) * 3, (True,) * 6
    if bc == "ragged":      # y periodic, outflow at the upper x and z faces
        return (False, True, False), (False, True, False, False, False, True)
    return (False,) * 3, (False,) * 6


def _grid(case, n=None):
    n = n or (case["nx"], case["ny"], case["nz"])
    h = case["box_kpc"] * KPC / max(n)
    per, dirich = _flags(case["bc"])
    return synth.Grid(n, (h, h, h), per, dirich, (0.0,) * 6)


def _params(case):
    return synth.Params(limiter=1 if case["limiter"] == "lp" else 0, precision=0 if case["precision"] == "fp64" else 1,
                        theta=case["theta"], L_unit=case["box_kpc"] * KPC, persistent_cells=case["persistent"],
                        sigma=1.0 if case["kind"] == "groups" else SIGMA)


def _wave2(shape, device):
    k2 = 0.0
    for a, n in enumerate(shape):
        f = (torch.fft.rfftfreq if a == 2 else torch.fft.fftfreq)(n, device=device, dtype=torch.float64)
        v = [1, 1, 1]
        v[a] = -1
        k2 = k2 + (2.0 * torch.sin(math.pi * f)).view(v) ** 2
    return k2


def _fields(case, seed, n=None):
    """E^n, n_HI, eta (and n_H) of a case, shaped (nz, ny, nx), on the GPU."""
    grid = _grid(case, n)
    shape = grid.shape
    gen = torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17 * grid.cells)
    f64 = dict(dtype=torch.float64, device="cuda")
    cells, h = grid.cells, grid.h[0]
    k2 = _wave2(shape, "cuda") if case["medium"] != "uniform" or case["state"] == "lit" else None
    ns = min(case["sources"], cells)
    if case["medium"] == "uniform":
        nH = torch.full(shape, case["mean"], **f64)
        at = torch.randint(cells, (ns,), generator=gen, device="cuda")
    else:
        # log-normal density of a Gaussian field with P(k) ~ k^-2, sources at
        # the densest local maxima
        f = torch.fft.rfftn(torch.randn(shape, generator=gen, **f64))
        f *= torch.where(k2 > 0, k2.clamp_min(1e-12) ** -0.5, torch.zeros_like(k2))
        g = torch.fft.irfftn(f, s=shape)
        del f
        s = case["sigma_ln"]
        nH = torch.exp(s * (g - g.mean()) / g.std())
        del g
        nH *= case["mean"] / nH.mean()
        nH.clamp_(1e-3 * case["mean"], 1e3 * case["mean"])
        top = nH.clone()
        for a in range(3):
            for d in (-1, 1):
                top = torch.where(nH >= nH.roll(d, a), top, torch.zeros_like(top))
        at = torch.topk(top.flatten(), ns).indices
        del top
    rates = NDOT * torch.exp(torch.rand(ns, generator=gen, **f64) * 2.0 - 1.0)
    eta = torch.zeros(cells, **f64).index_add_(0, at.sort().values, rates * HNU / grid.volume).view(shape)
    E = torch.full(shape, COLD, **f64)
    lit = None
    if case["state"] == "lit" or case["medium"] == "ionised":
        # the sources' radiation after one diffusive step through the mean
        # medium, weakened where the gas is denser, over a faint background
        w = DT * 0.006 * C * case["box_kpc"] * KPC / h ** 2
        m = 1.0 + DT * C * SIGMA * case["mean"]
        if k2 is None:
            k2 = _wave2(shape, "cuda")
        lit = torch.fft.irfftn(torch.fft.rfftn(DT * eta) / (m + w * k2), s=shape)
        lit *= m / (1.0 + DT * C * SIGMA * nH)
        lit.clamp_min_(1e-9 * float(lit.max()))
        if case["state"] == "lit":
            E = lit
    nHI = nH.clone()
    if case["medium"] == "ionised":
        lo = lit.mean()
        nHI *= (lo / (lo + lit)).clamp_min(1e-6)
    return E.contiguous(), nHI, eta.contiguous(), nH


def _spectrum(case):
    """Grey integrals of a 1e5 K blackbody over the groups, (K, P, H) of HI,
    HeI, HeII and the emissivity share, one row per group."""
    hp, kb, eV = 6.62607015e-27, 1.380649e-16, 1.602176634e-12
    nu1 = HNU / hp
    edges = nu1 * np.array(EDGES[case["groups"]] + (1000.0,))
    species = ((13.6, 6.30e-18, 1.34, 2.99), (24.6, 7.83e-18, 1.66, 2.05), (54.4, 1.58e-18, 1.34, 2.99))

    def chi(nu):
        return nu ** 3 * np.exp(-hp * nu / (kb * 1e5)) / -np.expm1(-hp * nu / (kb * 1e5))

    def quad(f, a, b):
        if b <= a:
            return 0.0
        x = np.linspace(math.log(a), math.log(b), 8193)
        wt = np.ones(8193)
        wt[1:-1:2], wt[2:-1:2] = 4.0, 2.0
        return float((wt * f(np.exp(x)) * np.exp(x)).sum() * (x[1] - x[0]) / 3.0)

    rows = []
    for a, b in zip(edges[:-1], edges[1:]):
        N = quad(chi, a, b)
        row = []
        for kind in range(3):
            for ev, s0, beta, s in species:
                nui = ev * eV / hp

                def f(nu):
                    y = s0 * (beta * (nu / nui) ** -s + (1 - beta) * (nu / nui) ** (-s - 1)) * chi(nu)
                    return y if kind == 0 else y / nu if kind == 1 else y * (1 - nui / nu)
                row.append(quad(f, max(a, nui), b) / N)
        rows.append(row + [N])
    out = np.array(rows)
    out[:, -1] /= out[:, -1].sum()
    return np.ascontiguousarray(out)


def _gas(nHI, nH):
    """Helium densities and the mass density that go with hydrogen."""
    return 0.08 * nHI, 0.08 * (nH - 0.9 * nHI), 1.673e-24 * 1.32 * nH


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    s.stream = torch.cuda.Stream()
    s.params = _params(case)
    if case["kind"] == "batch":
        s.ctx, s.E0, s.E, s.nHI, s.eta = [], [], [], [], []
        for q, n in enumerate(int(v) for v in case["sizes"].split(",")):
            E, nHI, eta, _ = _fields(case, seed * 64 + q, (n, n, n))
            s.ctx.append(fld.fld_create(_grid(case, (n, n, n)), s.params, s.stream))
            for to, v in ((s.E0, E), (s.E, E.clone()), (s.nHI, nHI), (s.eta, eta)):
                to.append(v.flatten())
    elif case["kind"] == "groups":
        g = case["groups"]
        E, nHI, eta, nH = _fields(case, seed)
        s.coef = _spectrum(case)
        s.gas = [v.flatten() for v in _gas(nHI, nH)]
        s.nHI, s.eta0 = nHI.flatten(), eta.flatten()
        s.E0 = [(E * s.coef[q, -1]).flatten() for q in range(g)]
        s.E = [v.clone() for v in s.E0]
        s.kappa = [torch.empty_like(s.nHI) for _ in range(g)]
        s.eta = [torch.empty_like(s.nHI) for _ in range(g)]
        s.rates = [torch.empty_like(s.nHI) for _ in range(4)]
        s.ctx = [fld.fld_create(_grid(case), s.params, s.stream) for _ in range(g)]
    elif case["kind"] == "host":
        E, nHI, eta, _ = _fields(case, seed)
        s.ctx = fld.fld_create(_grid(case), s.params, s.stream)
        # the sources fade and brighten from step to step
        s.E, s.nHI, s.eta = [[_pinned(v) for v in vs] for vs in ((E,), (nHI,), (eta, 0.5 * eta))]
        s.step = 0
    else:
        E, nHI, eta, nH = _fields(case, seed)
        s.ctx = fld.fld_create(_grid(case), s.params, s.stream)
        s.E0, s.E, s.nHI, s.eta = E.flatten(), E.clone().flatten(), nHI.flatten(), eta.flatten()
        if case["kind"] == "evolve":
            s.nH, s.nHI_new = nH.flatten(), torch.empty_like(s.nHI)
    return s


def _pinned(t):
    # numpy keeps the pinned storage alive
    return torch.empty(t.numel(), dtype=torch.float64, pin_memory=True).copy_(t.flatten()).numpy()


def run(s):
    kind = s.case["kind"]
    if kind == "host":
        eta = s.eta[s.step % 2]
        s.step += 1
        fld.fld_step_host(s.ctx, s.E[0], s.nHI[0], eta)
        return {"E": s.E[0]}
    with torch.cuda.stream(s.stream):
        if kind == "batch":
            torch._foreach_copy_(s.E, s.E0)
            fld.fld_step_batched(s.ctx, s.E, s.nHI, s.eta)
            return {"E": s.E}
        if kind == "groups":
            torch._foreach_copy_(s.E, s.E0)
            fld.fld_group_fields(s.coef, s.nHI, s.kappa, s.gas[0], s.gas[1], s.eta0, s.eta)
            fld.fld_step_batched(s.ctx, s.E, s.kappa, s.eta)
            fld.fld_photo_rates(s.coef, s.E, s.nHI, s.gas[0], s.gas[1], s.gas[2], C, *s.rates)
            return {"E": s.E, "rates": s.rates}
        s.E.copy_(s.E0)
        info = fld.fld_step(s.ctx, s.E, s.nHI, s.eta)
        out = {"E": s.E, "emitted": info["emitted"], "absorbed": info["absorbed"]}
        if kind == "evolve":
            fld.fld_opacity_update(s.E, s.nH, s.nHI, s.nHI_new, DT, C, SIGMA, HNU, synth.ALPHA_B, s.stream)
            out["nHI"] = s.nHI_new
        return out


def work(case):
    # bytes: E, n_HI and eta read and E written once (FP64); a multigroup
    # step reads the densities and the emissivity, every group's E, and
    # writes every group's E and the four rates; the opacity update reads n_H
    # and writes n_HI.  flops: the assembly (about 60 per cell), and ten
    # preconditioned CG iterations (one symmetric red/black V-cycle over all
    # levels, 8/7 of about 60 per cell, the operator and the vectors, 25)
    cells = sum(int(v) ** 3 for v in case["sizes"].split(",")) if case["kind"] == "batch" else \
        case["nx"] * case["ny"] * case["nz"]
    words, solves = 4, 1
    if case["kind"] == "groups":
        words, solves = 5 + 2 * case["groups"] + 4, case["groups"]
    elif case["kind"] == "evolve":
        words = 6
    return {"bytes": 8.0 * words * cells, "flops": solves * cells * (60.0 + 10 * (60 * 8 / 7 + 25))}


# -------------------------------------------------- the same step in 64 bits

def _diffusion(case, Ef, kf, dE_h, Dmax, Rmin):
    R = torch.where(Ef > 0, dE_h / Ef.clamp_min(1e-300), torch.zeros_like(Ef)).clamp_min(Rmin)
    if case["limiter"] == "lp":
        x = R / kf
        lam = torch.where(x < 1e-2, 1 / 3 - x * x / 45 + 2 * x ** 4 / 945,
                          (1 / torch.tanh(x.clamp_min(1e-2)) - 1 / x.clamp_min(1e-2)) / x.clamp_min(1e-2))
        D = C * lam / kf
    else:
        D = C / torch.sqrt(9 * kf * kf + R * R)
    return D.clamp_max(Dmax)


def _solve64(case, E, kappa, eta):
    """E^{n+1} of one step by conjugate gradients with the diagonal as
    preconditioner, to rounding."""
    grid, th = _grid(case, tuple(reversed(E.shape))), case["theta"]
    per, dirich = _flags(case["bc"])
    h, L = grid.h[0], case["box_kpc"] * KPC
    Dmax, Rmin = 0.006 * C * L, 1e-20 / L
    m, b = 1.0 + th * DT * C * kappa, DT * eta - DT * C * kappa * E
    faces = []
    for a in range(3):
        ax, n = 2 - a, grid.n[a]
        pairs = [(lambda t, ax=ax, n=n: t.narrow(ax, 0, n - 1), lambda t, ax=ax, n=n: t.narrow(ax, 1, n - 1))]
        if per[a]:
            pairs.append((lambda t, ax=ax, n=n: t.narrow(ax, n - 1, 1), lambda t, ax=ax: t.narrow(ax, 0, 1)))
        for p, q in pairs:
            kp, kq = p(kappa), q(kappa)
            w = DT / h ** 2 * _diffusion(case, 0.5 * (p(E) + q(E)), 2 * kp * kq / (kp + kq), (q(E) - p(E)).abs() / h,
                                         Dmax, Rmin)
            f = w * (q(E) - p(E))
            p(b).add_(f)
            q(b).sub_(f)
            faces.append((p, q, th * w))
        for side in (0, 1):
            if dirich[2 * a + side]:
                at = (lambda t, ax=ax, i=(n - 1) * side: t.narrow(ax, i, 1))
                w = DT / (h * h / 2) * _diffusion(case, 0.5 * at(E), at(kappa), at(E) / (h / 2), Dmax, Rmin)
                at(m).add_(th * w)
                at(b).sub_(w * at(E))
    diag = m.clone()
    for p, q, w in faces:
        p(diag).add_(w)
        q(diag).add_(w)

    def apply(u):
        y = m * u
        for p, q, w in faces:
            f = w * (q(u) - p(u))
            p(y).sub_(f)
            q(y).add_(f)
        return y

    x, r = torch.zeros_like(b), b.clone()
    z = r / diag
    p_, rz, goal = z.clone(), torch.vdot(r.flatten(), z.flatten()), 1e-13 * float(b.norm())
    for it in range(20000):
        q_ = apply(p_)
        alpha = rz / torch.vdot(p_.flatten(), q_.flatten())
        x += alpha * p_
        r -= alpha * q_
        if it % 20 == 19 and float(r.norm()) <= goal:
            break
        z = r / diag
        new = torch.vdot(r.flatten(), z.flatten())
        p_ = torch.addcmul(z, p_, new / rz)
        rz = new
    return (E + x).clamp_min_(0.0), x


def exact(case, seed):
    if case["kind"] == "batch":
        out = []
        for q, n in enumerate(int(v) for v in case["sizes"].split(",")):
            E, nHI, eta, _ = _fields(case, seed * 64 + q, (n, n, n))
            out.append(_solve64(case, E, SIGMA * nHI, eta)[0].flatten())
        return {"E": out}
    E, nHI, eta, nH = _fields(case, seed)
    if case["kind"] == "groups":
        coef = _spectrum(case)
        he1, he2, rho = _gas(nHI, nH)
        gas = (nHI, he1, he2)
        Es = [_solve64(case, E * k[-1], sum(k[i] * gas[i] for i in range(3)), k[-1] * eta)[0] for k in coef]
        hp = 6.62607015e-27
        rates = [sum(C / hp * k[3 + i] * e for k, e in zip(coef, Es)) for i in range(3)]
        heat = sum(C * e * sum(k[6 + i] * gas[i] for i in range(3)) for k, e in zip(coef, Es)) / rho
        return {"E": [e.flatten() for e in Es], "rates": [r.flatten() for r in rates + [heat]]}
    new, dE = _solve64(case, E, SIGMA * nHI, eta)
    if case["kind"] == "host":
        return {"E": new.flatten().cpu()}
    scale = _grid(case).volume / HNU
    out = {"E": new.flatten(), "emitted": float(DT * eta.sum()) * scale,
           "absorbed": float((DT * C * SIGMA * nHI * (E + case["theta"] * dE)).sum()) * scale}
    if case["kind"] == "evolve":
        x = nHI / nH
        x = (x + DT * synth.ALPHA_B * nH * (1 - x) ** 2) / (1 + DT * C * SIGMA * new / HNU)
        out["nHI"] = (x.clamp(1e-12, 1.0) * nH).flatten()
    return out
