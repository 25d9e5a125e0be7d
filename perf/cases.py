"""Performance cases: the work that a user of this solver has it do.

Each case is one call (or one time step's calls) through the public binding
(``paper_1110_1379_gb300.frmg``), on seeded synthetic inputs of the kinds the
tests and ``bench.py`` use: lognormal density fields of spectrum k^-1.5,
Zel'dovich-displaced particles, nested refinement patches and irregular masked
regions over the densest cells.  The rms residual is driven to 1e-11 (f(R);
production runs of the method ask for 1e-8 to 1e-12) or 1e-10 (Poisson and
symmetron), so that a converged solution is fixed to about ten digits whatever
path led to it.

``exact`` recomputes each case in plain torch FP64: Newton's method with a
Jacobi-preconditioned BiCGStab solver for the nonlinear equations, an FFT for
the Poisson equation, index_add_ for the particle assignment.
"""
from __future__ import annotations

import math

import torch

from paper_1110_1379_gb300 import frmg

OMEGA_M = 0.24
TOL, TOL_POISSON, TOL_SYMMETRON = 1e-11, 1e-10, 1e-10
F64 = torch.float64

_ctx = None


def _context():
    """The program's one solver context (it keeps the device workspace)."""
    global _ctx
    if _ctx is None:
        _ctx = frmg.Context(0)
    return _ctx


# ---------------------------------------------------------------------------
# cases
def listed():
    return [
        # smallest call: the 32^3 FP64 solve (config 1), launch latency
        dict(name="fp64_32", kind="solve", nx=32, ny=32, nz=32, cell=2.0, a=1.0, fr0=1e-5,
             sigma=1.0, prec="fp64", start="zero", host=False),
        # the plain FP64 method at the size of a test simulation (config 2)
        dict(name="fp64_128", kind="solve", nx=128, ny=128, nz=128, cell=1.0, a=0.5, fr0=1e-5,
             sigma=1.5, prec="fp64", start="zero", host=False),
        # small mixed-precision solve with library defaults
        dict(name="mixed_64", kind="solve", nx=64, ny=64, nz=64, cell=1.0, a=1.0, fr0=1e-5,
             sigma=1.5, prec="mixed", start="zero", host=False),
        # ragged box, strongly screened field, restarted from a guess
        dict(name="mixed_ragged_f6", kind="solve", nx=320, ny=192, nz=224, cell=0.5, a=1.0,
             fr0=1e-6, sigma=1.5, prec="mixed", start="linear", host=False),
        # host arrays: page-locked density in, page-locked solution out
        dict(name="mixed_256_host", kind="solve", nx=256, ny=256, nz=256, cell=0.5, a=1.0,
             fr0=1e-5, sigma=2.0, prec="mixed", start="zero", host=True),
        # the headline's grid: 512^3 with the setting the autotuner picks for it
        dict(name="mixed_512_tuned", kind="solve", nx=512, ny=512, nz=512, cell=0.5, a=1.0,
             fr0=1e-5, sigma=1.5, prec="mixed", start="zero", host=False, pre=1, post=1,
             relax=1.15, fmg=1, tiling=1, smooth_tile=16),
        # one time step of a particle-mesh run: TSC density, f(R) solve,
        # modified Poisson solve, forces at the particles (config 2's sizes)
        dict(name="step_128", kind="step", nx=128, ny=128, nz=128, cell=1.0, a=1.0, fr0=1e-5,
             np=128 ** 3, scheme="tsc"),
        # many independent fields of uneven size in one call (config 5's recipe)
        dict(name="batch_48", kind="batch", nfields=48, sizes="32 48 64 96 128", pick=5000),
        # domain grid and two nested refinement levels (config 4's sizes)
        dict(name="levels_256", kind="levels", n=256, count1=16, count2=12, fr0=1e-5, sigma=2.0),
        # general mask scheme: an irregular region in a 256^3 box
        dict(name="masked_256", kind="masked", n=256, spheres=16, rmin=14.0, rmax=30.0, fr0=1e-5,
             sigma=0.9, prec="mixed", pre=2, post=2, relax=1.0),
        # modified Poisson solve on a large grid
        dict(name="poisson_512", kind="poisson", nx=512, ny=512, nz=512, cell=0.5, a=1.0,
             fr0=1e-5, sigma=2.0, pre=1, post=1, relax=1.2),
        # the second scalar-field model on the headline's grid
        dict(name="symmetron_512", kind="symmetron", nx=512, ny=512, nz=512, cell=0.5, a=1.0,
             a_ssb=0.5, lambda0=1.0, sigma=2.0, pre=2, post=2, relax=1.15),
    ]


def _sides(rng, lo, hi, top=14):
    """Three sides within a factor of two of one another, 4 to `top` times a
    common power of two (so that the coarsest grid of the hierarchy is small):
    cubes of 48 or 256 cells, and boxes such as 80 x 112 x 96."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    p = 2 ** max(2, math.ceil(math.log2(v / top)))
    m = min(hi // p, max(-(-lo // p), round(v / p))) // 2 * 2
    s = [m * p] + [p * rng.randrange(max(4, m // 2 + m // 2 % 2), m + 1, 2) for _ in range(2)]
    rng.shuffle(s)
    return dict(zip(("nx", "ny", "nz"), s))


def draw(rng):
    kind = rng.choice(["solve"] * 5 + ["fp64", "step", "batch", "levels", "masked", "poisson",
                                       "symmetron"])
    fr0 = rng.choice([1e-6, 1e-5, 1e-4])
    if kind == "solve":
        c = dict(kind="solve", **_sides(rng, 32, 448), cell=rng.choice([0.5, 1.0, 2.0]),
                 a=round(rng.uniform(0.4, 1.0), 3), fr0=fr0, sigma=round(rng.uniform(0.7, 1.8), 2),
                 prec="mixed", start=rng.choice(["zero", "linear"]), host=rng.random() < 0.2)
        if fr0 == 1e-4:
            c["cell"] = 2.0
        if rng.random() < 0.4:  # settings the autotuner tries
            c.update(pre=rng.choice([1, 2]), post=rng.choice([1, 2]),
                     relax=rng.choice([1.0, 1.15]), tiling=rng.choice([0, 1]),
                     smooth_tile=rng.choice([8, 16]))
        return c
    if kind == "fp64":
        return dict(kind="solve", **_sides(rng, 32, 112), cell=rng.choice([1.0, 2.0]),
                    a=round(rng.uniform(0.4, 1.0), 3), fr0=fr0,
                    sigma=round(rng.uniform(0.7, 1.8), 2), prec="fp64",
                    start=rng.choice(["zero", "linear"]), host=False)
    if kind == "step":
        n = rng.choice([48, 64, 96, 128, 192])
        s = dict(nx=n, ny=n, nz=n)
        return dict(kind="step", **s, cell=rng.choice([1.0, 2.0]),
                    a=round(rng.uniform(0.5, 1.0), 3), fr0=rng.choice([1e-6, 1e-5]),
                    np=int(n ** 3 * rng.uniform(0.5, 2.0)) + rng.randrange(7),
                    scheme=rng.choice(["cic", "tsc"]))
    if kind == "batch":
        return dict(kind="batch", nfields=rng.randrange(3, 41), sizes="32 48 64 96 128",
                    pick=rng.randrange(10000))
    if kind == "levels":
        return dict(kind="levels", n=rng.choice([128, 160, 192, 224]), count1=rng.randrange(3, 13),
                    count2=rng.randrange(0, 9), fr0=rng.choice([1e-6, 1e-5]),
                    sigma=round(rng.uniform(1.0, 2.0), 2))
    if kind == "masked":
        n = rng.choice([96, 128, 160, 192])
        return dict(kind="masked", n=n, spheres=rng.randrange(4, 25),
                    rmin=round(n / rng.uniform(14, 20), 1), rmax=round(n / rng.uniform(6.5, 10), 1),
                    fr0=rng.choice([1e-6, 1e-5]), sigma=round(rng.uniform(0.7, 1.1), 2),
                    prec=rng.choice(["mixed", "mixed", "fp64"]), pre=2, post=2, relax=1.0)
    if kind == "poisson":
        return dict(kind="poisson", **_sides(rng, 64, 448, 8), cell=rng.choice([0.5, 1.0]), a=1.0,
                    fr0=1e-5, sigma=round(rng.uniform(1.0, 2.0), 2), pre=rng.choice([1, 2]),
                    post=rng.choice([1, 2]), relax=rng.choice([1.0, 1.2]))
    return dict(kind="symmetron", **_sides(rng, 48, 384), cell=rng.choice([0.5, 1.0]),
                a=round(rng.uniform(0.7, 1.0), 3), a_ssb=0.5, lambda0=1.0,
                sigma=round(rng.uniform(1.0, 2.0), 2), pre=2, post=2, relax=1.0)


# ---------------------------------------------------------------------------
# inputs
def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _phys(case):
    return dict(box=case["cell"] * case["nx"], a=case["a"], omega_m=OMEGA_M, fr0=case["fr0"])


def _options(case):
    return {k: case[k] for k in ("pre", "post", "relax", "fmg", "tiling", "smooth_tile")
            if k in case}


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _wavenumbers(shape):
    """k in units of the inverse x cell (cubic cells) on the rFFT grid: kz, ky, kx."""
    n2, n1, n0 = shape
    kz = torch.fft.fftfreq(n2, dtype=F64, device="cuda")[:, None, None] * (2 * math.pi)
    ky = torch.fft.fftfreq(n1, dtype=F64, device="cuda")[None, :, None] * (2 * math.pi)
    kx = torch.fft.rfftfreq(n0, dtype=F64, device="cuda")[None, None, :] * (2 * math.pi)
    return kz, ky, kx


def _gaussian(shape, gen, slope):
    """Unit-variance Gaussian field of spectrum |k|^slope without its mean."""
    w = torch.fft.rfftn(torch.randn(shape, generator=gen, dtype=F64, device="cuda"))
    kz, ky, kx = _wavenumbers(shape)
    k2 = kz * kz + ky * ky + kx * kx
    k2[0, 0, 0] = 1.0
    w *= k2.pow_(slope / 4.0)
    w[0, 0, 0] = 0.0
    g = torch.fft.irfftn(w, s=shape)
    return g.div_(g.std())


def _density(shape, seed, sigma):
    """Lognormal density of mean 1."""
    r = _gaussian(shape, _generator(seed), -1.5).mul_(sigma).sub_(0.5 * sigma * sigma).exp_()
    return r.div_(r.mean())


def _positions(case, seed):
    """Particles on a jittered lattice displaced by a Zel'dovich field to a
    few cells rms, in box units [0, 1)."""
    shape, np_ = _shape(case), case["np"]
    gen = _generator(seed)
    gk = torch.fft.rfftn(_gaussian(shape, gen, -2.5))
    kz, ky, kx = _wavenumbers(shape)
    k2 = kz * kz + ky * ky + kx * kx
    k2[0, 0, 0] = 1.0
    cells = shape[0] * shape[1] * shape[2]
    at = (torch.arange(np_, device="cuda", dtype=F64) * (cells / np_)).long().clamp_(max=cells - 1)
    pos = torch.empty((np_, 3), dtype=F64, device="cuda")
    norm = None
    for d, (k, n) in enumerate(zip((kx, ky, kz), shape[::-1])):
        s = torch.fft.irfftn(1j * k * gk / k2, s=shape).reshape(-1)
        norm = 3.0 / float(s.std()) if norm is None else norm
        lat = (at if d == 0 else at // shape[2] if d == 1 else at // (shape[1] * shape[2])) % n
        jitter = torch.rand(np_, generator=gen, dtype=F64, device="cuda")
        pos[:, d] = ((lat + jitter + norm * s[at]) / n).remainder_(1.0)
    pos[pos >= 1.0] = 0.0
    return pos


def _constants(box, n0, a, omega_m, fr0, h=None):
    """(alpha, beta, gamma) of the discrete equation at cell size h (box units)."""
    h = 1.0 / n0 if h is None else h
    ol, ct = 1.0 - omega_m, 299792.458 / (100.0 * box)
    k, k1 = a ** -3 + 4.0 * ol / omega_m, 1.0 + 4.0 * ol / omega_m
    fbar = a * a * fr0 * (k1 / k) ** 2
    return ct * ct * fbar / (h * h), omega_m * a ** 4 * k, omega_m * a


def _linear_u(rho, phys, h=None):
    """Linear-theory field of the density: the guess of a restarted run, and
    the outside values of an irregular region."""
    alpha, beta, gamma = _constants(n0=rho.shape[2], h=h, **phys)
    lap = sum(2.0 * torch.cos(k) - 2.0 for k in _wavenumbers(rho.shape))
    w = torch.fft.rfftn(rho - 1.0) * (gamma / (alpha * lap - 0.5 * beta))
    return torch.fft.irfftn(w, s=rho.shape).clamp_(-2.0, 2.0).contiguous()


def _dense_blocks(rho, block, count, margin=0):
    """(z, y, x) corners of the `count` densest blocks (non-overlapping, at
    least `margin` cells inside the box)."""
    r = rho[margin:rho.shape[0] - margin, margin:rho.shape[1] - margin,
            margin:rho.shape[2] - margin]
    p = torch.nn.functional.avg_pool3d(r[None, None], block)[0, 0]
    best = torch.topk(p.reshape(-1), min(count, p.numel())).indices.cpu().tolist()
    d1, d0 = p.shape[1], p.shape[2]
    return [(margin + block * (b // (d1 * d0)), margin + block * (b // d0 % d1),
             margin + block * (b % d0)) for b in best]


def _children(block, gen, sigma=0.5):
    """Density of the 2x2x2 children of every cell: seeded lognormal modulation
    of mean 1 over the children of a cell."""
    s = block.shape
    m = torch.randn((s[0], 2, s[1], 2, s[2], 2), generator=gen, dtype=F64, device="cuda")
    m = m.mul_(sigma).exp_()
    m = m / m.mean(dim=(1, 3, 5), keepdim=True) * block[:, None, :, None, :, None]
    return m.reshape(2 * s[0], 2 * s[1], 2 * s[2]).contiguous()


def _patches(case, rho, seed):
    """Patches of 32 to 64 cells over the densest blocks of the domain, one
    level-2 patch of 32 or 48 cells inside each of the first `count2`."""
    gen, out = _generator(seed + 1), []

    def add(parent, src, corner, room, n):
        o = [c + (room - n // 2) // 2 for c in corner]
        b = src[tuple(slice(v, v + n // 2) for v in o)]
        out.append(dict(parent=parent, origin=(o[2], o[1], o[0]), density=_children(b, gen),
                        u=torch.empty((n, n, n), dtype=F64, device="cuda")))

    for t, corner in enumerate(_dense_blocks(rho, 32, case["count1"])):
        add(-1, rho, corner, 32, (64, 48, 32)[t % 3])
    for t in range(min(case["count2"], len(out))):
        src = out[t]["density"]
        n = src.shape[0]
        add(t, src, (0, 0, 0), n, 48 if n >= 48 and t % 2 else 32)
    return out


def _mask(case, rho, seed):
    """+1 inside a union of spheres around the densest blocks, -1 elsewhere."""
    n, gen = case["n"], torch.Generator().manual_seed(seed + 2)
    edge = int(math.ceil(case["rmax"])) + n // 16
    block = max(8, n // 32)
    ax = torch.arange(n, dtype=F64, device="cuda")
    m = torch.full((n, n, n), -1.0, dtype=F64, device="cuda")
    for z, y, x in _dense_blocks(rho, block, case["spheres"], margin=edge):
        r = case["rmin"] + (case["rmax"] - case["rmin"]) * float(torch.rand(1, generator=gen))
        c = 0.5 * block
        d2 = (((ax - z - c) ** 2)[:, None, None] + ((ax - y - c) ** 2)[None, :, None] +
              ((ax - x - c) ** 2)[None, None, :])
        m[d2 < r * r] = 1.0
    return m


def _specs(case):
    """The fields of a batch: size, cell 1 Mpc/h, |f_R0|, a and sigma of each
    (config 5's ranges), fixed by the case."""
    import random
    r = random.Random(case["pick"])
    sizes = [int(v) for v in case["sizes"].split()]
    return [dict(n=r.choice(sizes), fr0=r.choice([1e-4, 1e-5, 1e-6]), a=r.uniform(0.3, 1.0),
                 sigma=r.uniform(0.5, 2.0)) for _ in range(case["nfields"])]


def _masked_phys(case):
    return dict(box=0.5 * case["n"], a=1.0, omega_m=OMEGA_M, fr0=case["fr0"])


def _levels_phys(case):
    return dict(box=float(case["n"]), a=1.0, omega_m=OMEGA_M, fr0=case["fr0"])


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    s = dict(case=case, ctx=ctx)
    if kind == "step":
        s["pos"] = _positions(case, seed)
        s["rho"], s["u"], s["phi"] = (torch.empty(_shape(case), dtype=F64, device="cuda")
                                      for _ in range(3))
        s["force"] = torch.empty((case["np"], 3), dtype=F64, device="cuda")
    elif kind == "batch":
        s["rho"] = [_density((f["n"],) * 3, 1000 * seed + i, f["sigma"])
                    for i, f in enumerate(_specs(case))]
        s["u"] = [torch.empty_like(r) for r in s["rho"]]
    elif kind == "levels":
        s["rho"] = _density((case["n"],) * 3, seed, case["sigma"])
        s["u"] = torch.empty_like(s["rho"])
        s["patches"] = _patches(case, s["rho"], seed)
    elif kind == "masked":
        s["rho"] = _density((case["n"],) * 3, seed, case["sigma"])
        s["mask"] = _mask(case, s["rho"], seed)
        s["u0"] = _linear_u(s["rho"], _masked_phys(case), 1.0 / (2 * case["n"]))
        s["u"] = torch.empty_like(s["rho"])
    else:
        s["rho"] = _density(_shape(case), seed, case["sigma"])
        s["u"] = torch.empty_like(s["rho"])
        if kind == "poisson":
            s["u"] = _linear_u(s["rho"], _phys(case))
            s["phi"] = torch.empty_like(s["rho"])
        elif case.get("start") == "linear":
            s["u0"] = _linear_u(s["rho"], _phys(case))
        if case.get("host"):
            for k in ("rho", "u", "u0"):
                if k in s:
                    s[k] = s[k].cpu().pin_memory()
    return s


# ---------------------------------------------------------------------------
# one pass
def _solve(s, rho, u, **opts):
    if "u0" in s:
        u.copy_(s["u0"])
    st, _ = s["ctx"].solve(rho, u, tol=TOL, initial_guess=int("u0" in s), **_phys(s["case"]),
                           **opts)
    return st


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "solve":
        return {"u": s["u"], "status": _solve(s, s["rho"], s["u"], prec=case["prec"],
                                              **_options(case))}
    if kind == "step":
        (ctx.tsc if case["scheme"] == "tsc" else ctx.cic)(s["pos"], s["rho"])
        st = _solve(s, s["rho"], s["u"], prec="mixed")
        s["phi"].zero_()
        st2, _, _ = ctx.poisson(s["rho"], s["u"], s["phi"], tol=TOL_POISSON, **_phys(case))
        ctx.forces(s["phi"], s["pos"], s["force"], scheme=case["scheme"])
        return {"rho": s["rho"], "u": s["u"], "phi": s["phi"], "force": s["force"],
                "status": [st, st2]}
    if kind == "batch":
        f = _specs(case)
        st, _ = ctx.solve_batch(s["rho"], s["u"], boxes=[float(v["n"]) for v in f],
                                avals=[v["a"] for v in f], fr0s=[v["fr0"] for v in f],
                                omega_m=OMEGA_M, tol=TOL, prec="mixed", initial_guess=0)
        return {"u": s["u"], "status": st}
    if kind == "levels":
        st, _ = ctx.solve_levels(s["rho"], s["u"], s["patches"], tol=TOL, prec="mixed",
                                 initial_guess=0, **_levels_phys(case))
        return {"u": s["u"], "patches": [p["u"] for p in s["patches"]], "status": st}
    if kind == "masked":
        s["u"].copy_(s["u0"])
        st, _ = ctx.solve_masked(s["rho"], s["mask"], s["u"], h=1.0 / (2 * case["n"]), tol=TOL,
                                 prec=case["prec"], **_options(case), **_masked_phys(case))
        return {"u": s["u"], "status": st}
    if kind == "poisson":
        s["phi"].zero_()
        st, _, mean = ctx.poisson(s["rho"], s["u"], s["phi"], tol=TOL_POISSON, **_options(case),
                                  **_phys(case))
        return {"phi": s["phi"], "mean": mean, "status": st}
    st, _ = ctx.symmetron(s["rho"], s["u"], box=case["cell"] * case["nx"], a=case["a"],
                          a_ssb=case["a_ssb"], lambda0=case["lambda0"], tol=TOL_SYMMETRON,
                          prec="mixed", initial_guess=0, **_options(case))
    return {"chi": s["u"], "status": st}


def work(case):
    """Inputs read once, outputs written once; one evaluation of the discrete
    equation (about 40 operations a cell) per grid."""
    kind = case["kind"]
    if kind == "batch":
        cells = sum(f["n"] ** 3 for f in _specs(case))
    elif kind == "levels":
        n1 = [(64, 48, 32)[t % 3] for t in range(case["count1"])]
        n2 = [48 if n1[t] >= 48 and t % 2 else 32 for t in range(min(case["count2"], len(n1)))]
        cells = case["n"] ** 3 + sum(v ** 3 for v in n1 + n2)
    elif kind == "masked":
        cells = case["n"] ** 3
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
    arrays = {"masked": 4, "poisson": 3}.get(kind, 2) + (case.get("start") == "linear")
    if kind == "step":  # positions in, density, u, Phi and forces out
        return {"bytes": 24 * cells + 48 * case["np"], "flops": 80 * cells + 200 * case["np"]}
    return {"bytes": 8 * arrays * cells, "flops": 40 * cells}


# ---------------------------------------------------------------------------
# plain FP64 solutions
def _newton(u, linearise, active=None, tol=3e-13):
    """Newton's method on F(u) = 0; linearise(u) -> (F, J's diagonal, matvec).
    Each step solves J x = -F by BiCGStab on the diagonally scaled system; the
    step is limited to 1 per cell."""
    def dot(a, b):
        return float(torch.dot(a.reshape(-1), b.reshape(-1)))

    for _ in range(40):
        F, diag, mul = linearise(u)
        inv = diag.reciprocal_()
        if active is not None:
            inv = torch.where(active, inv, 0.0)
        r = F.neg_().mul_(inv)
        norm0 = math.sqrt(dot(r, r))
        if norm0 <= 1e-15 * math.sqrt(r.numel()):
            break
        x, p, v, rh = torch.zeros_like(r), torch.zeros_like(r), torch.zeros_like(r), r.clone()
        rho = al = om = 1.0
        stop = max(1e-10 * norm0, 1e-2 * tol * math.sqrt(r.numel())) if norm0 < 1e-2 * math.sqrt(
            r.numel()) else 1e-3 * norm0
        for _ in range(2000):
            rho1 = dot(rh, r)
            if rho1 == 0.0 or om == 0.0:
                break
            p = p.sub_(v, alpha=om).mul_((rho1 / rho) * (al / om)).add_(r)
            rho = rho1
            v = mul(p).mul_(inv)
            al = rho / dot(rh, v)
            r = r.sub_(v, alpha=al)
            x.add_(p, alpha=al)
            t = mul(r).mul_(inv)
            tt = dot(t, t)
            om = dot(t, r) / tt if tt else 0.0
            x.add_(r, alpha=om)
            r = r.sub_(t, alpha=om)
            if dot(r, r) <= stop * stop:
                break
        big = float(x.abs().max())
        u = u + x.clamp_(-1.0, 1.0)
        if big < tol:
            break
    return u


_FACES = [(ax, s) for ax in (0, 1, 2) for s in (1, -1)]


def _exact_fr(rho, u0, alpha, beta, gamma, active=None):
    """Solution of the discrete f(R) equation; with `active`, on those cells
    only, ghosts across its surface being u0_i + u0_j - u_i."""
    near = None if active is None else [active.roll(s, ax) for ax, s in _FACES]
    src = gamma * (rho - 1.0)

    def linearise(u):
        B = torch.exp(u)
        e = torch.exp(-0.5 * u)
        F = beta * (e - 1.0) - src
        diag = e.mul_(-0.5 * beta)
        coef = []
        for f, (ax, s) in enumerate(_FACES):
            uj, Bj = u.roll(s, ax), B.roll(s, ax)
            if near is not None:
                ug = u0 + u0.roll(s, ax) - u
                uj, Bj = torch.where(near[f], uj, ug), torch.where(near[f], Bj, torch.exp(ug))
            w, sB = uj - u, B + Bj
            F.add_(sB * w, alpha=0.5 * alpha)
            d = B * w - sB
            c = Bj * w + sB
            if near is not None:
                d = torch.where(near[f], d, (B - Bj) * w - 2.0 * sB)
                c = torch.where(near[f], c, 0.0)
            diag.add_(d, alpha=0.5 * alpha)
            coef.append(c.mul_(0.5 * alpha))
        if active is not None:
            F = torch.where(active, F, 0.0)

        d0 = diag.clone()

        def mul(v):
            y = d0 * v
            for (ax, s), c in zip(_FACES, coef):
                y.addcmul_(c, v.roll(s, ax))
            return y
        return F, diag, mul
    return _newton(u0.clone(), linearise, active)


def _exact_symmetron(rho, case):
    A = 2.0 * case["lambda0"] ** 2 / (case["a"] * case["cell"]) ** 2
    s = (case["a_ssb"] / case["a"]) ** 3
    m = s * rho - 1.0

    def linearise(u):
        def lap(v):
            y = v * -6.0
            for ax, st in _FACES:
                y.add_(v.roll(st, ax))
            return y.mul_(A)
        d = m + 3.0 * u * u
        return lap(u) - (m + u * u) * u, -6.0 * A - d, lambda v: lap(v).sub_(d * v)
    return _newton(torch.full_like(rho, math.sqrt(1.0 - s)), linearise)


def _interpolate(parent, origin, n):
    """Trilinear (3/4, 1/4 per axis) values of the fine cells -1..n of a patch
    whose lower corner is the parent cell `origin` (x, y, z); wraps."""
    v = parent
    for ax, o in zip((0, 1, 2), origin[::-1]):
        at = torch.arange(o - 2, o + n // 2 + 2, device="cuda") % v.shape[ax]
        v = v.index_select(ax, at)
        m = v.shape[ax]
        c = v.narrow(ax, 1, m - 2)
        lo = 0.75 * c + 0.25 * v.narrow(ax, 0, m - 2)
        hi = 0.75 * c + 0.25 * v.narrow(ax, 2, m - 2)
        v = torch.stack((lo, hi), ax + 1).flatten(ax, ax + 1).narrow(ax, 1, n + 2)
    return v


def _exact_poisson(rho, u, phys):
    _, beta, gamma = _constants(n0=rho.shape[2], **phys)
    src = 2.0 * gamma * (rho - 1.0) - 0.5 * beta * (torch.exp(-0.5 * u) - 1.0)
    mean = src.mean()
    lap = sum(2.0 * torch.cos(k) - 2.0 for k in _wavenumbers(rho.shape)) * rho.shape[2] ** 2
    lap[0, 0, 0] = 1.0
    w = torch.fft.rfftn(src - mean) / lap
    w[0, 0, 0] = 0.0
    return torch.fft.irfftn(w, s=rho.shape), float(mean)


def _weights(pos, shape, scheme):
    """[(cell index, weight)] of every particle, one entry per stencil cell."""
    per = []
    for d, n in enumerate(shape[::-1]):
        g = pos[:, d] * n - 0.5
        if scheme == "cic":
            i = torch.floor(g)
            f = g - i
            w = [1.0 - f, f]
        else:
            i = torch.floor(g + 0.5)
            f = g - i
            w = [0.5 * (0.5 - f) ** 2, 0.75 - f * f, 0.5 * (0.5 + f) ** 2]
            i = i - 1
        i = i.long()
        per.append([((i + t) % n, w[t]) for t in range(len(w))])
    return [((kz * shape[1] + ky) * shape[2] + kx, wx * wy * wz)
            for kz, wz in per[2] for ky, wy in per[1] for kx, wx in per[0]]


def _exact_step(case, s):
    shape, phys = _shape(case), _phys(case)
    w = _weights(s["pos"], shape, case["scheme"])
    rho = torch.zeros(shape, dtype=F64, device="cuda")
    for c, v in w:
        rho.view(-1).index_add_(0, c, v)
    rho *= rho.numel() / case["np"]
    u = _exact_fr(rho, torch.zeros_like(rho), *_constants(n0=case["nx"], **phys))
    phi, _ = _exact_poisson(rho, u, phys)
    force = torch.zeros_like(s["force"])
    for d in range(3):  # box units: every side has length 1
        g = (phi.roll(1, 2 - d) - phi.roll(-1, 2 - d)) * (0.5 * shape[2 - d])
        for c, v in w:
            force[:, d] += v * g.view(-1)[c]
    return {"rho": rho, "u": u, "phi": phi, "force": force, "status": [0, 0]}


def exact(case, seed):
    s, kind = prepare(case, seed), case["kind"]
    if kind == "solve":
        rho = s["rho"].cuda()
        u0 = s["u0"].cuda() if "u0" in s else torch.zeros_like(rho)
        return {"u": _exact_fr(rho, u0, *_constants(n0=case["nx"], **_phys(case))), "status": 0}
    if kind == "step":
        return _exact_step(case, s)
    if kind == "batch":
        return {"u": [_exact_fr(r, torch.zeros_like(r), *_constants(
            float(f["n"]), f["n"], f["a"], OMEGA_M, f["fr0"]))
            for r, f in zip(s["rho"], _specs(case))], "status": 0}
    if kind == "levels":
        phys, n = _levels_phys(case), case["n"]
        u = _exact_fr(s["rho"], torch.zeros_like(s["rho"]), *_constants(n0=n, **phys))
        done = []
        for p in s["patches"]:
            m, depth = p["density"].shape[0], 1 if p["parent"] < 0 else 2
            u0 = _interpolate(u if depth == 1 else done[p["parent"]], p["origin"], m)
            act = torch.zeros(u0.shape, dtype=torch.bool, device="cuda")
            act[1:-1, 1:-1, 1:-1] = True
            rho = torch.nn.functional.pad(p["density"], (1,) * 6, value=1.0)
            v = _exact_fr(rho, u0, *_constants(n0=n, h=1.0 / (n << depth), **phys), active=act)
            done.append(v[1:-1, 1:-1, 1:-1].contiguous())
        return {"u": u, "patches": done, "status": 0}
    if kind == "masked":
        k = _constants(n0=case["n"], h=1.0 / (2 * case["n"]), **_masked_phys(case))
        return {"u": _exact_fr(s["rho"], s["u0"], *k, active=s["mask"] > 0), "status": 0}
    if kind == "poisson":
        phi, mean = _exact_poisson(s["rho"], s["u"], _phys(case))
        return {"phi": phi, "mean": mean, "status": 0}
    return {"chi": _exact_symmetron(s["rho"], case), "status": 0}
