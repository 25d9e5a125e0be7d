"""The one-cluster tail of the V-cycle (frmg_tail.cuh) at the edges of its
layout: grids that are all tail, levels kept in one block, planes that do not
divide evenly over the cluster, coarsest grids of more than one warp's cells,
and sets of more grids than run at once."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from oracle import oracle as O  # noqa: E402
from paper_1110_1379_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu

# n2 x n1 x n0: one level (8x6x10), coarsest grids of 48 to 2744 cells, 12, 20
# and 28 planes over 16 blocks, 16^3 and 32^3 tops, one level above the
# tail (launched cell by cell, and in tiles of which some are partial)
SHAPES = [(8, 6, 10), (8, 8, 8), (16, 8, 12), (12, 24, 16), (20, 20, 24), (28, 28, 28),
          (32, 16, 48), (40, 32, 24), (56, 64, 48), (64, 56, 72)]


@pytest.fixture(scope="module")
def C():
    c = ctx()
    yield c
    c.close()


def _case(shape, seed, fr0=1e-5):
    return synth.lognormal_density(shape, seed, sigma=1.0), dict(
        box=2.0 * shape[2], a=1.0, omega_m=0.24, fr0=fr0)


@pytest.mark.parametrize("shape", SHAPES)
def test_fp64_tail_vcycles_match_oracle(C, shape):
    """The same V-cycles as the oracle's: iterates agree to FP64 rounding (the
    bound of the other V-cycle parity tests)."""
    rho, P = _case(shape, 8100)
    ref = O.solve(rho, ncycles=2, **P)
    u = torch.zeros(shape, dtype=torch.float64, device="cuda")
    C.vcycles(dev(rho), u, 2, **P)
    assert np.abs(host(u) - ref.u).max() < 1e-10


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("opts", [{}, dict(pre=1, post=2, relax=1.15), dict(fmg=1),
                                  dict(tau_alpha=1e-13)])
def test_mixed_tail_solve_matches_oracle(C, shape, opts):
    """rms(L) <= 1e-11 fixes u to about 1e-10 (smallest mass term beta/2 ~ 1.6);
    the oracle is solved to 1e-12."""
    rho, P = _case(shape, 8200)
    ref = O.solve(rho, tol=1e-12, **P)
    u = torch.zeros(shape, dtype=torch.float64, device="cuda")
    st, s = C.solve(dev(rho), u, tol=1e-11, prec="mixed", **opts, **P)
    assert st == 0 and s.res_rms <= 1e-11
    assert np.abs(host(u) - ref.u).max() < 1e-8


@pytest.mark.parametrize("post", [1, 2])
def test_mixed_batch_of_tails_and_launched_grids(C, post):
    """Fields whose tails begin at different depths, more of them than clusters
    fit the GPU, with odd and even numbers of sweeps: each as if solved alone."""
    shapes = [(64, 64, 64), (32, 32, 32), (48, 32, 16), (16, 16, 16)] * 6
    cases = [_case(s, 8300 + i, fr0=(1e-5, 1e-6)[i % 2]) for i, s in enumerate(shapes)]
    us = [torch.zeros(s, dtype=torch.float64, device="cuda") for s in shapes]
    st, stats = C.solve_batch([dev(r) for r, _ in cases], us,
                              boxes=[p["box"] for _, p in cases], avals=[1.0] * len(cases),
                              fr0s=[p["fr0"] for _, p in cases], omega_m=0.24, tol=1e-11,
                              prec="mixed", pre=1, post=post, tiling=1)
    assert st == 0
    for i in range(8):
        ref = O.solve(cases[i][0], tol=1e-12, **cases[i][1])
        assert np.abs(host(us[i]) - ref.u).max() < 1e-8, shapes[i]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[(8, 8, 8)], [(24, 20, 28), (16, 16, 16), (32, 32, 32)],
                                   [(16, 12, 8)] * 10])
def test_patch_tails_match_oracle(C, prec, sizes):
    n = 40
    rho, P = _case((n,) * 3, 8400)
    patches, gp = [], []
    for i, s in enumerate(sizes):
        org = (2 + 3 * (i % 4), 1 + i, 3)
        b = rho[org[2]:org[2] + s[0] // 2, org[1]:org[1] + s[1] // 2, org[0]:org[0] + s[2] // 2]
        r = synth.refine_density(b, 8500 + i)
        patches.append(dict(parent=-1, origin=org, rho=r))
        gp.append(dict(parent=-1, origin=org, density=dev(r),
                       u=torch.zeros(s, dtype=torch.float64, device="cuda")))
    _, ref = O.solve_levels(rho, patches, tol=1e-12, **P)
    u = torch.zeros((n,) * 3, dtype=torch.float64, device="cuda")
    st, _ = C.solve_levels(dev(rho), u, gp, tol=1e-11, prec=prec, **P)
    assert st == 0
    for p, r in zip(gp, ref):
        assert np.abs(host(p["u"]) - r.u).max() < 1e-8


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("dims,count,relax", [((16, 18, 20), 1, 1.0), ((24, 24, 24), 3, 1.25),
                                              ((40, 36, 32), 6, 1.0)])
def test_masked_tail_matches_oracle(C, prec, dims, count, relax):
    """Regions whose levels are all in the one-block tail, and with launched
    levels above it (more than 4096 active cells FP32, 256 FP64); rms(L) <= 1e-11
    fixes u to about 1e-10."""
    from oracle import masked as OM
    rho = synth.lognormal_density(dims, 8600, sigma=1.0)
    r = 0.2 * min(dims)
    m = synth.sphere_union_mask(rho, count, (0.8 * r, 1.4 * r), 8601)
    m[m > 0] = np.where(np.arange((m > 0).sum()) % 3 == 0, 0.5, 1.0)
    u0 = 0.1 * np.cos(np.arange(m.size).reshape(m.shape) / 50.0)
    P = dict(box=64.0, a=1.0, omega_m=0.24, fr0=1e-5)
    ref = OM.solve(u0, m, rho, h=1.0 / 64, tol=1e-12, **P)
    u = dev(u0)
    st, s = C.solve_masked(dev(rho), dev(m), u, h=1.0 / 64, tol=1e-11, prec=prec, relax=relax, **P)
    assert st == 0 and s.res_rms <= 1e-11
    assert np.abs(host(u) - ref.u).max() < 1e-8


def _at8(a):
    """The array on the device at an address that is a multiple of 8, not of 16."""
    buf = torch.empty(a.size + 1, dtype=torch.float64, device="cuda")
    t = buf[1:].view(a.shape)
    assert t.data_ptr() % 16 == 8
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return t


def test_arrays_at_odd_multiples_of_8_bytes(C):
    """The FP64 tail and the Poisson passes read the caller's arrays: any
    address that is a multiple of 8 gives the aligned arrays' result."""
    rho, P = _case((16, 16, 16), 8700)
    u0 = np.zeros(rho.shape)
    ua, ub = dev(u0), _at8(u0)
    C.vcycles(dev(rho), ua, 2, **P)
    C.vcycles(_at8(rho), ub, 2, **P)
    assert np.array_equal(host(ua), host(ub))
    pa, pb = dev(u0), _at8(u0)
    C.poisson(dev(rho), ua, pa, tol=1e-10, **P)
    C.poisson(_at8(rho), ub, pb, tol=1e-10, **P)
    assert np.array_equal(host(pa), host(pb))


@pytest.mark.parametrize("shape", [(3, 5, 7), (1, 1, 1), (4, 6, 9), (16, 16, 32)])
def test_poisson_source_of_any_size(C, shape):
    """The source pass works on pairs of cells: odd numbers of cells, and more
    than one block, against the formula (double-float pairs: 1e-12 of its terms)."""
    from oracle import poisson as PO
    rng = np.random.default_rng(3)
    rho, u = np.exp(rng.standard_normal(shape)), rng.standard_normal(shape)
    P = dict(box=64.0, a=0.9, omega_m=0.24, fr0=1e-5)
    out = torch.empty(shape, dtype=torch.float64, device="cuda")
    C.poisson_source(_at8(rho), _at8(u), out, **P)
    ref = PO.source(u, rho, **P)
    assert np.abs(host(out) - ref).max() < 1e-12 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("shape", [(8, 8, 8), (16, 24, 12), (32, 32, 32), (48, 40, 56),
                                   (96, 64, 96), (40, 40, 40)])
@pytest.mark.parametrize("pre,post,relax", [(1, 1, 1.2), (2, 2, 1.0)])
def test_poisson_tail_matches_fft(C, shape, pre, post, relax):
    """Levels in the cluster and in one block, uneven planes, and a coarsest
    grid of odd sides (40 -> 5, launched): the exact discrete solution, to the
    tolerance times the inverse of the smallest eigenvalue (4 pi^2 per unit box)."""
    from oracle import poisson as PO
    rho, P = _case(shape, 8800)
    u, phi = np.zeros(shape), torch.zeros(shape, dtype=torch.float64, device="cuda")
    st, s, _ = C.poisson(dev(rho), dev(u), phi, tol=1e-10, pre=pre, post=post, relax=relax, **P)
    if max(shape) == min(shape) == 40 and st != 0:
        pytest.skip("odd coarsest grids need not converge")
    ref, _ = PO.solve_periodic(PO.source(u, rho, **P), 1.0 / shape[2])
    assert st == 0 and s.res_rms <= 1e-10
    assert np.abs(host(phi) - ref).max() < 1e-9


@pytest.mark.parametrize("shape", [(24, 40, 72), (2, 18, 66), (24, 512, 1280)])
def test_symmetron_prolongation_tiles(C, shape):
    """One FP64 V-cycle on grids whose coarse level ends inside a prolongation
    tile, has one plane, and has a short last chunk of planes: the oracle's
    iterate up to rounding.  (Coarsest grids of even sides: on odd ones cells of
    one colour are neighbours across the boundary.)"""
    from oracle import symmetron as SY
    P = dict(a=1.0, a_ssb=0.5, lambda0=1.0)
    rho = synth.lognormal_density(shape, 77, sigma=1.0)
    ref = SY.solve(rho, box=0.5 * shape[2], tol=1e-30, max_cycles=1, **P)
    chi = torch.empty(shape, dtype=torch.float64, device="cuda")
    C.symmetron(dev(rho), chi, box=0.5 * shape[2], tol=1e-30, prec="fp64", initial_guess=0,
                max_vcycles=1, **P)
    assert np.abs(host(chi) - ref.chi).max() < 1e-10


@pytest.mark.parametrize("bg", [False, True])
@pytest.mark.parametrize("shape", [(40, 34, 66), (40, 36, 132), (64, 52, 36), (34, 50, 70)])
def test_tiled_residual_and_restriction(C, shape, bg):
    """Tiles that end within the grid in x and y, rows of whole quads and not,
    several chunks: two V-cycles (the second after an outer step in the
    correction form) with the tiled kernels and with one thread per cell give
    the same iterate up to FP32 rounding.  The sums of a residual's terms round
    to 6 eps of |u| <= 20 each; a neighbour mixed up changes u by its
    variation between cells, of order 1e-2 and more."""
    rho, P = _case(shape, 8900)
    out = []
    for tiling in (-1, 1):
        u = torch.zeros(shape, dtype=torch.float64, device="cuda")
        C.solve(dev(rho), u, tol=1e-30, prec="mixed", tiling=tiling, fmg=0,
                max_vcycles=12 if bg else 2, **P)
        out.append(host(u))
    assert np.abs(out[0]).max() > 0.1
    assert np.abs(out[0] - out[1]).max() < 12 * 6e-8 * 20


def test_tiled_patch_of_pairs(C):
    """A patch whose rows are not whole quads and end within a tile."""
    n = 48
    rho, P = _case((n,) * 3, 8901)
    prho = synth.lognormal_density((40, 36, 70), 8902, sigma=1.0)
    org = (4, 4, 6)
    dom, pres = O.solve_levels(rho, [dict(parent=-1, origin=org, rho=prho)], tol=1e-11, **P)
    u0 = torch.zeros((n,) * 3, dtype=torch.float64, device="cuda")
    vc = []
    for tiling in (-1, 1):
        u0.zero_()
        g = dict(parent=-1, origin=org, density=dev(prho),
                 u=torch.zeros(prho.shape, dtype=torch.float64, device="cuda"))
        st, stats = C.solve_levels(dev(rho), u0, [g], tol=1e-11, prec="mixed", tiling=tiling, **P)
        assert st == 0
        assert np.abs(host(g["u"]) - pres[0].u).max() < 1e-8
        vc.append(sum(s.vcycles for s in stats))
    assert abs(vc[0] - vc[1]) <= 1


@pytest.mark.parametrize("tiled", [1, 8, 16])
@pytest.mark.parametrize("c", [-6.0, -2.1, -0.7, -0.35, -0.05, 0.05, 0.36, 1.1])
def test_sweeps_over_the_range_of_u(C, tiled, c):
    """The sweeps' e^u - 1 on both sides of the ends of its reduction (u = +-ln2
    / 2, multiples of ln2) and near zero: two FP32 sweeps against the FP64
    oracle, to a few hundred FP32 roundings of u (at least 1)."""
    shape = (24, 20, 36)
    rng = np.random.default_rng(29)
    P = dict(box=128.0, a=1.0, omega_m=0.24, fr0=1e-5, h=1.0 / 40)
    f32 = lambda a: a.astype(np.float32).astype(np.float64)  # noqa: E731
    u0, f = f32(c + 0.04 * rng.standard_normal(shape)), f32(rng.standard_normal(shape) * 0.05)
    ref = O.smooth(u0, np.ones(shape), 2, f=f, **P)
    u = torch.from_numpy(u0.astype(np.float32)).cuda()
    C.smooth_f32(u, 2, f=torch.from_numpy(f.astype(np.float32)).cuda(), tiled=tiled, **P)
    assert np.abs(host(u) - ref).max() < 2e-5 * max(1.0, abs(c))


@pytest.mark.parametrize("shape,patch", [((36, 34, 132), True), ((96, 48, 64), False),
                                         ((32, 64, 96), False), ((96, 96, 96), False)])
def test_poisson_tiled_residual_and_restriction(C, shape, patch):
    """Tiles that end within the grid, and periodic grids whose coarsest sides of
    3 amplify a residual that does not sum to zero: the oracle's equation is
    met to the tolerance, in the number of cycles multigrid takes."""
    from oracle import poisson as PO
    rho, P = _case(shape, 9000)
    u = 0.3 * np.random.default_rng(9001).standard_normal(shape)
    h = 1.0 / 256 if patch else 1.0 / shape[2]
    s = PO.source(u, rho, **P)
    phi = torch.zeros(shape, dtype=torch.float64, device="cuda")
    kw = {}
    if patch:
        phib = np.random.default_rng(9002).uniform(-1e-3, 1e-3, sum(O.face_sizes(shape)))
        kw = dict(phib=dev(phib), h=h)
    st, stats, _ = C.poisson(dev(rho), dev(u), phi, tol=1e-9, **kw, **P)
    assert st == 0 and stats.res_rms <= 1e-9 and stats.vcycles <= 25
    if patch:
        assert np.sqrt(np.mean(PO.residual(host(phi), s, h, phib) ** 2)) <= 2e-9
    else:
        ref, _ = PO.solve_periodic(s, h)
        assert np.abs(host(phi) - ref).max() <= 1e-7 / 39.0


@pytest.mark.parametrize("shape", [(36, 34, 66), (24, 36, 130), (34, 36, 70)])
def test_poisson_tiled_rows_of_pairs(C, shape):
    """Rows that are not whole quads (their coarsest grids are odd, so these
    solves stall later): the first cycles contract as multigrid does, a factor
    of 10 or more each."""
    rho, P = _case(shape, 9000)
    u = 0.3 * np.random.default_rng(9001).standard_normal(shape)
    phib = np.random.default_rng(9002).uniform(-1e-3, 1e-3, sum(O.face_sizes(shape)))
    phi = torch.zeros(shape, dtype=torch.float64, device="cuda")
    _, s, _ = C.poisson(dev(rho), dev(u), phi, tol=1e-9, phib=dev(phib), h=1.0 / 256, **P)
    h = [abs(v) for v in list(s.hist)[:4]]
    assert h[3] <= 1e-3 * h[0], h
