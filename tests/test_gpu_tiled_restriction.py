"""The f(R) solver's tiled residual + restriction on grids that have coarser
levels and end inside its 64 x 16 tiles, against one thread per cell."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from oracle import oracle as O  # noqa: E402
from paper_1110_1379_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    c = ctx()
    yield c
    c.close()


def _launched(shape):
    """The grid has a coarser level and more cells than a one-cluster tail takes."""
    return O.num_levels(shape) > 1 and np.prod(shape) > 48 ** 3


def _case(shape, seed):
    return synth.lognormal_density(shape, seed, sigma=1.0), dict(
        box=2.0 * shape[2], a=1.0, omega_m=0.24, fr0=1e-5)


@pytest.mark.parametrize("bg", [False, True])
@pytest.mark.parametrize("shape", [(40, 36, 132), (64, 52, 36), (44, 40, 68), (72, 28, 64),
                                   (20, 88, 196)])
def test_matches_one_thread_per_cell(C, shape, bg):
    """Two V-cycles (the second after an outer step in the correction form) give
    the same iterate up to FP32 rounding: the sums of a residual's terms round to
    6 eps of |u| <= 20 each; a neighbour mixed up changes u by its variation
    between cells, of order 1e-2 and more."""
    assert _launched(shape)
    rho, P = _case(shape, 8900)
    out = []
    for tiling in (-1, 1):
        u = torch.zeros(shape, dtype=torch.float64, device="cuda")
        C.solve(dev(rho), u, tol=1e-30, prec="mixed", tiling=tiling, fmg=0,
                max_vcycles=12 if bg else 2, **P)
        out.append(host(u))
    assert np.abs(out[0]).max() > 0.1
    assert np.abs(out[0] - out[1]).max() < 12 * 6e-8 * 20


@pytest.mark.parametrize("pshape", [(44, 40, 68), (24, 52, 132)])
def test_patch_with_coarser_levels(C, pshape):
    """A patch that ends within a tile: the oracle's solution, in as many cycles
    with the tiled kernels as without."""
    assert _launched(pshape)
    n = 80
    rho, P = _case((n,) * 3, 8901)
    prho = synth.lognormal_density(pshape, 8902, sigma=1.0)
    org = (4, 4, 6)
    dom, pres = O.solve_levels(rho, [dict(parent=-1, origin=org, rho=prho)], tol=1e-11, **P)
    vc = []
    for tiling in (-1, 1):
        u0 = torch.zeros((n,) * 3, dtype=torch.float64, device="cuda")
        g = dict(parent=-1, origin=org, density=dev(prho),
                 u=torch.zeros(pshape, dtype=torch.float64, device="cuda"))
        st, stats = C.solve_levels(dev(rho), u0, [g], tol=1e-11, prec="mixed", tiling=tiling, **P)
        assert st == 0
        assert np.abs(host(g["u"]) - pres[0].u).max() < 1e-8
        vc.append(stats[1].vcycles)
    assert abs(vc[0] - vc[1]) <= 1
