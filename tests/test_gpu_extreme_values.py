"""Values of u far beyond the physical range, where products of the update or
its exponentials leave the range of FP64 or FP32: the operators' results stay
what the formulas give."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from oracle import masked as OM  # noqa: E402
from oracle import oracle as O  # noqa: E402

pytestmark = pytest.mark.gpu
P = dict(box=40.0, a=1.0, omega_m=0.24, fr0=1e-5)


@pytest.fixture(scope="module")
def C():
    c = ctx()
    yield c
    c.close()


@pytest.mark.parametrize("u0", [-30.0, 340.0, 360.0, 500.0, 690.0, 705.0])
def test_fp64_sweeps_of_large_u(C, u0):
    """e^u squared overflows above u = 355; e^u itself is finite up to 709.  An
    update is rounded to about 1e-16 of u."""
    shape = (8, 10, 12)
    u = u0 + 1e-3 * np.random.default_rng(1).standard_normal(shape)
    rho = np.ones(shape)
    ref = O.smooth(u, rho, 2, **P)
    out = dev(u)
    C.smooth(out, dev(rho), 2, **P)
    assert np.abs(ref - u).max() > 1e-4
    assert np.abs(host(out) - ref).max() < 1e-11


@pytest.mark.parametrize("u0", [-720.0, -700.0, 20.0])
def test_fp64_masked_sweep_where_exp_u_is_subnormal(C, u0):
    """e^u is subnormal below u = -708; e^{-u/2} and the step are not.  One level
    (odd sides), one sweep: the residual's square overflows, which ends the
    coarsest solve after it."""
    n = 9
    m = -np.ones((n,) * 3)
    m[1:-1, 1:-1, 1:-1] = 1.0
    rho = np.ones(m.shape)
    u = u0 + 1e-2 * np.random.default_rng(2).standard_normal(m.shape)
    with np.errstate(over="ignore"):
        ref = OM.solve(u, m, rho, h=1.0 / n, tol=1e-9, ncycles=1, cap=4.0, **P)
    out = dev(u)
    C.solve_masked(dev(rho), dev(m), out, h=1.0 / n, tol=1e-9, prec="fp64", max_vcycles=1,
                   newton_step_cap=4.0, **P)
    assert np.abs(ref.u - u).max() > 1e-4
    assert np.abs(host(out) - ref.u).max() < 1e-9
