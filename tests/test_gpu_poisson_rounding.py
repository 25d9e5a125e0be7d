"""Accumulations of the Poisson solve's double-float passes, on fields whose
sums can be followed exactly."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402

pytestmark = pytest.mark.gpu
P = dict(box=64.0, a=1.0, omega_m=0.24, fr0=1e-5)
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def C():
    c = ctx()
    yield c
    c.close()


def _runs(shape, run, seed):
    """Densities that are constant on every `run` consecutive cells (and repeat
    after 512 of them): sums of equal values by halves are exact."""
    rng = np.random.default_rng(seed)
    v = np.repeat(np.exp(rng.standard_normal(512 // run)), run)
    return np.tile(v, math.prod(shape) // 512).reshape(shape)


@pytest.mark.parametrize("seed", range(8))
def test_source_mean_is_summed_in_fp64(C, seed):
    """One block: groups of 32 equal values, then five FP64 additions."""
    shape = (8, 8, 16)
    rho, z = _runs(shape, 16, seed), np.zeros(shape)
    s = torch.empty(shape, dtype=torch.float64, device="cuda")
    C.poisson_source(dev(rho), dev(z), s, **P)
    s = host(s).ravel()
    _, _, mean = C.poisson(dev(rho), dev(z), dev(z), tol=1e-10, max_outer=1, max_vcycles=1, **P)
    assert abs(mean - math.fsum(s) / s.size) <= 6 * EPS * np.abs(s).mean()


@pytest.mark.parametrize("seed", range(2))
def test_defect_norm_is_summed_in_fp64(C, seed):
    """phi = 0: the defect is the source less its mean.  Runs of 32 equal squares,
    FP64 beyond."""
    shape = (16, 16, 32)
    rho, z = _runs(shape, 32, 10 + seed), np.zeros(shape)
    s = torch.empty(shape, dtype=torch.float64, device="cuda")
    C.poisson_source(dev(rho), dev(z), s, **P)
    _, st, mean = C.poisson(dev(rho), dev(z), dev(z), tol=1e-10, max_outer=1, max_vcycles=1, **P)
    d = (host(s) - mean).astype(np.float32).astype(np.float64)
    # d d rounded to FP32, then d d + it rounded to FP32 once
    q = (d * d + (d * d).astype(np.float32).astype(np.float64)).astype(np.float32)
    ref = math.sqrt(math.fsum(q.astype(np.float64).ravel() / 2) / d.size)
    assert abs(st.res0_rms - ref) <= 20 * EPS * ref
