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


# ---- FP32 pair arithmetic on arrays (the operations of frmg_dfmath.cuh)
f32, f64 = np.float32, np.float64


def _two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def _fast_two_sum(a, b):
    s = a + b
    return s, b - (s - a)


def _fma(a, b, c):
    return (a.astype(f64) * b.astype(f64) + c.astype(f64)).astype(f32)


def _add(a, b):
    s, e = _two_sum(a[0], b[0])
    return _fast_two_sum(s, e + (a[1] + b[1]))


def _mul(a, b):
    p = a[0] * b[0]
    e = _fma(a[0], b[0], -p)
    return _fast_two_sum(p, _fma(a[0], b[1], _fma(a[1], b[0], e)))


def _split(v):
    h = np.asarray(v, dtype=f64).astype(f32)
    return h, (v - h.astype(f64)).astype(f32)


def _defect(phi, s, mean, h):
    """L(phi) - (s - mean), every sum of pairs normalised, neighbours in the order
    -x, +x, -y, +y, -z, +z, then the diagonal."""
    p, s = _split(phi), _split(s)
    full = lambda v: tuple(np.full(phi.shape, w, dtype=f32) for w in _split(f64(v)))  # noqa: E731
    acc = None
    for ax in (2, 1, 0):
        for step in (1, -1):
            nb = tuple(np.roll(w, step, axis=ax) for w in p)
            acc = nb if acc is None else _add(acc, nb)
    m = p[0] * f32(-6)
    e = _fma(p[0], np.full(phi.shape, -6, f32), -m)
    acc = _add(acc, _fast_two_sum(m, _fma(p[1], np.full(phi.shape, -6, f32), e)))
    d = _mul(acc, full(1.0 / (h * h)))
    t = _add(s, tuple(-w for w in full(mean)))
    d = _add(d, tuple(-w for w in t))
    return d[0] + d[1]


@pytest.mark.parametrize("shape", [(16, 24, 32), (32, 32, 64)])
def test_defect_rounds_like_normalised_pairs(C, shape):
    """A density made so that phi solves its equation: what is left of the defect
    is the rounding of its own arithmetic, the neighbour sum's above all."""
    n = shape[2]
    rng = np.random.default_rng(7)
    phi = 1.0 + 5e-3 / n ** 2 * rng.standard_normal(shape)  # (a density within 1 +- 0.9)
    phi = sum(w.astype(f64) for w in _split(phi))  # representable as a pair
    lap = -6.0 * phi.astype(np.longdouble)
    for ax in range(3):
        for step in (1, -1):
            lap = lap + np.roll(phi, step, axis=ax)
    z = np.zeros(shape)
    one, s = np.ones(shape), torch.empty(shape, dtype=torch.float64, device="cuda")
    C.poisson_source(dev(2.0 * one), dev(z), s, **P)
    two_gamma = float(host(s).ravel()[0])  # s = 2 gamma (rho - 1) at u = 0
    rho = (1.0 + lap * (n * n) / two_gamma).astype(f64)
    assert rho.min() > 0
    C.poisson_source(dev(rho), dev(z), s, **P)
    _, st, mean = C.poisson(dev(rho), dev(z), dev(phi), tol=1e-30, max_outer=1, max_vcycles=1, **P)
    d = _defect(phi, host(s), mean, 1.0 / n).astype(f64)
    rms = math.sqrt((d * d).mean())
    assert 0 < rms < 20 * 2.0 ** -48 * n * n
    assert abs(st.res0_rms - rms) <= 1e-3 * rms
