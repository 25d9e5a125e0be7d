"""Caller's device arrays at the smallest alignment their type has (a slice of a
larger tensor): the same results, bit for bit, as with aligned arrays."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from paper_1110_1379_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def C():
    c = ctx()
    yield c
    c.close()


def offset(a, dtype=torch.float64):
    """The array on the device one element past an aligned address."""
    buf = torch.empty(a.size + 1, dtype=dtype, device="cuda")
    t = buf[1:].view(a.shape)
    assert t.data_ptr() % (2 * t.element_size()) == t.element_size()
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
    return t


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [(16, 16, 16), (24, 40, 72)])
def test_symmetron_arrays_at_odd_multiples_of_8_bytes(C, prec, shape):
    """The FP64 V-cycle works on the caller's chi itself."""
    P = dict(a=1.0, a_ssb=0.5, lambda0=1.0, box=0.5 * shape[2])
    rho = synth.lognormal_density(shape, 7, sigma=1.0)
    chi0 = 0.5 + 0.1 * np.random.default_rng(8).standard_normal(shape)
    out = []
    for put in (dev, offset):
        chi = put(chi0)
        C.symmetron(put(rho), chi, tol=1e-30, prec=prec, initial_guess=1, max_vcycles=3, **P)
        out.append(host(chi))
    assert not np.array_equal(out[0], chi0)
    assert np.array_equal(out[0], out[1])


def test_residual_df_arrays_at_odd_multiples_of_8_bytes(C):
    """The double-float defect is written to the caller's d."""
    shape = (12, 16, 20)
    P = dict(box=40.0, a=1.0, omega_m=0.24, fr0=1e-5)
    rho = synth.lognormal_density(shape, 9, sigma=1.0)
    u = 0.3 * np.random.default_rng(10).standard_normal(shape)
    out = []
    for put in (dev, offset):
        d = put(np.zeros(shape))
        C.residual_df(put(u), put(rho), d, **P)
        out.append(host(d))
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("tiled", [0, 1, 8, 16])
@pytest.mark.parametrize("corr", [False, True])
def test_smooth_f32_arrays_at_odd_multiples_of_4_bytes(C, tiled, corr):
    """The tiled FP32 sweeps read the caller's right-hand side and background."""
    shape = (20, 24, 36)
    P = dict(box=40.0, a=1.0, omega_m=0.24, fr0=1e-5)
    rng = np.random.default_rng(11)
    u0 = 0.1 * rng.standard_normal(shape).astype(np.float32)
    bg = rng.standard_normal(shape).astype(np.float32) if corr else None
    f = 0.05 * rng.standard_normal(shape).astype(np.float32)
    out = []
    for put in (lambda a: torch.from_numpy(a).cuda(), lambda a: offset(a, torch.float32)):
        u = put(u0)
        C.smooth_f32(u, 2, f=put(f), bg=None if bg is None else put(bg), tiled=tiled, **P)
        out.append(host(u))
    assert not np.array_equal(out[0], u0)
    assert np.array_equal(out[0], out[1])
