"""FP32 coarsest solves of masked regions: 500 sweeps where the slow mode of a
large region falls by a fraction of a per cent per sweep, few at the floor of
FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from paper_1110_1379_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _ball(n, radius):
    g = np.indices((n,) * 3) - (n - 1) / 2
    r = np.sqrt((g ** 2).sum(0))
    return np.where(r <= radius, 1.0, np.where(r < radius + 2, -0.5, -1.0))


def test_large_coarsest_region_keeps_sweeping():
    """Odd sides: one level, 40 cells in radius, diffusion far above the mass
    term.  The slowest mode of a ball of radius R falls by about 1 - (pi / R)^2 / 3
    per Gauss-Seidel sweep (the square of Jacobi's cos), by 0.36 in 500: each FP32
    cycle brings the residual below half of the one before, and no FP64 cycle
    is needed."""
    n = 87
    m = _ball(n, 40.0)
    rho = synth.lognormal_density((n + 1,) * 3, 8600, sigma=1.0)[:n, :n, :n].copy()
    u = dev(0.3 * np.cos(np.arange(n ** 3).reshape(m.shape) / 50.0) - 0.5)
    C = ctx()
    st, s = C.solve_masked(dev(rho), dev(m), u, h=1.0 / n, tol=1e-9, prec="mixed", max_vcycles=3,
                           box=2.0, a=1.0, omega_m=0.24, fr0=1e-4)
    h = list(s.hist)[:4]
    assert s.nhist >= 4 and min(h) > 0, h  # FP64 residuals are recorded as negative values
    assert h[2] < 0.5 * h[1] and h[3] < 0.5 * h[2], h
    C.close()
