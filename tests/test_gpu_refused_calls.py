"""What a refused call leaves behind."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import ctx, dev, host  # noqa: E402
from paper_1110_1379_gb300 import frmg, synth  # noqa: E402

pytestmark = pytest.mark.gpu
P = dict(box=32.0, a=1.0, omega_m=0.24, fr0=1e-5)


@pytest.mark.parametrize("bad", [np.nan, -1.0, np.inf])
@pytest.mark.parametrize("which", [0, 1])
def test_patch_of_invalid_density_leaves_its_u(bad, which):
    """A patch whose density is refused keeps the u its caller gave, and the
    context goes on to solve."""
    C = ctx()
    rho = synth.lognormal_density((16,) * 3, 31, sigma=1.0)
    u = torch.zeros(rho.shape, dtype=torch.float64, device="cuda")
    patches = []
    for i in range(2):
        r = synth.lognormal_density((8, 8, 8), 32 + i, sigma=1.0)
        if i == which:
            r[3, 2, 1] = bad
        patches.append(dict(parent=-1, origin=(2, 2, 2 + 6 * i), density=dev(r),
                            u=torch.full((8, 8, 8), 7.0, dtype=torch.float64, device="cuda")))
    with pytest.raises(frmg.FRError) as ei:
        C.solve_levels(dev(rho), u, patches, tol=1e-8, prec="mixed", **P)
    assert ei.value.status == frmg.FR_EINVAL
    assert b"density" in frmg.load().fr_last_error()
    assert np.array_equal(host(patches[which]["u"]), np.full((8, 8, 8), 7.0))
    patches[which]["density"].fill_(1.0)
    st, _ = C.solve_levels(dev(rho), u, patches, tol=1e-8, prec="mixed", **P)
    assert st == 0
    C.close()
