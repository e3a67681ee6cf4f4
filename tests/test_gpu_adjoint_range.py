"""The adjoint over the range of the field's values: its transposes take the
pieces of the limiter and of the interpolation that the forward step takes.

- The FP64 limiter drops a wave below the normal range or beside a NaN; a
  dropped wave has no partial derivatives, so where every wave is dropped the
  adjoint is the first-order scheme's, bit for bit up to the order of the
  atomic additions (1e-14: some tens of additions)."""
import numpy as np
import pytest

import synth
from gpu_helpers import desc_for, relerr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


def _adjoint(F, q, lam, dt):
    F.set_q(q)
    lam = lam.clone()
    ds = torch.zeros(1, dtype=torch.float64, device="cuda")
    F.adjoint_step_global(0.1, dt, lam, ds)
    return lam.cpu().numpy().astype(np.float64), float(ds)


@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("velocity", [("swirl", 4.0), ("const", 1.0, -0.5)])
@pytest.mark.parametrize("field", ["below the normal range", "one cell NaN"])
def test_a_dropped_wave_has_no_partials(mx, velocity, field):
    w = synth.swirl(3, lmin=2, lmax=2, mx=mx)
    w.velocity = velocity
    g = np.random.Generator(np.random.PCG64(mx))
    q = g.integers(0, 5, (16, mx, mx)) * 1e-310
    if field == "one cell NaN":  # beside jumps of 0, and one of its neighbours set off
        q = np.ones((16, mx, mx))
        q[5, 3, 3] = np.nan
        q[5, 3, 4] = 2.0
    lam = torch.tensor(g.uniform(-1.0, 1.0, q.shape), dtype=torch.float64, device="cuda")
    out = []
    for limiter in ("mc", "first"):
        w.limiter = limiter
        F = fc.Forest(desc_for(fc, w, fc.F64), fc.uniform_leaves(2, 1))
        out.append(_adjoint(F, q, lam, 0.3 / (4 * mx))[0])
    assert np.isfinite(out[1]).all()
    assert relerr(out[0], out[1]) <= 1e-14
