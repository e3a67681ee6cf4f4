"""The adjoint over the range of the field's values: its transposes take the
pieces of the limiter and of the interpolation that the forward step takes
(and the staged update's limiter, which the row walks' tests do not reach).

- The scheme is homogeneous, so the adjoint of the step of a field times a
  power of two is that of the field (and its velocity derivative times the
  power), also where products of two jumps leave the range; tolerances as in
  the parity tests (FP64 1e-10, FP32 1e-5: one step, some tens of roundings).
- The FP64 limiter drops a wave below the normal range or beside a NaN; a
  dropped wave has no partial derivatives, so where every wave is dropped the
  adjoint is the first-order scheme's, bit for bit up to the order of the
  atomic additions (1e-14: some tens of additions)."""
import numpy as np
import pytest

import synth
from gpu_helpers import desc_for, pair, relerr

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
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
def test_adjoint_of_a_scaled_field(mx, dtype):
    w = synth.swirl(3, lmin=1, lmax=3, mx=mx)
    _, F = pair(fc, w, dtype)
    assert sum(n > 0 for n in F.info()["leaves_per_level"]) > 1
    g = np.random.Generator(np.random.PCG64(mx))
    q = g.choice([0.0, -0.0, 1.0, -1.0, 0.5, 0.25, -0.75], (len(F), mx, mx))
    tol = 1e-10 if dtype == fc.F64 else 1e-5
    lam = torch.tensor(g.uniform(-1.0, 1.0, q.shape), device="cuda",
                       dtype=torch.float64 if dtype == fc.F64 else torch.float32)
    dt = 0.3 / (8 * mx)
    want, ds = _adjoint(F, q, lam, dt)
    for k in (-990, -520, 500) if dtype == fc.F64 else (-100, -60, 100):
        got, dsk = _adjoint(F, np.ldexp(q, k), lam, dt)
        assert relerr(got, want) <= tol, k
        # the sum's terms cancel: against the sum of their magnitudes' scale
        assert abs(np.ldexp(dsk, -k) - ds) <= tol * np.abs(want).sum(), k


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


@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
def test_staged_step_of_a_scaled_field(mx, dtype):
    """The staged update decides signs as the band and walk updates do."""
    w = synth.swirl(3, lmin=1, lmax=2, mx=mx)
    _, F = pair(fc, w, dtype)
    g = np.random.Generator(np.random.PCG64(mx))
    q = g.choice([0.0, -0.0, 1.0, -1.0, 0.5, 0.25, -0.75], (len(F), mx, mx))
    F.set_advance_variant(0, 4)
    out = []
    for k in (0,) + ((-990, -520, 500) if dtype == fc.F64 else (-100, -60, 100)):
        F.set_q(np.ldexp(q, k))
        F.step_global(0.1, 0.3 / (4 * mx))
        out.append(np.ldexp(F.get_q().astype(np.float64), -k))
        assert relerr(out[-1], out[0]) <= (1e-12 if dtype == fc.F64 else 1e-5), k
