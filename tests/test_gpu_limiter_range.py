"""The limited waves of the row-walking updates over the range of the field's
values: the band and walk kernels take minima and signs from the bits (FP64)
or from min/max (FP32), so zero jumps, jumps of either sign and fields scaled
to tiny and large magnitudes (products of two jumps leave the range there)
must give the oracle's step.  Each scale is a power of two, so the oracle's
step of the scaled field is the scaled step; bounds: FP64 1e-12 as every
parity test, FP32 1e-5 (one step of fields of a few cells' variation, some
tens of roundings of 6e-8)."""
import numpy as np
import pytest

import synth
from gpu_helpers import F64_TOL, pair, relerr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("variant", [1, 2, 3])
@pytest.mark.parametrize("mx", [8, 16, 32])
def test_limited_waves_over_the_range(variant, mx):
    w = synth.swirl(3, lmin=1, lmax=2, mx=mx)
    g = np.random.Generator(np.random.PCG64(mx))
    for dtype, tol, scales in ((fc.F64, F64_TOL, (-990, -520, 0, 500)),
                               (fc.F32, 1e-5, (-100, -60, 0, 100))):
        ref, gpu = pair(fc, w, dtype)
        q = g.choice([0.0, -0.0, 1.0, -1.0, 0.5, 0.25, -0.75], ref.get_q().shape)
        gpu.set_advance_variant(variant, 4)
        ref.set_q(q)
        ref.step_global(0.1, 0.3 / (4 * mx))
        want = ref.get_q()
        for k in scales:
            gpu.set_q(np.ldexp(q, k))
            gpu.step_global(0.1, 0.3 / (4 * mx))
            assert relerr(np.ldexp(gpu.get_q().astype(np.float64), -k), want) <= tol, k


@pytest.mark.parametrize("variant", [1, 3])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_limited_waves_beside_cells_without_value(variant, bad):
    """A jump that is NaN limits to 0: what the oracle computes from the
    cells around one that is not finite, the updates compute too."""
    for mx in (8, 32):
        w = synth.swirl(3, lmin=1, lmax=2, mx=mx)
        g = np.random.Generator(np.random.PCG64(mx))
        for dtype, tol in ((fc.F64, F64_TOL), (fc.F32, 1e-5)):
            ref, gpu = pair(fc, w, dtype)
            q = g.random(ref.get_q().shape)
            q.reshape(-1)[g.integers(0, q.size, 3)] = bad
            gpu.set_advance_variant(variant, 4)
            ref.set_q(q)
            gpu.set_q(q)
            ref.step_global(0.1, 0.3 / (4 * mx))
            gpu.step_global(0.1, 0.3 / (4 * mx))
            want, got = ref.get_q(), gpu.get_q().astype(np.float64)
            ok = np.isfinite(want)
            assert 0 < np.count_nonzero(~ok) < 200
            assert np.abs(got[ok] - want[ok]).max() <= tol
