"""The autotuner times the updates that untuned launches run: on small FP64
launches band takes half the time of staged (64 and 256 patches of 8^2: 8.3
against 14.4 us; of 32^2: 18.5 / 32.9 and 24.7 / 57), so a tuned forest runs it
too, and its steps are those of the untuned forest to rounding."""
import numpy as np
import pytest

from gpu_helpers import F64_TOL, relerr

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("nforests", [1, 4])
def test_small_launches_are_tuned_to_band(mx, nforests):
    d = fc.make_desc(domain=fc.WALLS, mx=mx, lmin=3, lmax=3, dtype=fc.F64,
                     velocity=("swirl", 4.0), nforests=nforests)
    q = np.random.Generator(np.random.PCG64(mx)).uniform(-1.0, 1.0, (64 * nforests, mx, mx))
    out = []
    for tuned in (False, True):
        F = fc.Forest(d, fc.uniform_leaves(3, nforests))
        if tuned:
            rep = F.autotune()
            assert [v[0] for v in rep.values()] == [3], rep
        F.set_q(q)
        F.step_multirate(0.1, 0.4 / (8 * mx))
        out.append(F.get_q())
    assert relerr(out[1], out[0]) <= F64_TOL
