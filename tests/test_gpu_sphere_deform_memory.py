"""The deformational flow's fluxes from kept edge coefficients and, for layouts
beyond the budget, from grid corners: the same bits through multirate steps
(captured and direct), a regrid, global steps and a change of the budget on the
way, and the memory each takes."""
import numpy as np
import pytest

import synth
from gpu_helpers import pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("mx,lmin,lmax", [(8, 1, 3), (16, 1, 3), (32, 2, 3)])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
@pytest.mark.parametrize("graphs", [True, False])
def test_corners_give_the_kept_coefficients_bits(mx, lmin, lmax, dtype, graphs):
    w = synth.sphere_deform(seed=3, lmin=lmin, lmax=lmax, mx=mx)
    _, a = pair(fc, w, dtype)
    _, b = pair(fc, w, dtype)
    b.set_coef_budget(0)
    # (a captured step adds its start time on the device, a direct one on the
    # host: times that differ in the last bit, so both forests take one of them)
    a.graphs(graphs)
    b.graphs(graphs)
    dtc = w.dt_lmin
    coef, corners = 64 * (mx + 1) * (mx + 2), 24 * (mx + 3) ** 2

    def same():
        np.testing.assert_array_equal(a.get_q(), b.get_q())
        assert len(a) == len(b)
        return a.info()["device_bytes"] - b.info()["device_bytes"]

    assert same() == len(a) * (coef - corners)
    for n in range(2):
        a.step_multirate(0.2 + n * dtc, dtc)
        b.step_multirate(0.2 + n * dtc, dtc)
    same()
    assert a.tag_regrid(w.tau_refine, w.tau_coarsen) == b.tag_regrid(w.tau_refine, w.tau_coarsen)
    assert same() == len(a) * (coef - corners)
    a.step_multirate(0.5, dtc)
    b.step_multirate(0.5, dtc)
    a.set_velocity_scale(0.5)
    b.set_velocity_scale(0.5)
    a.set_coef_budget(len(a) * coef - 1)  # the first layout beyond it
    b.set_coef_budget(len(b) * coef)      # and within it
    assert same() == len(a) * (corners - coef)
    a.step_global(0.6, dtc / 4)
    b.step_global(0.6, dtc / 4)
    same()
    a.set_coef_budget()
    assert same() == 0
