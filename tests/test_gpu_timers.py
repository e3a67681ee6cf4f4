"""The phases that the timers book a call's launches under."""
import pytest

import synth
from gpu_helpers import pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("fused", [True, False])
def test_a_tag_is_booked_as_regrid(fused):
    w = synth.swirl(2, lmin=2, lmax=4, mx=16)
    _, F = pair(fc, w, fc.F32)
    F.fused_fill(fused)
    F.tag()
    F.timers(True)
    F.tag()
    ms, launches, nbytes = F.read_timer(2)
    assert launches == 1 and ms > 0.0
    assert nbytes >= len(F) * 16 * 16 * 4  # every interior value read
    fills = F.read_timer(1)[1]
    F.fill_ghosts()
    ms, launches, nbytes = F.read_timer(1)
    assert launches == (1 if fused else 2) and nbytes > 0.0
    assert fills == (0 if fused else 2)
    F.timers(False)
