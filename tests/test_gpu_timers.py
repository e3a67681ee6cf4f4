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


def test_only_launches_are_booked():
    """The fused updates of a step fill their ghosts themselves: no launch is
    booked as a ghost fill, as none runs."""
    w = synth.swirl(2, lmin=2, lmax=4, mx=16)
    _, dtc = synth.time_step(w)
    _, F = pair(fc, w, fc.F32)
    for fused in (True, False):
        F.fused_fill(fused)
        for graphs in (True, False):
            F.graphs(graphs)
            F.timers(True)
            F.step_multirate(0.0, dtc)
            assert F.read_timer(0)[1] > 0
            assert (F.read_timer(1)[1] == 0) == fused
            F.timers(False)
