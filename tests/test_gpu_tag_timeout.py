"""A tag whose bounded wait gives up, or that follows a step whose wait gave
up, reports it before anything is decided: tag and tag_regrid raise the
timeout, the layout and the field stay, and with the limit restored the same
forest tags and regrids as one that never timed out."""
import numpy as np
import pytest

import synth
from gpu_helpers import pair

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("call", ["tag", "tag_regrid"])
@pytest.mark.parametrize("from_step", [False, True])
def test_a_tag_that_gave_up_changes_nothing(call, from_step):
    w = synth.swirl(2, lmin=2, lmax=4, mx=16)
    _, dtc = synth.time_step(w)
    _, ref = pair(fc, w, fc.F64)
    _, gpu = pair(fc, w, fc.F64)
    leaves, q0 = gpu.leaves(), gpu.get_q()
    gpu.set_limits(wait_polls=0)
    if from_step:  # the step gives up, the tag itself does not
        gpu.step_multirate(0.0, dtc)
        gpu.set_limits(wait_polls=-1)
    with pytest.raises(fc.FcError) as e:
        gpu.tag() if call == "tag" else gpu.tag_regrid(w.tau_refine, w.tau_coarsen)
    assert e.value.status == 5  # FC_ERR_TIMEOUT
    gpu.set_limits(wait_polls=-1)
    np.testing.assert_array_equal(gpu.leaves(), leaves)
    if not from_step:
        np.testing.assert_array_equal(gpu.get_q(), q0)
    gpu.set_q(q0)
    np.testing.assert_array_equal(gpu.tag(), ref.tag())
    assert gpu.tag_regrid(w.tau_refine, w.tau_coarsen) == \
        ref.tag_regrid(w.tau_refine, w.tau_coarsen)
    np.testing.assert_array_equal(gpu.leaves(), ref.leaves())
    np.testing.assert_array_equal(gpu.get_q(), ref.get_q())
