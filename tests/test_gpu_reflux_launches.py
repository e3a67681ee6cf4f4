"""Refluxing launches of any size run the update that records the face fluxes
as they are chosen untuned (band: the same bits), and a step too short to
change a value changes none."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")


@pytest.mark.parametrize("dtype,warps", [(fc.F32, 8), (fc.F64, 4)])
@pytest.mark.parametrize("nforests", [5, 13, 17])  # 320, 832, 1088 patches a launch
def test_untuned_launches_run_band(dtype, warps, nforests):
    d = fc.make_desc(domain=fc.PERIODIC, mx=32, lmin=3, lmax=3, dtype=dtype,
                     velocity=("swirl", 4.0), nforests=nforests, reflux=1)
    q = np.random.Generator(np.random.PCG64(nforests)).uniform(-1.0, 1.0, (64 * nforests, 32, 32))
    out = {}
    for variant in (-1, 0, 3):
        F = fc.Forest(d, fc.uniform_leaves(3, nforests))
        F.set_q(q)
        F.set_advance_variant(variant, warps)
        F.step_multirate(0.1, 0.4 / 256)
        out[variant] = F.get_q()
    np.testing.assert_array_equal(out[-1], out[3])
    assert not np.array_equal(out[-1], out[0])  # (what tells the two updates apart)


@pytest.mark.parametrize("domain,velocity", [(fc.PERIODIC, ("swirl", 4.0)),
                                             (fc.SPHERE, ("rotation", 1.0, -2.0, 0.5))])
@pytest.mark.parametrize("dtype,dt", [(fc.F32, 1e-42), (fc.F64, 1e-312)])
def test_a_step_too_short_to_change_anything(domain, velocity, dtype, dt):
    """The recorded fluxes are the update's over dt / h, which leaves the range
    of the field's type here."""
    g = np.random.Generator(np.random.PCG64(7))
    d = fc.make_desc(domain=domain, mx=8, lmin=0, lmax=2, dtype=dtype, velocity=velocity, reflux=1)
    lv = fc.uniform_leaves(0, 1, 6 if domain == fc.SPHERE else 1)
    for _ in range(2):
        lv = fc.layout_regrid(d, lv, np.arange(len(lv)) % 3 == 0, 0.6, 0.0)
    F = fc.Forest(d, lv)
    assert sum(n > 0 for n in F.info()["leaves_per_level"]) > 1
    q = g.uniform(0.5, 1.0, (len(lv), 8, 8))
    F.set_q(q)
    q = F.get_q()
    F.step_multirate(0.1, dt)
    np.testing.assert_array_equal(F.get_q(), q)
