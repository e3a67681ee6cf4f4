"""Global steps with the ghosts filled inside the updates against the separate
fill kernels (fused_fill off): the same operations on every ghost, so equal
bits, for every update variant, on layouts of several levels; on the sphere
with both flows, whose edge fluxes come from kept coefficients."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")

PROBLEMS = {"walls": (fc.WALLS, ("swirl", 4.0)), "periodic": (fc.PERIODIC, ("const", 1.0, -0.5)),
            "rotation": (fc.SPHERE, ("rotation", 1.0, -2.0, 0.5)),
            "deform": (fc.SPHERE, ("deform", 2.0, 0.5, 5.0))}


@pytest.mark.parametrize("problem", sorted(PROBLEMS))
@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
def test_fused_global_steps_bitwise(problem, mx, dtype):
    dom, vel = PROBLEMS[problem]
    g = np.random.Generator(np.random.PCG64(mx))
    d = fc.make_desc(domain=dom, mx=mx, lmin=1, lmax=4, dtype=dtype, velocity=vel)
    lv = fc.uniform_leaves(1, 1, 6 if dom == fc.SPHERE else 1)
    for _ in range(3):
        lv = fc.layout_regrid(d, lv, g.uniform(0.0, 1.0, len(lv)), 0.6, 0.0)
    q = g.uniform(0.0, 1.0, (len(lv), mx, mx))
    for variant in (0, 1, 3):
        out = []
        for fused in (True, False):
            F = fc.Forest(d, lv)
            F.set_advance_variant(variant, 4)
            F.fused_fill(fused)
            F.set_q(q)
            for k in range(3):
                F.step_global(0.1 + 1e-4 * k, 1e-4)
            out.append(F.get_q())
        np.testing.assert_array_equal(out[0], out[1])
