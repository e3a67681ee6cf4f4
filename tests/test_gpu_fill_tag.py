"""The one-launch ghost fill and indicator against the separate kernels
(fused_fill off): the same operations on every ghost and cell, so the whole
patch arrays and the indicators are equal bit for bit, on layouts of several
levels of every domain (the cubed sphere's patches at cube edges and vertices
among them), both indicators, both precisions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")

PROBLEMS = {"walls": (fc.WALLS, ("swirl", 4.0), (1, 1)),
            "periodic": (fc.PERIODIC, ("const", 1.0, -0.5), (1, 1)),
            "brick": (fc.BRICK, ("const", 1.0, -0.5), (2, 3)),
            "sphere": (fc.SPHERE, ("rotation", 1.0, -2.0, 0.5), (1, 1))}


@pytest.mark.parametrize("problem", sorted(PROBLEMS))
@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
@pytest.mark.parametrize("indicator", [0, 1])
def test_fill_and_tag_in_one_launch_bitwise(problem, mx, dtype, indicator):
    dom, vel, brick = PROBLEMS[problem]
    g = np.random.Generator(np.random.PCG64(mx + indicator))
    d = fc.make_desc(domain=dom, mx=mx, lmin=0, lmax=4, dtype=dtype, velocity=vel,
                     indicator=indicator, brick=brick)
    lv = fc.uniform_leaves(0, 1, 6 if dom == fc.SPHERE else brick[0] * brick[1])
    for _ in range(4):
        lv = fc.layout_regrid(d, lv, g.uniform(0.0, 1.0, len(lv)), 0.6, 0.0)
    q = g.uniform(-1.0, 1.0, (len(lv), mx, mx))
    out = []
    for fused in (True, False):
        F = fc.Forest(d, lv)
        F.fused_fill(fused)
        F.set_q(q)
        F.poison(float("nan"))
        F.fill_ghosts()
        out.append((F.get_q(full=True), F.tag()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
    assert np.isfinite(out[0][0]).all()
