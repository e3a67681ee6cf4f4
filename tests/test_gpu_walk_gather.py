"""The walk update's own ghost ring (face by face, coarse neighbours computed
where they are read) against the separate fill kernels, and the field's moves
to and from arrays that are not 16-byte aligned.

Both fills apply the same operations in the same order to every ghost, so the
steps are equal bit for bit; layouts of several levels and forests, on every
square domain, give every kind of face and corner, first and last positions of
a coarse patch's side, walls, wraps, and groups of a warp that are not full."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)
fc = pytest.importorskip("paper_1703_03116_gb300")

DOMAINS = {"walls": (fc.WALLS, ("swirl", 4.0), (1, 1)),
           "periodic": (fc.PERIODIC, ("const", 1.0, -0.5), (1, 1)),
           "brick": (fc.BRICK, ("const", -0.5, 0.75), (2, 3))}


def random_forest(domain, mx, dtype, seed, forests):
    dom, vel, brick = DOMAINS[domain]
    g = np.random.Generator(np.random.PCG64(seed))
    d = fc.make_desc(domain=dom, mx=mx, lmin=1, lmax=4, dtype=dtype, velocity=vel,
                     nforests=forests, brick=brick)
    lv = fc.uniform_leaves(1, forests, brick[0] * brick[1])
    for _ in range(4):
        lv = fc.layout_regrid(d, lv, g.uniform(0.0, 1.0, len(lv)), 0.85, 0.0)
    return d, lv, g.uniform(0.0, 1.0, (len(lv), mx, mx))


@pytest.mark.parametrize("domain", sorted(DOMAINS))
@pytest.mark.parametrize("mx", [8, 16, 32])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
def test_walk_gather_is_the_fill_bitwise(domain, mx, dtype):
    d, lv, q = random_forest(domain, mx, dtype, mx + len(domain), 8)
    out = []
    for fused in (True, False):
        F = fc.Forest(d, lv)
        F.set_advance_variant(1, 4)
        F.fused_fill(fused)
        F.set_q(q)
        dt = 0.4 / (mx * 16)
        for k in range(2):
            F.step_multirate(8 * k * dt, 8 * dt)
        out.append(F.get_q())
    assert len({int(x) for x in lv[:, 2]}) >= 3
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("mx", [8, 32])
@pytest.mark.parametrize("dtype", [fc.F32, fc.F64])
def test_field_moves_of_any_alignment(mx, dtype):
    d, lv, q = random_forest("walls", mx, dtype, 5, 2)
    F = fc.Forest(d, lv)
    t = torch.float32 if dtype == fc.F32 else torch.float64
    q = torch.tensor(q, dtype=t, device="cuda")
    for off in (0, 1, 3):
        a = torch.zeros(q.numel() + 8, dtype=t, device="cuda")
        b = torch.zeros_like(a)
        a[off:off + q.numel()] = q.reshape(-1)
        F.set_q(a[off:off + q.numel()])
        F.get_q(out=b[off:off + q.numel()])
        assert torch.equal(a, b)
