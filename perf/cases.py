"""The calls that users of the package make, with their sizes.

A case names a problem (domain, velocity, patch size, levels, precision), a
layout that surrounds seeded fronts with finest-level patches (as tagging a
front leaves it), and the calls made on it (``kind``):

* ``global``      ``steps`` global time steps from a given field,
* ``multirate``   ``steps`` coarse multirate steps from a given field,
* ``regrid``      twice: a field whose fronts have moved, one tag and regrid,
                  ``steps`` coarse steps on the new layout (there and back, so
                  a pass ends on the layout it started from),
* ``adjoint``     ``steps`` coarse steps and the gradient of a misfit with
                  respect to the initial field and the velocity scale,
* ``adjoint_global``  the adjoint of one global step.

``exact`` computes the same results with dense arrays: each level of each
block is one array over the whole block, its cells outside the level's leaves
filled from the finer or the coarser level, so the update of a level is the
update of one large patch.
"""
import math

import numpy as np
import torch

import paper_1703_03116_gb300 as fc
from paper_1703_03116_gb300.autograd import advect

TAU_REFINE, TAU_COARSEN = 0.05, 0.0125  # the package's defaults
FLOPS_PER_CELL = 50  # of one update with MC limiter and transverse terms


def _case(name, kind, domain, velocity, mx, lmin, lmax, dtype, steps, forests=1, reflux=False,
          place=0):
    """place: seeds where the fronts are, so which layout the case has."""
    c = dict(kind=kind, domain=domain, velocity=velocity, mx=mx, lmin=lmin, lmax=lmax,
             dtype=dtype, steps=steps, forests=forests, reflux=reflux, place=place)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem: 64 patches, every launch far from filling the GPU
        _case("uniform64_mx16_f64", "global", "periodic", "const", 16, 3, 3, "f64", 10),
        # one adaptive forest between two regrids, in both precisions
        _case("swirl_mx32_f32", "multirate", "walls", "swirl", 32, 2, 6, "f32", 4),
        _case("swirl_mx32_f64", "multirate", "walls", "swirl", 32, 2, 6, "f64", 1),
        # the same run with its regrids: one every four coarse steps
        _case("swirl_regrid_mx32_f32", "regrid", "walls", "swirl", 32, 2, 6, "f32", 4),
        # a batched ensemble: launches of thousands of patches
        _case("ensemble256_mx32_f32", "multirate", "walls", "swirl", 32, 2, 6, "f32", 1, 256),
        _case("ensemble64_mx16_f64", "multirate", "walls", "swirl", 16, 2, 6, "f64", 1, 64),
        # the cubed sphere's capacity form: solid-body rotation, deformational flow
        _case("sphere_mx32_f32", "multirate", "sphere", "rotation", 32, 1, 7, "f32", 1),
        _case("deform_mx32_f32", "multirate", "sphere", "deform", 32, 2, 6, "f32", 1),
        # one large uniform grid (4096 x 4096 cells)
        _case("uniform16k_mx32_f32", "global", "walls", "swirl", 32, 7, 7, "f32", 1),
        # small patches with the conservative coarse/fine correction
        _case("reflux_mx8_f32", "multirate", "walls", "swirl", 8, 2, 5, "f32", 2, 1, True),
        # a checkpoint-free gradient, and the adjoint of a global step
        _case("adjoint_mx32_f64", "adjoint", "walls", "swirl", 32, 2, 5, "f64", 4),
        _case("adjoint_global_mx32_f32", "adjoint_global", "walls", "swirl", 32, 2, 6, "f32", 1),
    ]


def draw(rng):
    kind = rng.choice(["global", "multirate", "multirate", "multirate", "regrid", "adjoint",
                       "adjoint_global"])
    mx = rng.choice([8, 16, 32])
    dtype = "f64" if kind == "adjoint" else rng.choice(["f32", "f32", "f64"])
    domain = rng.choice(["walls", "walls", "periodic", "sphere"]
                        if kind in ("global", "multirate") else
                        ["walls"] if kind == "regrid" else ["walls", "periodic"])
    velocity = (rng.choice(["rotation", "deform"]) if domain == "sphere" else
                "const" if domain == "periodic" else "swirl")
    lmin = rng.randint(1, 3)
    # (a regrid needs room to refine; deep narrow forests are in the listed range too)
    lmax = lmin + rng.randint(2 if kind == "regrid" else 0, 4 if kind != "regrid" else 3)
    forests = 1
    if domain != "sphere" and kind in ("global", "multirate"):
        forests = int(round(math.exp(rng.uniform(0.0, math.log(200.0)))))
    reflux = kind == "multirate" and domain != "sphere" and rng.random() < 0.25
    steps = rng.randint(1, 4)
    c = _case("", kind, domain, velocity, mx, lmin, lmax, dtype, steps, forests, reflux,
              rng.randrange(1 << 20))
    most = _updates(dict(listed()[4]))
    while True:  # no dearer than the largest listed case (FP64 runs on a narrow pipe)
        cost = _updates(c) * (8 if dtype == "f64" else 1)
        if cost <= most:
            return c
        c["forests"] = max(1, min(c["forests"] - 1, int(c["forests"] * most / cost)))
        if c["forests"] == 1 and c["steps"] > 1:
            c["steps"] -= 1
        elif c["forests"] == 1 and c["lmax"] > c["lmin"]:
            c["lmax"] -= 1


# ------------------------------------------------------------------ problem


def _blocks(case):
    return 6 if case["domain"] == "sphere" else 1


def _tdtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


_OMEGA = 2.0 * np.pi * np.array([0.48, -0.6, 0.64])  # one revolution in unit time


def _velocity(case):
    return {"const": ("const", 1.0, 0.5), "swirl": ("swirl", 4.0),
            "rotation": ("rotation", *_OMEGA), "deform": ("deform", 2.0, 0.5, 5.0)}[
                case["velocity"]]


def _dt(case):
    """Time step of the finest level (CFL 0.9; the deformational flow's fixed step)."""
    h = 1.0 / (case["mx"] * 2 ** case["lmax"])
    if case["velocity"] == "deform":
        return 2.5e-3 * 4.0 / 2 ** case["lmax"] * 32.0 / case["mx"]
    if case["velocity"] == "rotation":
        return 0.9 * 0.7 * (np.pi / 2) * h / (2 * np.pi)
    return 0.9 * h


def _dt_coarse(case):
    return _dt(case) * 2 ** (case["lmax"] - case["lmin"])


def _desc(case):
    dom = {"walls": fc.WALLS, "periodic": fc.PERIODIC, "sphere": fc.SPHERE}[case["domain"]]
    return fc.make_desc(domain=dom, mx=case["mx"], lmin=case["lmin"], lmax=case["lmax"],
                        dtype=fc.F32 if case["dtype"] == "f32" else fc.F64,
                        velocity=_velocity(case), nforests=case["forests"],
                        reflux=int(case["reflux"]))


def _draws(case):
    """Per forest: its finest level and its front (disc centre, or points on
    the sphere)."""
    g = np.random.Generator(np.random.PCG64([case["place"], 17]))
    lo = max(case["lmin"], case["lmax"] - 2)
    out = []
    for f in range(case["forests"]):
        top = int(g.integers(lo, case["lmax"] + 1)) if case["forests"] > 1 else case["lmax"]
        if case["domain"] == "sphere":
            v = g.normal(size=(3, 3))
            out.append((top, v / np.linalg.norm(v, axis=1, keepdims=True)))
        else:
            out.append((top, g.uniform(0.3, 0.7, 2)))
    return out


# the cube's faces: normal and the two axes of the block coordinates
_FACES = np.array([[(0, 0, 1), (1, 0, 0), (0, 1, 0)], [(0, 0, -1), (1, 0, 0), (0, -1, 0)],
                   [(1, 0, 0), (0, 1, 0), (0, 0, 1)], [(-1, 0, 0), (0, -1, 0), (0, 0, 1)],
                   [(0, 1, 0), (-1, 0, 0), (0, 0, 1)], [(0, -1, 0), (1, 0, 0), (0, 0, 1)]],
                  dtype=np.float64)


def _sphere_points(x, y, faces):
    """Unit vectors (..., 3) of block points; faces: (..., 3, 3) frames."""
    ta, tb = torch.tan((x - 0.5) * math.pi / 2)[..., None], torch.tan((y - 0.5) * math.pi / 2)[..., None]
    P = faces[..., 0, :] + ta * faces[..., 1, :] + tb * faces[..., 2, :]
    return P / P.norm(dim=-1, keepdim=True)


_DISC, _BELL = 0.2, 0.5  # radius of a disc; of the sphere's bells and cylinder


# ------------------------------------------------------------------ layout


def _closure(R, case):
    """Refine until quadrants that touch differ by one level at most."""
    for l in range(max(R), case["lmin"], -1):
        R[l - 1] = R[l - 1] | _halve(_dilate(R[l], case))
    return R


def _halve(M):
    b, n, _ = M.shape
    return M.reshape(b, n // 2, 2, n // 2, 2).any(axis=(2, 4))


def _dilate(M, case):
    P = _pad(torch.from_numpy(M.astype(np.float64)), 1, case).numpy() > 0
    n = M.shape[1]
    return np.logical_or.reduce([P[:, a:a + n, b:b + n] for a in range(3) for b in range(3)])


def _front(case, top, at, l):
    """Quadrants of level l that a front (or a bell) passes through."""
    n = 1 << l
    c = (torch.arange(n, dtype=torch.float64) + 0.5) / n
    y, x = torch.meshgrid(c, c, indexing="ij")
    if case["domain"] == "sphere":
        F = torch.from_numpy(_FACES)[:, None, None]
        X = _sphere_points(x.expand(6, n, n), y.expand(6, n, n), F.expand(6, n, n, 3, 3))
        r = torch.arccos((X @ torch.from_numpy(at).T).clamp(-1, 1))
        half = 0.75 * (math.pi / 2) / n
        hit = (r[..., 2] - _BELL).abs() < half
        if math.pi * (math.pi / 2) / (case["mx"] * n) > TAU_REFINE:  # a bell's slope tags
            hit |= (r[..., :2] < _BELL + half).any(-1)
        return hit.numpy()
    d = torch.hypot(x - at[0], y - at[1])
    return ((d - _DISC).abs() < 0.75 / n).numpy()[None]


def _refined(case):
    """Per forest {level: which quadrants of that level are subdivided}."""
    out = []
    for top, at in _draws(case):
        R = {l: np.ones((_blocks(case), 1 << l, 1 << l), dtype=bool) for l in range(case["lmin"])}
        above = None
        for l in range(case["lmin"], case["lmax"] + 1):
            n = 1 << l
            R[l] = np.zeros((_blocks(case), n, n), dtype=bool)
            if l < top:
                R[l] = _front(case, top, at, l)
                if above is not None:
                    R[l] &= above.repeat(2, 1).repeat(2, 2)
                above = R[l]
        if case["kind"] in ("global", "adjoint_global") and case["lmin"] == case["lmax"]:
            out.append(R)
        else:
            out.append(_closure(R, case))
    return out


def _leaf_masks(R, case):
    """{level: which quadrants are leaves}, from which are subdivided."""
    out = {}
    for l in range(case["lmin"], case["lmax"] + 1):
        inside = np.ones_like(R[l]) if l == case["lmin"] else R[l - 1].repeat(2, 1).repeat(2, 2)
        out[l] = inside & ~R[l]
    return out


def _leaves(case, refined):
    """Leaf rows (forest, block, level, x, y) in field order (Morton within a block)."""
    rows, keys = [], []
    for f, R in enumerate(refined):
        for l, M in _leaf_masks(R, case).items():
            b, y, x = np.nonzero(M)
            rows.append(np.stack([np.full(len(b), f), b, np.full(len(b), l), x, y], 1))
            s = case["lmax"] - l
            k = np.zeros(len(b), dtype=np.int64)
            for i in range(case["lmax"]):
                k |= ((((x << s) >> i) & 1) | ((((y << s) >> i) & 1) << 1)) << (2 * i)
            keys.append(np.stack([rows[-1][:, 0], b, k], 1))
    rows, keys = np.concatenate(rows), np.concatenate(keys)
    return np.ascontiguousarray(rows[np.lexsort((keys[:, 2], keys[:, 1], keys[:, 0]))], np.int32)


def _updates(case):
    """Cell updates of one pass (the first forests counted)."""
    n, few = 0, dict(case, forests=min(case["forests"], 8))
    for R in _refined(few):
        for l, M in _leaf_masks(R, case).items():
            multirate = case["kind"] in ("multirate", "regrid", "adjoint")
            n += int(M.sum()) * (2 ** (l - case["lmin"]) if multirate else 1)
    n = n * case["forests"] / few["forests"] * case["mx"] ** 2 * case["steps"]
    return n * {"regrid": 2, "adjoint": 4, "adjoint_global": 3}.get(case["kind"], 1)


# ------------------------------------------------------------------ fields


def _field(case, seed, leaves, device, shift=0.0):
    """The initial field (n, mx, mx) in the case's precision: fronts of seeded
    heights over a seeded level and ripple; shift moves the fronts along x."""
    mx = case["mx"]
    lv = torch.as_tensor(np.asarray(leaves), device=device).long()
    at = torch.tensor(np.array([a for _, a in _draws(case)]), device=device)[lv[:, 0]]
    h = 1.0 / (mx * 2.0 ** lv[:, 2].double())
    g = np.random.Generator(np.random.PCG64([seed, 29]))
    tall, base, p1, p2 = (torch.tensor(v, device=device)[lv[:, 0], None, None] for v in (
        g.uniform(0.6, 1.0, case["forests"]), g.uniform(0.0, 0.5, case["forests"]),
        *g.uniform(0.0, 6.0, (2, case["forests"]))))
    i = torch.arange(mx, dtype=torch.float64, device=device) + 0.5
    x = ((lv[:, 3, None] * mx + i) * h[:, None])[:, None, :].expand(-1, mx, mx)
    y = ((lv[:, 4, None] * mx + i) * h[:, None])[:, :, None].expand(-1, mx, mx)
    if case["domain"] == "sphere":
        F = torch.from_numpy(_FACES).to(device)[lv[:, 1]][:, None, None]
        X = _sphere_points(x, y, F)
        r = torch.arccos((X[..., None, :] * at[:, None, None]).sum(-1).clamp(-1, 1))
        bell = torch.where(r < _BELL, 0.5 * (1 + torch.cos(math.pi * r / _BELL)), torch.zeros_like(r))
        slot = ((X - at[:, None, None, 2])[..., 2] > -0.25) & ((X - at[:, None, None, 2])[..., 0].abs() < 0.05)
        ripple = torch.sin(4 * X[..., 0] + p1) * torch.cos(3 * X[..., 1] + p2)
        q = bell[..., 0] + bell[..., 1] + ((r[..., 2] < _BELL) & ~slot)
    else:
        dx, dy = x - at[:, 0, None, None] - shift, y - at[:, 1, None, None]
        r2 = dx * dx + dy * dy
        if case["kind"] in ("adjoint", "adjoint_global"):  # smooth: the limiter's pieces are sharp
            q = torch.exp(-r2 / 0.04) + 0.25 * torch.sin(5 * x + 3 * y + p1)
        else:
            q = (r2 < _DISC * _DISC).double()
        ripple = torch.sin(4 * x + p1) * torch.cos(3 * y + p2)
    return (base + tall * q + 0.005 * ripple).to(_tdtype(case)).contiguous()


# ------------------------------------------------------------------ the calls


def prepare(case, seed):
    dev = torch.device("cuda")
    leaves = _leaves(case, _refined(case))
    F = fc.Forest(_desc(case), leaves)
    s = {"case": case, "forest": F, "dt": _dt(case), "dtc": _dt_coarse(case)}
    q0 = _field(case, seed, leaves, dev)
    s["q0"], s["out"] = q0, torch.empty_like(q0)
    if case["kind"] == "regrid":
        # go to and fro until the two layouts repeat
        fields = [_shift(case), 0.0]
        seen = leaves
        for _ in range(8):
            pair = []
            for move in fields:
                F.set_q(_field(case, seed, F.leaves(), dev, move))
                F.tag_regrid(TAU_REFINE, TAU_COARSEN)
                pair.append(F.leaves())
            if len(pair[1]) == len(seen) and (pair[1] == seen).all():
                break
            seen = pair[1]
        # each half starts on the layout that the other half ends on
        s["moved"] = [_field(case, seed, pair[1], dev, fields[0]),
                      _field(case, seed, pair[0], dev, fields[1])]
        s["outs"] = [torch.empty((len(p), case["mx"], case["mx"]), dtype=q0.dtype, device=dev)
                     for p in pair]
    elif case["kind"] == "adjoint":
        s["target"] = _field(case, seed, leaves, dev, 0.03)
        s["scale"] = torch.ones((), dtype=q0.dtype, device=dev, requires_grad=True)
        s["q0"] = q0.clone().requires_grad_(True)
    elif case["kind"] == "adjoint_global":
        s["lam0"] = q0 - _field(case, seed, leaves, dev, 0.03)
        s["lam"] = torch.empty_like(q0)
        s["dscale"] = torch.zeros(1, dtype=torch.float64, device=dev)
    return s


def _shift(case):
    """About as far as fronts move between two regrids."""
    return 0.5 / 2 ** case["lmax"] + 4 * 0.9 * 2 ** (case["lmax"] - case["lmin"]) / (
        case["mx"] * 2 ** case["lmax"])


def run(s):
    c, F, dt, dtc = s["case"], s["forest"], s["dt"], s["dtc"]
    if c["kind"] == "adjoint":
        qn = advect(s["q0"], s["scale"], F, 0.0, dtc, c["steps"], multirate=True)
        loss = 0.5 * ((qn - s["target"]) ** 2).sum()
        gq, gs = torch.autograd.grad(loss, (s["q0"], s["scale"]))
        return {"q": qn.detach(), "grad_q": gq, "grad_scale": gs}
    if c["kind"] == "adjoint_global":
        F.set_q(s["q0"])
        s["lam"].copy_(s["lam0"])
        s["dscale"].zero_()
        F.adjoint_step_global(0.0, dt, s["lam"], s["dscale"])
        return {"grad_q": s["lam"], "grad_scale": s["dscale"]}
    if c["kind"] == "regrid":
        out = {}
        for half in range(2):
            F.set_q(s["moved"][half])
            F.tag_regrid(TAU_REFINE, TAU_COARSEN)
            for k in range(c["steps"]):
                F.step_multirate(k * dtc, dtc)
            out["leaves%d" % half] = F.leaves()
            out["q%d" % half] = F.get_q(out=s["outs"][half])
        return out
    F.set_q(s["q0"])
    for k in range(c["steps"]):
        if c["kind"] == "global":
            F.step_global(k * dt, dt)
        else:
            F.step_multirate(k * dtc, dtc)
    return {"q": F.get_q(out=s["out"])}


def work(case):
    """The field in and the field out once (the sphere: its FP64 capacities and
    edge fluxes too), and the arithmetic of the updates."""
    few = dict(case, forests=min(case["forests"], 8))
    cells = len(_leaves(few, _refined(few))) * case["forests"] / few["forests"] * case["mx"] ** 2
    e = 4 if case["dtype"] == "f32" else 8
    arrays = {"regrid": 4, "adjoint": 4, "adjoint_global": 3}.get(case["kind"], 2)
    per = arrays * e + (24 if case["domain"] == "sphere" else 0)
    return {"bytes": cells * per, "flops": _updates(case) * FLOPS_PER_CELL}


# ------------------------------------------------------------------ 64 bits


def _pad(A, g, case):
    """A (blocks, n, n) with g ghost layers: wrapped, extended, or folded over
    the cube's edges."""
    if case["domain"] != "sphere":
        mode = "circular" if case["domain"] == "periodic" else "replicate"
        return torch.nn.functional.pad(A[:, None], (g, g, g, g), mode=mode)[:, 0]
    n = A.shape[1]
    P = torch.nn.functional.pad(A[:, None], (g, g, g, g))[:, 0]
    for b in range(6):
        for side in range(4):
            src = _strip(n, g, b, side).to(A.device)
            strip = A.reshape(-1)[src]
            if side < 2:
                c = 0 if side == 0 else n + g
                P[b, g:g + n, c:c + g] = strip
            else:
                r = 0 if side == 2 else n + g
                P[b, r:r + g, g:g + n] = strip
        for cy in (0, 1):  # beyond a vertex of the cube: the mean of the edge ghosts beside
            for cx in (0, 1):
                rows = slice(0, g) if cy == 0 else slice(n + g, n + 2 * g)
                cols = slice(0, g) if cx == 0 else slice(n + g, n + 2 * g)
                jr, ic = (g if cy == 0 else n + g - 1), (g if cx == 0 else n + g - 1)
                P[b, rows, cols] = 0.5 * (P[b, jr, cols][None, :] + P[b, rows, ic][:, None])
    return P


_STRIPS = {}


def _strip(n, g, b, side):
    """Flat indices of the cells that fill the ghosts of face b beyond a side
    (-x, +x, -y, +y): overshoot becomes depth, the index along the edge stays."""
    key = (n, g, b, side)
    if key not in _STRIPS:
        nrm, ex, ey = _FACES[b]
        # doubled cell-centre coordinates in [-n, n] along each axis
        lay = (2 * np.arange(g) + 1).astype(np.float64)  # depth beyond the edge
        lay = lay[::-1] if side in (0, 2) else lay
        along = 2 * np.arange(n) + 1.0 - n
        out, t = (ex, ey) if side < 2 else (ey, ex)
        sgn = -1.0 if side in (0, 2) else 1.0
        if side < 2:
            D, T = np.meshgrid(lay, along)          # (n, g)
        else:
            T, D = np.meshgrid(along, lay)          # (g, n)
        P = (sgn * n) * out + T[..., None] * t + (n - D)[..., None] * nrm
        c = int(np.argmax(_FACES[:, 0] @ (sgn * out)))
        i = ((P @ _FACES[c, 1] + n - 1) / 2).round().astype(np.int64)
        j = ((P @ _FACES[c, 2] + n - 1) / 2).round().astype(np.int64)
        _STRIPS[key] = torch.from_numpy((c * n + j) * n + i)
    return _STRIPS[key]


def _minmod(a, b):
    return torch.where(a * b <= 0, torch.zeros_like(a), torch.where(a.abs() < b.abs(), a, b))


class _Dense:
    """One forest's levels as dense arrays in 64 bits."""

    def __init__(self, case, R, device, scale=None):
        self.c, self.dev, self.mx = case, device, case["mx"]
        self.scale = 1.0 if scale is None else scale
        self.levels = range(case["lmin"], case["lmax"] + 1)
        masks = _leaf_masks(R, case)
        up = lambda M: torch.from_numpy(M).to(device).repeat_interleave(self.mx, 1).repeat_interleave(self.mx, 2)  # noqa: E731
        self.leaf = {l: up(masks[l]) for l in self.levels}
        self.fine = {l: up(R[l]) for l in self.levels}
        self.any = {l: bool(masks[l].any()) for l in self.levels}
        self.K = {l: self._metric(l) for l in self.levels} if case["domain"] == "sphere" else None
        self.trig = {}
        self.D, self.old, self.flux = {}, {}, {}

    # -- geometry
    def _metric(self, l):
        n = self.mx << l
        k = (torch.arange(-2, n + 3, dtype=torch.float64, device=self.dev)) / n
        y, x = torch.meshgrid(k, k, indexing="ij")
        faces = torch.from_numpy(_FACES).to(self.dev)
        X = torch.stack([_sphere_points(x, y, faces[b].expand(*x.shape, 3, 3)) for b in range(6)])
        a, b, c, d = X[:, :-1, :-1], X[:, :-1, 1:], X[:, 1:, 1:], X[:, 1:, :-1]

        def tri(a, b, c):
            num = (a * torch.linalg.cross(b - a, c - a)).sum(-1).abs()
            den = 1 + (a * b).sum(-1) + (b * c).sum(-1) + (c * a).sum(-1)
            return 2 * torch.atan2(num, den)

        K = tri(a, b, c) + tri(a, c, d)
        if self.c["velocity"] == "rotation":
            w = torch.tensor(_OMEGA, device=self.dev)
            fx = (X[:, 1:] - X[:, :-1]) @ w
            fy = (X[:, :, :-1] - X[:, :, 1:]) @ w
            return K, fx, fy
        return K, X, None

    def _speeds(self, l, t):
        """Speeds (sphere: volume fluxes) of x-edges (rows -1..n, columns 0..n)
        and y-edges (rows 0..n, columns -1..n)."""
        n, c = self.mx << l, self.c
        if c["velocity"] == "const":
            one = torch.ones((1, 1, 1), dtype=torch.float64, device=self.dev)
            return 1.0 * one * self.scale, 0.5 * one * self.scale
        if c["velocity"] == "swirl":
            h = 1.0 / n
            if l not in self.trig:
                k = torch.arange(-1, n + 2, dtype=torch.float64, device=self.dev)
                self.trig[l] = torch.sin(math.pi * k * h) ** 2, torch.sin(math.pi * (2 * k + 1) * h)
            s2, s1 = self.trig[l]
            u = math.cos(math.pi * t / 4.0) * math.sin(math.pi * h) / (math.pi * h) * self.scale
            return ((u * s2[1:-1])[None, None, :] * s1[:-1][None, :, None],
                    -(u * s2[1:-1])[None, :, None] * s1[:-1][None, None, :])
        K, A, B = self.K[l]
        if c["velocity"] == "rotation":
            return A[:, 1:-1, 2:-2], B[:, 2:-2, 1:-1]
        a = 2 * math.pi * t / 0.5
        s = A[..., 1] * math.cos(a) - A[..., 0] * math.sin(a)
        kc, Z, rot = 2.0 * math.cos(math.pi * t / 0.5), A[..., 2], 2 * math.pi / 5.0
        diff = lambda p, q, zp, zq: kc * (q - p) * (q + p) - rot * (zq - zp)  # noqa: E731
        fx = diff(s[:, 1:], s[:, :-1], Z[:, 1:], Z[:, :-1])
        fy = diff(s[:, :, :-1], s[:, :, 1:], Z[:, :, :-1], Z[:, :, 1:])
        return fx[:, 1:-1, 2:-2], fy[:, 2:-2, 1:-1]

    # -- filling
    def average(self, F, l):
        """Level l+1's array F averaged onto level l."""
        b, n, _ = F.shape
        quad = lambda X: X.reshape(b, n // 2, 2, n // 2, 2)  # noqa: E731
        if self.K is None:
            return quad(F).mean(dim=(2, 4))
        K = self.K[l + 1][0][:, 2:-2, 2:-2]
        return quad(F * K).sum(dim=(2, 4)) / quad(K).sum(dim=(2, 4))

    def interpolate(self, A):
        P = _pad(A, 1, self.c)
        q = P[:, 1:-1, 1:-1]
        sx = 0.25 * _minmod(P[:, 1:-1, 2:] - q, q - P[:, 1:-1, :-2])
        sy = 0.25 * _minmod(P[:, 2:, 1:-1] - q, q - P[:, :-2, 1:-1])
        b, n, _ = q.shape
        rows = [torch.stack([q - sx + k * sy, q + sx + k * sy], -1).reshape(b, n, 2 * n) for k in (-1, 1)]
        return torch.stack(rows, 2).reshape(b, 2 * n, 2 * n)

    def filled(self, l, own, coarse):
        """Level l over its whole blocks: its leaves' values `own`, averages of
        the finer level, interpolation of the (filled) coarser one."""
        out = own
        if l < self.c["lmax"] and l + 1 in self.D:
            out = torch.where(self.fine[l], self.average(self.D[l + 1], l), out)
        if coarse is not None:
            out = torch.where(self.leaf[l] | self.fine[l], out, self.interpolate(coarse))
        return out

    # -- the update
    def update(self, l, A, t, dt):
        n = self.mx << l
        Q = _pad(A, 2, self.c)
        u, v = self._speeds(l, t)
        if self.K is None:
            w = lambda rows, cols: float(n)  # noqa: E731
        else:
            iK = 1.0 / self.K[l][0]
            w = lambda rows, cols: iK[:, rows, cols]  # noqa: E731
        r = slice(1, n + 3)  # rows / columns -1..n
        m = slice(2, n + 2)  # rows / columns 0..n-1

        def edges(s, a, b, c, d, wb, wc):
            W = c - b
            Wup = torch.where(s >= 0, b - a, d - c)
            half, dW, dU = 0.5 * (W + Wup), 2 * W, 2 * Wup
            pick_h = (half.abs() <= dW.abs()) & (half.abs() <= dU.abs())
            lim = torch.where(pick_h, half, torch.where(dW.abs() <= dU.abs(), dW, dU))
            lim = torch.where(W * Wup > 0, lim, torch.zeros_like(lim))
            ab = s.abs()
            cor = 0.5 * ab * (1 - dt * ab * 0.5 * (wb + wc)) * lim
            sp, sm = torch.where(s > 0, s, 0 * s), torch.where(s < 0, s, 0 * s)
            return sp * b + sm * c + cor, sp * W - cor, sm * W + cor, sp, sm

        col = lambda k: slice(k, k + n + 1)  # noqa: E731
        Fx, XP, XM, up, um = edges(u, Q[:, r, col(0)], Q[:, r, col(1)], Q[:, r, col(2)],
                                   Q[:, r, col(3)], w(r, col(1)), w(r, col(2)))
        Gy, YP, YM, vp, vm = edges(v, Q[:, col(0), r], Q[:, col(1), r], Q[:, col(2), r],
                                   Q[:, col(3), r], w(col(1), r), w(col(2), r))
        X = (XP[:, :, :-1] + XM[:, :, 1:]) * w(r, m)  # into cells, rows -1..n
        Y = (YP[:, :-1] + YM[:, 1:]) * w(m, r)
        inner = lambda s, rows, cols: s[:, rows if s.shape[1] > 1 else slice(None), cols if s.shape[2] > 1 else slice(None)]  # noqa: E731
        rx, cy = slice(1, n + 1), slice(1, n + 1)
        F = Fx[:, rx] - 0.5 * dt * (inner(up, rx, slice(None)) * Y[:, :, :-1] + inner(um, rx, slice(None)) * Y[:, :, 1:])
        G = Gy[:, :, cy] - 0.5 * dt * (inner(vp, slice(None), cy) * X[:, :-1] + inner(vm, slice(None), cy) * X[:, 1:])
        new = A - dt * w(m, m) * ((F[:, :, 1:] - F[:, :, :-1]) + (G[:, 1:] - G[:, :-1]))
        return torch.where(self.leaf[l], new, torch.zeros_like(new)), F, G

    # -- stepping
    def step_global(self, t, dt):
        A = None
        new = {}
        for l in self.levels:
            A = self.filled(l, self.D[l], A)
            new[l] = self.update(l, A, t + 0.5 * dt, dt)[0] if self.any[l] else self.D[l]
        self.D = new

    def step_multirate(self, t, dt):
        self.old, self.flux = {}, {}
        self._level(self.c["lmin"], t, dt, 0.0)

    def _level(self, l, t, dt, alpha):
        if self.any[l]:
            coarse = None
            if l > self.c["lmin"]:
                T = self.old[l - 1]
                if alpha > 0:
                    T = (1 - alpha) * T + alpha * self.D[l - 1]
                coarse = torch.where(self.fine[l - 1], self.average(self.D[l], l - 1), T)
            new, F, G = self.update(l, self.filled(l, self.D[l], coarse), t + 0.5 * dt, dt)
        else:
            new = self.D[l]
        self.old[l], self.D[l] = self.D[l], new
        if self.c["reflux"] and self.any[l]:
            self.flux[l, alpha > 0] = F, G
        if l < self.c["lmax"]:
            self._level(l + 1, t, 0.5 * dt, 0.0)
            self._level(l + 1, t + 0.5 * dt, 0.5 * dt, 0.5)
            if self.c["reflux"] and self.any[l] and self.any[l + 1]:
                self._reflux(l, dt, alpha > 0)

    def _reflux(self, l, dt, slot):
        """Cells beside a finer face exchange their flux for the fine fluxes' mean."""
        n, leaf = self.mx << l, self.leaf[l]
        nu = dt * n
        (F0, G0), (F1, G1) = self.flux[l + 1, False], self.flux[l + 1, True]
        F, G = self.flux[l, slot]
        f = (F0 + F1)[:, :, ::2]
        g = (G0 + G1)[:, ::2]
        dF = F - 0.25 * (f[:, ::2] + f[:, 1::2])
        dG = G - 0.25 * (g[:, :, ::2] + g[:, :, 1::2])
        P = _pad(self.fine[l].double(), 1, self.c) > 0
        if self.c["domain"] == "walls":  # nothing lies beyond a wall
            P[:, 0] = P[:, -1] = False
            P[:, :, 0] = P[:, :, -1] = False
        z = torch.zeros_like(leaf, dtype=torch.float64)
        fix = torch.where(P[:, 1:-1, 2:], nu * dF[:, :, 1:], z) - torch.where(P[:, 1:-1, :-2], nu * dF[:, :, :-1], z)
        fix = fix + torch.where(P[:, 2:, 1:-1], nu * dG[:, 1:], z) - torch.where(P[:, :-2, 1:-1], nu * dG[:, :-1], z)
        self.D[l] = self.D[l] + torch.where(leaf, fix, z)

    # -- the field layout
    def place(self, q, lv):
        """Level arrays from leaf values q (n, mx, mx); lv: rows (block, level, x, y)."""
        for l in self.levels:
            n = 1 << l
            k = torch.nonzero(lv[:, 1] == l)[:, 0]
            A = torch.zeros((_blocks(self.c) * n * n, self.mx, self.mx), dtype=torch.float64, device=self.dev)
            A = A.index_copy(0, (lv[k, 0] * n + lv[k, 3]) * n + lv[k, 2], q[k])
            self.D[l] = A.reshape(-1, n, n, self.mx, self.mx).transpose(2, 3).reshape(-1, n * self.mx, n * self.mx)

    def read(self, lv):
        out = torch.zeros((len(lv), self.mx, self.mx), dtype=torch.float64, device=self.dev)
        for l in self.levels:
            n = 1 << l
            k = torch.nonzero(lv[:, 1] == l)[:, 0]
            A = self.D[l].reshape(-1, n, self.mx, n, self.mx).transpose(2, 3).reshape(-1, self.mx, self.mx)
            out = out.index_copy(0, k, A[(lv[k, 0] * n + lv[k, 3]) * n + lv[k, 2]])
        return out


def _regrid_masks(case, R, front):
    """Subdivided quadrants after one tag and regrid; front: {level: tagged leaves}
    (an untagged leaf's field is flat: it may be coarsened)."""
    leaf = _leaf_masks(R, case)
    N = _closure({l: R[l] | (leaf[l] & front[l] if case["lmin"] <= l < case["lmax"] else False) for l in R}, case)
    new = {l: N[l].copy() for l in N}
    for l in range(case["lmin"], case["lmax"]):
        flat = leaf[l + 1] & ~front[l + 1] & ~N[l + 1]
        n = 1 << l
        family = flat.reshape(-1, n, 2, n, 2).all(axis=(2, 4))
        new[l] &= ~(family & ~_halve(_dilate(N[l + 1], case)))
    return new


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    refined = _refined(case)
    leaves = _leaves(case, refined)
    # dense arrays of every forest take their time on the finest level
    fine = (case["mx"] << case["lmax"]) ** 2 * _blocks(case) * case["forests"] * case["steps"]
    rate = 1 if case["kind"] in ("global", "adjoint_global") else 2 ** (case["lmax"] - case["lmin"] + 1)
    launches = case["forests"] * case["steps"] * rate
    if fine * rate * 2e-9 + launches * 2.5e-3 > 18:
        return None
    q0 = _field(case, seed, leaves, dev).double()
    rows = torch.as_tensor(leaves, device=dev).long()
    dt, dtc = _dt(case), _dt_coarse(case)
    if case["kind"] == "regrid":
        return _exact_regrid(case, seed, refined[0], dev)
    if case["kind"] in ("adjoint", "adjoint_global"):
        q0.requires_grad_(True)
        sc = torch.ones((), dtype=torch.float64, device=dev, requires_grad=True)
        S = _Dense(case, refined[0], dev, sc)
        S.place(q0, rows[:, 1:])
        target = _field(case, seed, leaves, dev, 0.03).double()
        if case["kind"] == "adjoint_global":
            lam = (_field(case, seed, leaves, dev) - _field(case, seed, leaves, dev, 0.03)).double()
            S.step_global(0.0, dt)
            gq, gs = torch.autograd.grad((S.read(rows[:, 1:]) * lam).sum(), (q0, sc))
            return {"grad_q": gq, "grad_scale": gs.reshape(1)}
        for k in range(case["steps"]):
            S.step_multirate(k * dtc, dtc)
        qn = S.read(rows[:, 1:])
        gq, gs = torch.autograd.grad(0.5 * ((qn - target) ** 2).sum(), (q0, sc))
        return {"q": qn.detach(), "grad_q": gq, "grad_scale": gs}
    out = torch.empty_like(q0)
    with torch.no_grad():
        for f, R in enumerate(refined):
            k = torch.nonzero(rows[:, 0] == f)[:, 0]
            S = _Dense(case, R, dev)
            S.place(q0[k], rows[k, 1:])
            for i in range(case["steps"]):
                if case["kind"] == "global":
                    S.step_global(i * dt, dt)
                else:
                    S.step_multirate(i * dtc, dtc)
            out[k] = S.read(rows[k, 1:])
    return {"q": out}


def _exact_regrid(case, seed, R, dev):
    """The two halves of a pass; layouts from the same tags, to and fro."""
    dtc = _dt_coarse(case)
    moves = [_shift(case), 0.0]

    def start(R, move):
        lv = torch.as_tensor(_leaves(case, [R]), device=dev).long()
        S = _Dense(case, R, dev)
        S.place(_field(case, seed, lv.cpu().numpy(), dev, move).double(), lv[:, 1:])
        return S

    def tags(S):
        A, hit = None, {}
        for l in S.levels:
            A = S.filled(l, S.D[l], A)
            P = _pad(A, 1, case)
            g = torch.hypot(P[:, 1:-1, 2:] - P[:, 1:-1, :-2], P[:, 2:, 1:-1] - P[:, :-2, 1:-1]) * 0.5
            n = 1 << l
            hit[l] = (g.reshape(-1, n, S.mx, n, S.mx).amax(dim=(2, 4)) > TAU_REFINE).cpu().numpy()
        return hit

    def moved(S, N):
        """S's field on the layout N (one regrid): averaged or interpolated."""
        T, A = _Dense(case, N, dev), None
        for l in S.levels:
            B = S.filled(l, S.D[l], A)
            T.D[l] = torch.where(T.leaf[l], B, torch.zeros_like(B))
            A = B
        return T

    with torch.no_grad():
        for _ in range(8):
            seen = R
            for move in moves:
                R = _regrid_masks(case, R, tags(start(R, move)))
            if all((R[l] == seen[l]).all() for l in R):
                break
        out = {}
        for half, move in enumerate(moves):
            S = start(R, move)
            R = _regrid_masks(case, R, tags(S))
            S = moved(S, R)
            for k in range(case["steps"]):
                S.step_multirate(k * dtc, dtc)
            lv = _leaves(case, [R])
            out["leaves%d" % half] = lv
            out["q%d" % half] = S.read(torch.as_tensor(lv, device=dev).long()[:, 1:])
    return out
