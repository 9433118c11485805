"""The work this library is used for, as cases that can be timed and checked through its public calls.

A case is one call (or one fitting step) on seeded synthetic inputs: a shape or a batch of shapes, a
set of Q points and a precision.  ``prepare`` makes what a user's program holds before the call,
``run`` makes the call, ``work`` counts what the call cannot do without, and ``exact`` evaluates the
same transform (Maranville, arXiv 2104.08309, Eqs. 6 and 14) in float64 with plain torch.

Pair counts: every (Q point, segment) or (Q point, face) pair is one term of the sum.  The flops of a
term are those of its formula (a multiply-add is two): ``FLOPS`` below.
"""
from __future__ import annotations

import functools
import math
import random

import torch

import paper_2104_08309_gb300 as pft
from paper_2104_08309_gb300 import synth

# flops of one term: 2D three dot products (9), a sine and a cosine (2), sinc as a polynomial (14), the
# product and the complex sum (5); 3D four dot products (20), the in-face invariants (6), the shortest
# series (16), a sine and a cosine (2), two complex products and the sum (12).  A gradient evaluates the
# term, its derivatives and the update of the record's (or the Q point's) adjoint: about twice as much
# again.
FLOPS = {2: 30, 3: 56}
GRAD = 2.0


def listed():
    return [
        # The smallest calls: a coarse sphere along one scan line, as a form factor is looked at
        # interactively (the paper's sphere along Q_x, Sec. 4.3) ...
        {"name": "mesh_line", "kind": "mesh", "level": 2, "q": "line", "n": 241, "hi": 60.0, "precision": "fp32"},
        # ... and one polygon on a detector image (Sec. 4.1).
        {"name": "loop_image", "kind": "loop", "verts": 64, "nx": 128, "ny": 128, "hi": 40.0, "precision": "fp32"},
        # A powder-averaged small-angle scattering curve: log-spaced |Q| from the Guinier range up, several
        # directions each.  Much of it lies at |Q| R < 1.
        {"name": "mesh_curve", "kind": "mesh", "level": 5, "q": "curve", "n": 48, "dirs": 61, "lo": 0.01, "hi": 20.0,
         "precision": "fp32"},
        # A volume of reciprocal space of an ordinary mesh.
        {"name": "mesh_grid", "kind": "mesh", "level": 5, "q": "grid", "nx": 64, "ny": 64, "nz": 64, "hi": 30.0,
         "precision": "fp32"},
        # The largest: a finely meshed rough particle on a fine volume with odd sides.
        {"name": "mesh_large", "kind": "mesh", "level": 7, "q": "grid", "nx": 97, "ny": 90, "nz": 101, "hi": 60.0,
         "precision": "fp32"},
        # A surface of planar polygon faces (a prism over a many-sided outline), as CAD data come.
        {"name": "prism_grid", "kind": "prism", "verts": 8191, "nx": 64, "ny": 64, "nz": 32, "hi": 30.0,
         "precision": "fp32"},
        # Thousands of polygons of uneven size on one image each, with the schedule kept between calls.
        {"name": "loops_batch", "kind": "loops", "shapes": 4096, "most": 4096, "nx": 64, "ny": 64, "hi": 50.0},
        # One fitting step on a batch of polygons: transform, loss on the amplitudes, vertex gradients.
        {"name": "loops_fit", "kind": "loops_fit", "shapes": 1000, "most": 1500, "nx": 63, "ny": 65, "hi": 50.0},
        # The same for a batch of closed meshes (a set of candidate shapes fitted side by side).
        {"name": "meshes_fit", "kind": "meshes_fit", "shapes": 96, "nx": 24, "ny": 24, "nz": 24, "hi": 30.0},
        # One fitting step of a union of spheres to intensities on a grid (Sec. 4.4's shape).
        {"name": "mesh_fit_grid", "kind": "mesh_fit", "spheres": 16, "level": 4, "q": "grid", "nx": 32, "ny": 32,
         "nz": 32, "hi": 30.0, "q_grad": False},
        # One fitting step of a particle to a small-angle curve, with the gradient of Q as well (the
        # instrument's calibration is fitted along).
        {"name": "mesh_fit_curve", "kind": "mesh_fit", "spheres": 1, "level": 4, "q": "curve", "n": 40, "dirs": 13,
         "lo": 0.02, "hi": 20.0, "q_grad": True},
        # The double-precision path, as a check of single-precision results.
        {"name": "mesh_fp64", "kind": "mesh", "level": 4, "q": "grid", "nx": 24, "ny": 24, "nz": 24, "hi": 30.0,
         "precision": "fp64"},
    ]


def _log(rng, lo, hi):
    return max(int(lo), min(int(hi), int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_q(rng, most):
    """A Q set of at most about ``most`` points."""
    kind = rng.choice(["line", "curve", "grid", "grid"])
    if kind == "line":
        return {"q": "line", "n": _log(rng, 30, min(3000, most)), "hi": round(rng.uniform(10, 60), 2)}
    if kind == "curve":
        n = _log(rng, 12, min(120, max(13, most // 2)))
        return {"q": "curve", "n": n, "dirs": _log(rng, 1, max(2, min(100, most // n))),
                "lo": round(10 ** rng.uniform(-3, -1), 5), "hi": round(rng.uniform(5, 40), 2)}
    side = max(3.0, most ** (1 / 3))
    return {"q": "grid", "nx": _log(rng, 3, side), "ny": _log(rng, 3, side), "nz": _log(rng, 3, side),
            "hi": round(rng.uniform(8, 60), 2)}


def draw(rng):
    kind = rng.choice(["mesh", "mesh", "mesh", "loop", "prism", "loops", "loops_fit", "meshes_fit", "mesh_fit",
                       "mesh_fit"])
    case = {"kind": kind}
    if kind == "mesh":
        case["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        case["level"] = rng.randint(1, 7 if case["precision"] == "fp32" else 4)
        case.update(_draw_q(rng, 900000 if case["precision"] == "fp32" else 14000))
    elif kind == "loop":
        case["precision"] = rng.choice(["fp32", "fp32", "fp64"])
        top = 400 if case["precision"] == "fp32" else 100
        case.update(verts=_log(rng, 3, 20000 if top == 400 else 1000), nx=_log(rng, 5, top), ny=_log(rng, 5, top),
                    hi=round(rng.uniform(10, 60), 2))
    elif kind == "prism":
        case.update(verts=_log(rng, 4, 20000), nx=_log(rng, 4, 70), ny=_log(rng, 4, 70), nz=_log(rng, 4, 70),
                    hi=round(rng.uniform(8, 40), 2), precision="fp32")
    elif kind in ("loops", "loops_fit"):
        case.update(shapes=_log(rng, 2, 4000 if kind == "loops" else 1500), most=_log(rng, 20, 4096),
                    nx=_log(rng, 8, 64), ny=_log(rng, 8, 64), hi=round(rng.uniform(10, 60), 2))
    elif kind == "meshes_fit":
        case.update(shapes=_log(rng, 2, 120), nx=_log(rng, 4, 26), ny=_log(rng, 4, 26), nz=_log(rng, 4, 26),
                    hi=round(rng.uniform(8, 40), 2))
    else:
        case.update(spheres=_log(rng, 1, 16), level=rng.randint(1, 4), q_grad=rng.random() < 0.3)
        case.update(_draw_q(rng, 33000 if rng.random() < 0.5 else 2000))
        if case["q"] == "curve":
            case["dirs"] = min(case["dirs"], 20)
    return case


# --------------------------------------------------------------------------------------------------
# Inputs.
# --------------------------------------------------------------------------------------------------

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    return torch.Generator().manual_seed(int(seed))


@functools.lru_cache(maxsize=None)
def _sphere(level):
    v, f = synth.icosphere(level)
    return torch.from_numpy(v), torch.from_numpy(f)


def _axis(n, hi):
    return -hi + torch.arange(n, dtype=torch.float64) * (2.0 * hi / n)


def _counts(case):
    """Vertex counts of a batch of outlines: log-uniform in [8, most], in a shuffled order."""
    n, most = case["shapes"], max(9, case["most"])
    counts = [int(round(math.exp(math.log(8) + (i + 0.5) / n * (math.log(most) - math.log(8))))) for i in range(n)]
    random.Random(n).shuffle(counts)
    return counts


def _q_points(case, seed):
    if case.get("q") == "line":
        q = torch.zeros(case["n"], 3, dtype=torch.float64)
        q[:, 0] = torch.linspace(0.0, case["hi"], case["n"], dtype=torch.float64)
        return q
    if case.get("q") == "curve":
        mag = torch.logspace(math.log10(case["lo"]), math.log10(case["hi"]), case["n"], dtype=torch.float64)
        d = torch.randn(case["dirs"], 3, dtype=torch.float64, generator=_gen(seed + 1000003))
        d = d / d.norm(dim=1, keepdim=True)
        return (mag[:, None, None] * d[None]).reshape(-1, 3).contiguous()
    axes = [_axis(case[k], case["hi"]) for k in ("nx", "ny", "nz") if k in case]
    return torch.stack(torch.meshgrid(*axes, indexing="ij"), dim=-1).reshape(-1, len(axes)).contiguous()


def _inputs(case, seed):
    """The case's inputs on the CPU (tensors), from the seed alone."""
    g = _gen(seed)
    kind = case["kind"]
    s = {"q": _q_points(case, seed)}
    if kind == "mesh":      # a particle with a rough surface
        v, f = _sphere(case["level"])
        r = 1.0 + 0.03 * (2.0 * torch.rand(v.shape[0], 1, generator=g) - 1.0)
        s.update(verts=(v * r).contiguous(), faces=f)
    elif kind == "loop":
        s["verts"] = torch.from_numpy(synth.star_polygon(case["verts"], seed))
        s["off"] = torch.tensor([0, case["verts"]], dtype=torch.int64)
    elif kind == "prism":
        s["outline"] = torch.from_numpy(synth.star_polygon(case["verts"], seed))
        v, idx, off = synth.extruded_polygon(s["outline"].numpy(), 0.75)
        s.update(verts=torch.from_numpy(v), idx=torch.from_numpy(idx), off=torch.from_numpy(off))
    elif kind in ("loops", "loops_fit"):   # star outlines about centres in [-1, 1)^2
        counts = torch.tensor(_counts(case))
        off = torch.cat([torch.zeros(1, dtype=torch.int64), counts.cumsum(0)])
        k = torch.arange(int(off[-1])) - off[:-1].repeat_interleave(counts)
        t = 2.0 * math.pi * k.double() / counts.repeat_interleave(counts)
        r = 1.0 + 0.3 * torch.rand(t.shape[0], generator=g, dtype=torch.float64)
        c = (2.0 * torch.rand(case["shapes"], 2, generator=g, dtype=torch.float64) - 1.0).repeat_interleave(counts, dim=0)
        s.update(verts=(c + torch.stack([r * t.cos(), r * t.sin()], dim=1)).float(), off=off)
    elif kind == "meshes_fit":   # rough spheres about centres in [-1, 1)^3
        parts, faces, off, n = [], [], [0], 0
        for i in range(case["shapes"]):
            u, f = _sphere(1 + i % 4)
            radius, amp = 0.2 + 0.3 * torch.rand(1, generator=g), 0.05 * (2.0 * torch.rand(u.shape[0], 1, generator=g) - 1.0)
            parts.append(u * radius * (1.0 + amp) + 2.0 * torch.rand(1, 3, generator=g) - 1.0)
            faces.append(f + n)
            off.append(off[-1] + f.shape[0])
            n += u.shape[0]
        s.update(verts=torch.cat(parts).contiguous(), faces=torch.cat(faces).to(torch.int32).contiguous(),
                 off=torch.tensor(off, dtype=torch.int64))
    elif kind == "mesh_fit":
        n = case["spheres"]
        u, f = _sphere(case["level"])
        radius = 0.2 + 0.3 * torch.rand(n, generator=g, dtype=torch.float64) if n > 1 else torch.ones(1, dtype=torch.float64)
        centre = torch.rand(n, 3, generator=g, dtype=torch.float64)
        r = 1.0 + 0.02 * (2.0 * torch.rand(n, u.shape[0], 1, generator=g, dtype=torch.float64) - 1.0)
        v = u.double()[None] * radius[:, None, None] * r + centre[:, None]
        fs = f[None] + u.shape[0] * torch.arange(n, dtype=torch.int32)[:, None, None]
        s.update(verts=v.reshape(-1, 3).float().contiguous(), faces=fs.reshape(-1, 3).to(torch.int32).contiguous())
        # the measured intensities: those of the smooth spheres (Eq. 23), with the usual relative error
        a = s["q"].norm(dim=1)[:, None] * radius[None]
        form = torch.where(a < 0.05, 1.0 / 3.0 - a * a / 30.0, (a.sin() - a * a.cos()) / a.clamp(min=0.05) ** 3)
        amp = (torch.exp(1j * (s["q"] @ centre.T)) * (4.0 * math.pi * radius ** 3 * form)).sum(dim=1)
        s["intensity"] = amp.abs() ** 2
        s["sigma"] = 0.05 * s["intensity"] + 1e-5 * s["intensity"].max()
    if kind in ("loops_fit", "meshes_fit"):   # the measured amplitudes
        n = (case["shapes"], s["q"].shape[0], 2)
        s["data"] = torch.view_as_complex(0.1 * torch.randn(*n, dtype=torch.float64, generator=g))
    return s


def prepare(case, seed):
    dev = _dev()
    s = {k: t.to(dev) for k, t in _inputs(case, seed).items()}
    s["kind"], s["options"] = case["kind"], {"precision": case.get("precision", "fp32")}
    if case["kind"] == "loops":
        s["plan"] = pft.pft2d_batched_prepare(s["off"].cpu(), s["q"].shape[0])
    if case["kind"].endswith("_fit"):
        s["verts"].requires_grad_(True)
        s["q"].requires_grad_(bool(case.get("q_grad")))
    return s


# --------------------------------------------------------------------------------------------------
# One pass.
# --------------------------------------------------------------------------------------------------

def _chi2(f, s):
    """The loss of a fit: chi^2 of the intensities, or of the amplitudes where the data hold those."""
    if "data" in s:
        r = f - s["data"]
        return (r.real * r.real + r.imag * r.imag).sum()
    r = (f.real * f.real + f.imag * f.imag - s["intensity"]) / s["sigma"]
    return (r * r).sum()


def run(s):
    kind = s["kind"]
    if kind == "mesh":
        return pft.pft3d_mesh(s["verts"], s["faces"], s["q"], options=s["options"])
    if kind == "loop":
        return pft.pft2d_polygons(s["verts"], s["q"], s["off"], options=s["options"])
    if kind == "prism":
        return pft.pft3d_polymesh(s["verts"], s["idx"], s["off"], s["q"], options=s["options"])
    if kind == "loops":
        return pft.pft2d_polygons_batched(s["verts"], s["off"], s["q"], prepared=s["plan"])
    if kind == "loops_fit":
        f = pft.ft2d_batched(s["verts"], s["off"], s["q"])
    elif kind == "meshes_fit":
        f = pft.ft3d_batched(s["verts"], s["faces"], s["off"], s["q"])
    else:
        f = pft.ft3d(s["verts"], s["faces"], s["q"])
    wrt = [s["verts"]] + ([s["q"]] if s["q"].requires_grad else [])
    grads = torch.autograd.grad(_chi2(f, s), wrt)
    return [f.detach(), *grads]


# --------------------------------------------------------------------------------------------------
# What a pass cannot do without.
# --------------------------------------------------------------------------------------------------

def _sizes(case):
    """(dim, items, vertices, Q points, pairs, outputs of the transform)."""
    kind = case["kind"]
    nq = {"line": case.get("n"), "curve": case.get("n", 0) * case.get("dirs", 0)}.get(case.get("q"))
    if nq is None:
        nq = case["nx"] * case["ny"] * case.get("nz", 1)
    if kind == "loop":
        return 2, case["verts"], case["verts"], nq, nq * case["verts"], nq
    if kind == "prism":
        faces = 2 * (case["verts"] - 2) + 2 * case["verts"]
        return 3, faces, 2 * case["verts"], nq, nq * faces, nq
    if kind in ("loops", "loops_fit"):
        items = sum(_counts(case))
        return 2, items, items, nq, nq * items, nq * case["shapes"]
    if kind == "meshes_fit":
        faces = sum(20 * 4 ** (1 + i % 4) for i in range(case["shapes"]))
        return 3, faces, faces // 2, nq, nq * faces, nq * case["shapes"]
    faces = 20 * 4 ** case["level"] * case.get("spheres", 1)
    return 3, faces, faces // 2, nq, nq * faces, nq


def work(case):
    dim, items, verts, nq, pairs, outputs = _sizes(case)
    read = 4 * dim * verts + (12 * items if dim == 3 else 0) + 8 * dim * nq
    flops = FLOPS[dim] * pairs
    nbytes = read + 16 * outputs
    if case["kind"].endswith("_fit"):
        # the data, the amplitudes' gradient, the inputs again, and the gradients written
        nbytes += 16 * outputs + read + 16 * outputs + 4 * dim * verts
        flops += GRAD * FLOPS[dim] * pairs
        if case.get("q_grad"):
            nbytes += 8 * dim * nq
            flops += GRAD * FLOPS[dim] * pairs
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------------------------------
# The same in float64 (plain torch).
# --------------------------------------------------------------------------------------------------

def _simplex(x, p):
    """sum_k i^k h_k(x) / (k + p)! over the last dimension's nodes, for |x| up to about 1."""
    h = [torch.ones_like(x[..., 0])] + [torch.zeros_like(x[..., 0]) for _ in range(20)]
    for j in range(x.shape[-1]):
        new = [h[0]]
        for k in range(1, 21):
            new.append(h[k] + x[..., j] * new[k - 1])
        h = new
    re = sum(h[k] * ((-1) ** (k // 2) / math.factorial(k + p)) for k in range(0, 21, 2))
    im = sum(h[k] * ((-1) ** (k // 2) / math.factorial(k + p)) for k in range(1, 21, 2))
    return torch.complex(re, im)


def _segments(p0, p1, q):
    """Eq. 6 for |Q| well above 0: [n_q]."""
    m, d = 0.5 * (p0 + p1), p1 - p0
    qx, qy = q[:, :1], q[:, 1:]
    ph = qx * m[:, 0] + qy * m[:, 1]
    w = (qx * d[:, 1] - qy * d[:, 0]) * torch.sinc((qx * d[:, 0] + qy * d[:, 1]) / (2.0 * math.pi))
    q2 = (q * q).sum(dim=1)
    return torch.complex((w * ph.sin()).sum(dim=1), -(w * ph.cos()).sum(dim=1)) / q2


def _faces(p, q):
    """Eq. 14 (sign-corrected) for |Q| well above 0, p [n, 3, 3]: [n_q]."""
    g = p.mean(dim=1)
    c = p - g[:, None]
    n = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    mu, s = q @ g.T, q @ n.T
    a = [q @ c[:, k].T for k in range(3)]
    P = a[0] * a[0] + a[0] * a[1] + a[1] * a[1]
    T = a[0] * a[1] * a[2]
    short = P < 0.02
    gre = 0.5 - P / 24.0 + P * P / 720.0 - (P ** 3 + T * T) / 40320.0
    gim = T * (-1.0 / 120.0 + 2.0 * P / 5040.0 - 3.0 * P * P / 362880.0)
    X = [n[:, i][None] * q[:, j][:, None] - n[:, j][None] * q[:, i][:, None] for i, j in ((1, 2), (2, 0), (0, 1))]
    x2 = X[0] * X[0] + X[1] * X[1] + X[2] * X[2]
    inv = 1.0 / torch.where(short | (x2 == 0), torch.ones_like(x2), x2)
    zr, zi = torch.zeros_like(P), torch.zeros_like(P)
    for l in range(3):
        k = (l + 1) % 3
        d = c[:, k] - c[:, l]
        w = (d[:, 0] * X[0] + d[:, 1] * X[1] + d[:, 2] * X[2]) * torch.sinc((a[k] - a[l]) / (2.0 * math.pi)) * inv
        psi = 0.5 * (a[k] + a[l])
        zr = zr + w * psi.cos()
        zi = zi + w * psi.sin()
    zr = torch.where(short, -gim, zr)
    zi = torch.where(short, gre, zi)
    f = -(torch.exp(1j * mu) * torch.complex(s * zr, s * zi)).sum(dim=1)
    return f / (q * q).sum(dim=1)


def _transform(corners, q, most):
    """FT(Q) of corners [n, d, d] (segments or triangles, double), in pieces of at most ``most`` pairs
    along Q: yields (rows, amplitudes of those rows)."""
    dim = corners.shape[-1]
    with torch.no_grad():
        lo, hi = corners.reshape(-1, dim).min(dim=0).values, corners.reshape(-1, dim).max(dim=0).values
        c = 0.5 * (lo + hi)
        small = q.detach().norm(dim=1) * (corners.detach() - c).norm(dim=-1).max() < 0.5
    rows = max(1, most // corners.shape[0])
    for series, which in ((True, torch.nonzero(small)[:, 0]), (False, torch.nonzero(~small)[:, 0])):
        for at in which.split(rows):
            p, k = corners - c, q[at]
            if series:
                x = torch.einsum("qd,njd->qnj", k, p)
                f = (torch.linalg.det(p) * _simplex(x, dim)).sum(dim=1)
            else:
                f = _segments(p[:, 0], p[:, 1], k) if dim == 2 else _faces(p, k)
            yield at, f * torch.exp(1j * (k @ c))


def _loop_corners(v):
    return torch.stack([v, v.roll(-1, dims=0)], dim=1)


def exact(case, seed):
    dim, items, _, nq, pairs, outputs = _sizes(case)
    fit = case["kind"].endswith("_fit")
    if pairs > (2.5e9 if fit and case.get("q_grad") else 3.5e9 if fit else 8e9 if dim == 3 else 1.5e10):
        return None
    if case["kind"] in ("loops", "loops_fit", "meshes_fit") and case["shapes"] > 1500:
        return None
    dev = _dev()
    s = {k: t.to(dev) for k, t in _inputs(case, seed).items()}
    q = s["q"]
    if case["kind"] == "prism":
        v = s["verts"].double()
        z0, z1 = v[0, 2], v[-1, 2]
        f = torch.empty(nq, dtype=torch.complex128, device=dev)
        flat = q[:, :2].contiguous()
        for at, part in _transform(_loop_corners(v[:case["verts"], :2]), flat, 1 << 24):
            f[at] = part
        u = 0.5 * q[:, 2] * (z1 - z0)
        f = f * (z1 - z0) * torch.sinc(u / math.pi) * torch.exp(0.5j * q[:, 2] * (z0 + z1))
        return torch.view_as_real(f)
    v = s["verts"].double()

    # the shapes' corners, and the rows of v that they are
    if case["kind"] in ("loop", "loops", "loops_fit"):
        at = torch.arange(v.shape[0], device=dev).split((s["off"][1:] - s["off"][:-1]).tolist())
        rows = [torch.stack([k, k.roll(-1)], dim=1) for k in at]
    else:
        rows = [s["faces"].long()]
        if "off" in s:
            rows = rows[0].split((s["off"][1:] - s["off"][:-1]).tolist())
    one = case["kind"] in ("loop", "mesh", "mesh_fit")
    f = torch.empty(len(rows), nq, dtype=torch.complex128, device=dev)
    with torch.no_grad():
        for i, k in enumerate(rows):
            for at, part in _transform(v[k], q, 1 << 24):
                f[i, at] = part
    if not fit:
        return torch.view_as_real(f[0] if one else f)
    # d loss / d F, then one backward pass per piece of the transform
    leaf = f.clone().requires_grad_(True)
    (w,) = torch.autograd.grad(_chi2(leaf[0] if one else leaf, s), leaf)
    q = q.clone().requires_grad_(True)
    gv, gq = torch.zeros_like(v), torch.zeros_like(q)
    for i, k in enumerate(rows):
        corners = v[k].requires_grad_(True)
        for at, part in _transform(corners, q, 1 << 21):
            a, b = torch.autograd.grad(part, [corners, q], w[i, at])
            gv.index_add_(0, k.reshape(-1), a.reshape(-1, dim))
            gq += b
    out = [f[0] if one else f, gv]
    return out + ([gq] if case.get("q_grad") else [])
