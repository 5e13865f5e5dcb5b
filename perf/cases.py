"""What the speed of this framework is measured on.

Every case is one call sequence of a user's program on inputs that are already
on the GPU, through the public binding:

- "solve": one AMR level's step.  The level's mask, right-hand side and
  Dirichlet values are handed over (the mask hierarchy is rebuilt when the
  level changed shape), the guess is reset and the solve runs to its
  tolerance; the potential is read back into a device tensor.
- "batch": the same step for many independent patches of one level, solved
  together; the patches' masks stay, their sources and boundary values change.
- "norm": the allocation-free residual norm of a caller's own fields.
- "unet_forward", "unet_train": the learned initial guess's network,
  inference, and the forward and backward pass of a training step.

The domains are this repository's workloads, synthesised on the GPU: a ball
with a smooth manufactured potential, a union of spheres, a cube with holes of
a few cells, and thresholded-noise blobs with boundary values from a coarser
level.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_1104_1703_gb300 import binding as B

BOUNDARY = {"ball": "faces", "union": "zero", "holes": "zero", "blob": "coarse"}
TOLERANCE = {"ball": 1e-10, "union": 1e-8, "holes": 1e-8, "blob": 1e-8}
PATCH_EDGES = (32, 48, 64, 96, 128)


def _solve(domain, nx, ny, nz, mixed, inner=1, n_cycles=1, rebuild=True):
    return {"kind": "solve", "domain": domain, "nx": nx, "ny": ny, "nz": nz, "mixed": mixed, "inner": inner,
            "n_cycles": n_cycles, "rebuild": rebuild}


def listed():
    return [
        # the smallest level of a run, to a tight tolerance: launches and latency count
        {"name": "ball_32_fp64", **_solve("ball", 32, 32, 32, False)},
        # a small refined patch of odd sizes with values from its parent, the mask kept from the last step
        {"name": "blob_57x43x61_fp64", **_solve("blob", 57, 43, 61, False, rebuild=False)},
        # one 128^3 patch as the learned guess is compared on: one FP32 cycle per refinement step
        {"name": "blob_128_mixed", **_solve("blob", 128, 128, 128, True)},
        # a mid-size box riddled with sub-cell holes and of ragged sizes: the order switch trips
        {"name": "holes_161x200x143_fp64", **_solve("holes", 161, 200, 143, False)},
        # the headline workload in the fast form, 8 FP32 cycles per refinement step
        {"name": "union_256_mixed", **_solve("union", 256, 256, 256, True, inner=8)},
        # the same in the plain FP64 method
        {"name": "union_256_fp64", **_solve("union", 256, 256, 256, False)},
        # W-cycles: a level solved with two coarse iterations per level, new sources on a kept mask
        {"name": "union_128_w2_fp64", **_solve("union", 128, 128, 128, False, n_cycles=2, rebuild=False)},
        # the largest level: 512^3 minus 20000 holes
        {"name": "holes_512_mixed", **_solve("holes", 512, 512, 512, True, inner=8)},
        # all patches of an AMR level together
        {"name": "batch_96", "kind": "batch", "patches": 96},
        # a caller's own convergence check between its own steps
        {"name": "norm_256", "kind": "norm", "nx": 256, "ny": 256, "nz": 256, "faces": True},
        # the learned guess's inference at its own size
        {"name": "unet_forward_128", "kind": "unet_forward", "levels": 4, "nx": 128, "ny": 128, "nz": 128},
        # its training direction at the same size
        {"name": "unet_train_128", "kind": "unet_train", "levels": 4, "nx": 128, "ny": 128, "nz": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    edge = _log_int(rng, lo, hi)
    return {a: max(lo, int(round(edge * rng.uniform(0.6, 1.0)))) for a in ("nx", "ny", "nz")}


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "solve", "batch", "norm", "unet_forward", "unet_train"))
    if kind == "batch":
        return {"kind": kind, "patches": _log_int(rng, 4, 96)}
    if kind == "norm":
        return {"kind": kind, **_box(rng, 32, 400), "faces": rng.random() < 0.5}
    if kind.startswith("unet"):
        return {"kind": kind, "levels": rng.choice((2, 3, 4)),
                **{a: min(128, 8 * _log_int(rng, 3, 18)) for a in ("nx", "ny", "nz")}}
    domain = rng.choice(("ball", "union", "holes", "blob"))
    mixed = rng.random() < 0.5
    w_cycle = not mixed and domain != "holes" and rng.random() < 0.25
    box = _box(rng, 24, 160 if w_cycle else 320)
    return _solve(domain, box["nx"], box["ny"], box["nz"], mixed, inner=rng.choice((1, 2, 4, 8)) if mixed else 1,
                  n_cycles=2 if w_cycle else 1, rebuild=rng.random() < 0.7)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

class _Draws:
    """Uniform and normal draws on the GPU from a seed."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))

    def uniform(self, shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(shape, generator=self.gen, device="cuda", dtype=torch.float64)

    def normal(self, shape):
        return torch.randn(shape, generator=self.gen, device="cuda", dtype=torch.float64)


def _centres(n, h):
    return (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h


def _edges(n, h):
    return torch.arange(n + 1, device="cuda", dtype=torch.float64) * h


def _waves(a, p, z, y, x):
    """sum_m a_m prod_axis sin(pi c + p_m) on the grid z, y, x."""
    sz, sy, sx = (torch.sin(math.pi * c[None, :] + p[:, d:d + 1]) for d, c in enumerate((z, y, x)))
    return torch.einsum("m,mk,mj,mi->kji", a, sz, sy, sx).contiguous()


def _ball(d, shape, h):
    """Active inside a ball; a sum of sines as the potential, its Laplacian as rho and its values on the faces."""
    nz, ny, nx = shape
    z, y, x = _centres(nz, h), _centres(ny, h), _centres(nx, h)
    half = [0.5 * n * h for n in shape]
    c = [v + float(s) for v, s in zip(half, d.uniform((3,), -0.02, 0.02).cpu() * min(half))]
    r2 = (z - c[0]).square()[:, None, None] + (y - c[1]).square()[None, :, None] + (x - c[2]).square()[None, None, :]
    mask = (r2 < (0.8 * min(half)) ** 2).to(torch.int8)
    a, p = d.normal((3,)), d.uniform((3, 3), 0.0, math.pi)
    rho = -3.0 * math.pi ** 2 * _waves(a, p, z, y, x)
    faces = [_waves(a, p, z, y, _edges(nx, h)), _waves(a, p, z, _edges(ny, h), x), _waves(a, p, _edges(nz, h), y, x)]
    return {"mask": mask, "rho": rho, "faces": faces}


def _union(d, shape, h):
    """Active inside any of 40 spheres; rho a sum of 8 narrow Gaussians; Phi = 0 on the boundary."""
    axes = [_centres(n, h) / (n * h) for n in shape]
    centres, radii = d.uniform((40, 3), 0.2, 0.8).cpu(), d.uniform((40,), 0.05, 0.2).cpu()
    mask = torch.zeros(shape, device="cuda", dtype=torch.bool)
    for c, r in zip(centres.tolist(), radii.tolist()):
        lo = [max(0, int((c[a] - r) * shape[a]) - 1) for a in range(3)]
        hi = [min(shape[a], int((c[a] + r) * shape[a]) + 2) for a in range(3)]
        s = [(axes[a][lo[a]:hi[a]] - c[a]).square() for a in range(3)]
        mask[lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] |= (
            s[0][:, None, None] + s[1][None, :, None] + s[2][None, None, :] < r * r)
    amp, g = d.normal((8,)), d.uniform((8, 3), 0.2, 0.8)
    e = [torch.exp(-(axes[a][None, :] - g[:, a:a + 1]).square() / (2 * 0.03 ** 2)) for a in range(3)]
    rho = torch.einsum("m,mk,mj,mi->kji", amp, *e).contiguous()
    return {"mask": mask.to(torch.int8), "rho": rho}


def _holes(d, shape, h):
    """The whole box minus balls of 0.5 to 4 cells, 20000 per 512^3 cells; rho ~ U[-1, 1]; Phi = 0 on the boundary."""
    n = max(1, int(round(20000 * math.prod(shape) / 512.0 ** 3)))
    size = torch.tensor(shape, device="cuda", dtype=torch.float64)
    c, r = d.uniform((n, 3)) * size, d.uniform((n,), 0.5, 4.0)
    base = torch.floor(c).to(torch.int64)
    mask = torch.ones(shape, device="cuda", dtype=torch.int8)
    o = torch.arange(-5, 6, device="cuda")
    offs = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(-1, 3)
    for part in range(0, n, 5000):
        cell = base[part:part + 5000, None, :] + offs[None]
        inside = (cell + 0.5 - c[part:part + 5000, None, :]).square().sum(-1) < r[part:part + 5000, None].square()
        inside &= ((cell >= 0) & (cell < size.to(torch.int64))).all(-1)
        k = cell[inside]
        mask[k[:, 0], k[:, 1], k[:, 2]] = 0
    return {"mask": mask, "rho": d.uniform(shape, -1.0, 1.0)}


def _blob(d, shape, h):
    """White noise smoothed over 8 cells and cut at its median; rho ~ U[-1, 1]; a smooth coarse potential around it."""
    f = torch.fft.rfftn(d.normal(shape))
    for a, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device="cuda") if a == 2 else torch.fft.fftfreq(n, device="cuda")
        f *= torch.exp(-0.5 * (2 * math.pi * 8.0 * k.double()).square()).reshape([-1 if b == a else 1 for b in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    mask = (f > f.flatten().median()).to(torch.int8)
    rho = d.uniform(shape, -1.0, 1.0)
    shape_c = [(n + 1) // 2 + 2 for n in shape]
    amp, phase = d.normal((6,)), d.uniform((6, 3), 0.0, 2 * math.pi)
    wave = 1 + torch.floor(3 * d.uniform((6, 3)))
    s = [torch.cos(2 * math.pi * wave[:, a:a + 1] * _centres(n, 1.0 / n)[None, :] + phase[:, a:a + 1])
         for a, n in enumerate(shape_c)]
    return {"mask": mask, "rho": rho, "phi_c": torch.einsum("m,mk,mj,mi->kji", amp, *s).contiguous()}


DOMAINS = {"ball": _ball, "union": _union, "holes": _holes, "blob": _blob}
ORIGIN = (-2, -2, -2)


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _patches(case, seed):
    """The patches of a batch: edges drawn from PATCH_EDGES, every patch a blob at one cell size."""
    rng = np.random.default_rng(4 + case["patches"])  # the sizes belong to the case, what is in them to the seed
    shapes = rng.choice(PATCH_EDGES, (case["patches"], 3)).tolist()
    return [_blob(_Draws(seed * 1009 + p), tuple(s), 1.0 / 512) for p, s in enumerate(shapes)]


def _norm_inputs(case, seed):
    shape, d = _shape(case), _Draws(seed)
    nz, ny, nx = shape
    w = _blob(d, shape, 1.0 / max(shape))
    faces = [None] * 3
    if case["faces"]:
        faces = [d.uniform(s, -1.0, 1.0) for s in ((nz, ny, nx + 1), (nz, ny + 1, nx), (nz + 1, ny, nx))]
    return {"mask": w["mask"], "rho": w["rho"], "phi": d.normal(shape), "faces": faces}


def _unet_channels(levels):
    """(inputs, outputs) of every convolution of the network with 16 base channels, in parameter order."""
    ch = [16 << l for l in range(levels)]
    down = [c for l in range(levels) for c in ((3 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l]))]
    return down + [c for l in range(levels - 1) for c in ((ch[l] + ch[l + 1], ch[l]), (ch[l], ch[l]))]


def _unet_inputs(case, seed):
    """He-normal weights, small biases, the three channels of a blob patch, and the loss gradient of a training's start:
    2 (pred - y) / sum(y^2) on the active cells for a smooth target y and a prediction near 0."""
    shape, d = _shape(case), _Draws(seed)
    w = _blob(d, shape, 1.0 / max(shape))
    act = w["mask"].double()
    smooth = F.interpolate(w["phi_c"][None, None], size=shape, mode="trilinear", align_corners=False)[0, 0]
    edge = act * (F.avg_pool3d(act[None, None], 3, 1, 1)[0, 0] < 0.99)
    x = torch.stack([act * w["rho"] / w["rho"].std(), 2 * act - 1, edge * smooth]).float().contiguous()
    parts = []
    for ci, co in _unet_channels(case["levels"]):
        parts += [d.normal((co * ci * 27,)) * math.sqrt(2.0 / (27 * ci)), 0.1 * d.normal((co,))]
    parts += [d.normal((16,)) * math.sqrt(1.0 / 16), 0.1 * d.normal((1,))]
    y = act * (1.0 + smooth)
    g = (-2.0 * y / y.square().sum()).float().contiguous()
    return {"params": torch.cat(parts), "x": x, "g": g}


# ---------------------------------------------------------------------------
# What a user's program keeps, and one pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        shape = _shape(case)
        h = 1.0 / max(shape)
        w = DOMAINS[case["domain"]](_Draws(seed), shape, h)
        H = B.Hierarchy(w["mask"], h, precision=int(case["mixed"]), inner_cycles=case["inner"],
                        n_cycles=case["n_cycles"])
        return {"case": case, **w, "H": H, "phi": torch.empty(shape, dtype=torch.float64, device="cuda")}
    if kind == "batch":
        ws = _patches(case, seed)
        batch = B.Batch([w["mask"] for w in ws], [1.0 / 512] * len(ws))
        return {"case": case, "patches": ws, "batch": batch, "phi": [torch.empty_like(w["rho"]) for w in ws]}
    if kind == "norm":
        return {"case": case, **_norm_inputs(case, seed), "out": torch.empty(1, dtype=torch.float64, device="cuda")}
    w = _unet_inputs(case, seed)
    net = B.UNet(case["levels"], 16, _shape(case))
    net.set_params(w["params"].cpu().numpy())
    return {"case": case, "x": w["x"], "g": w["g"], "net": net, "pred": torch.empty_like(w["g"])}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        H = state["H"]
        if case["rebuild"]:
            H.update_mask(state["mask"])
        H.set_rhs(state["rho"])
        bc = BOUNDARY[case["domain"]]
        if bc == "coarse":
            H.set_dirichlet_from_coarse(state["phi_c"], ORIGIN)
        else:
            H.set_dirichlet(*(state["faces"] if bc == "faces" else (None, None, None)))
        H.set_solution(None)
        H.hold = 0
        status, info = H.solve(TOLERANCE[case["domain"]], 200)
        H.get_solution(state["phi"])
        return {"phi": state["phi"], "status": status}
    if kind == "batch":
        batch = state["batch"]
        for p, w in enumerate(state["patches"]):
            patch = batch.patch(p)
            patch.set_rhs(w["rho"])
            patch.set_dirichlet_from_coarse(w["phi_c"], ORIGIN)
            patch.set_solution(None)
            patch.hold = 0
        status, infos = batch.solve(1e-8, 200)
        for p, phi in enumerate(state["phi"]):
            batch.patch(p).get_solution(phi)
        # outputs are written down one by one, at most 64 of them: the patches' potentials as one tensor
        return {"phi": torch.cat([phi.reshape(-1) for phi in state["phi"]]), "status": status}
    if kind == "norm":
        B.mg_residual_norm_noalloc(state["mask"], state["phi"], state["rho"], 1.0 / max(_shape(case)), state["out"],
                                   *state["faces"])
        return {"norm": state["out"]}
    net = state["net"]
    net.forward(state["x"], state["pred"])
    if kind == "unet_forward":
        return {"pred": state["pred"]}
    net.backward(state["g"])
    # FP32 gradients (the binding hands them out widened), as an optimiser of FP32 weights takes them
    return {"pred": state["pred"], "grads": net.get_grads().astype(np.float32)}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    """Inputs read and outputs written once.  Operations: for a solve or a norm one evaluation of the 7-point residual
    (the iterations in between are the method's choice); for the network its multiply-adds."""
    kind = case["kind"]
    if kind == "batch":
        shapes = np.random.default_rng(4 + case["patches"]).choice(PATCH_EDGES, (case["patches"], 3))
        v = int(shapes.prod(1).sum())
        return {"bytes": v * (1 + 8 + 8 + 1), "flops": 9 * v}
    v = case["nx"] * case["ny"] * case["nz"]
    if kind == "solve":
        return {"bytes": v * (1 + 8 + 8), "flops": 9 * v}
    if kind == "norm":
        return {"bytes": v * (1 + 8 + 8 + (24 if case["faces"] else 0)), "flops": 9 * v}
    channels = _unet_channels(case["levels"])
    levels = [i // 2 if i < 2 * case["levels"] else (i - 2 * case["levels"]) // 2 for i in range(len(channels))]
    flops = sum(2 * 27 * ci * co * (v >> (3 * l)) for (ci, co), l in zip(channels, levels))
    params = sum((27 * ci + 1) * co for ci, co in channels) + 17
    if kind == "unet_forward":
        return {"bytes": 16 * v + 2 * params, "flops": flops}
    return {"bytes": 20 * v + 6 * params, "flops": 3 * flops}


# ---------------------------------------------------------------------------
# The same results by plain torch in 64 bits
# ---------------------------------------------------------------------------

def _interpolate(n_coarse, o, points):
    """Linear interpolation matrix from coarse centres o + 2I + 1 to points, all in fine-cell units."""
    u = (points - o) * 0.5 - 0.5
    i = torch.floor(u).clamp(0, n_coarse - 2)
    m = torch.zeros(len(points), n_coarse, dtype=torch.float64, device="cuda")
    rows = torch.arange(len(points), device="cuda")
    m[rows, i.long()] = 1 - (u - i)
    m[rows, i.long() + 1] = u - i
    return m


def _coarse_faces(phi_c, shape):
    """The coarse potential at every face centre of the three face families (bx, by, bz)."""
    out = []
    for family in (2, 1, 0):
        ms = []
        for a in range(3):
            pts = _edges(shape[a], 1.0) if a == family else _centres(shape[a], 1.0)
            ms.append(_interpolate(phi_c.shape[a], ORIGIN[a], pts))
        out.append(torch.einsum("ak,bj,ci,kji->abc", *ms, phi_c))
    return out


def _neighbour(a, axis, step):
    """a shifted so that each cell holds its neighbour's value, 0 outside the box."""
    out = torch.zeros_like(a)
    n = a.shape[axis]
    out.narrow(axis, 0 if step > 0 else 1, n - 1).copy_(a.narrow(axis, 1 if step > 0 else 0, n - 1))
    return out


def _operator(mask, faces):
    """The diagonal of the modified Laplacian (ghost faces at half a cell) and twice the boundary values' sum."""
    act = (mask > 0).double()
    diag = torch.full_like(act, 6.0)
    bc = torch.zeros_like(act)
    for axis in range(3):
        n = act.shape[axis]
        for step in (-1, 1):
            ghost = 1.0 - _neighbour(act, axis, step)
            diag += ghost
            if faces is not None and faces[2 - axis] is not None:
                bc += 2.0 * ghost * faces[2 - axis].narrow(axis, 0 if step < 0 else 1, n)
    return act, diag, bc


def _neighbour_sum(v, out):
    out.zero_()
    for axis in range(3):
        n = v.shape[axis]
        out.narrow(axis, 0, n - 1).add_(v.narrow(axis, 1, n - 1))
        out.narrow(axis, 1, n - 1).add_(v.narrow(axis, 0, n - 1))
    return out


def _exact_solution(mask, rho, h, faces):
    """Conjugate gradients, preconditioned by the diagonal, until the residual is 1e-13 of the right-hand side's."""
    act, diag, bc = _operator(mask, faces)
    r = act * (bc - h * h * rho)  # of (diag - neighbours) phi = bc - h^2 rho
    phi, q = torch.zeros_like(r), torch.empty_like(r)
    inv = act / diag
    z = inv * r
    p = z.clone()
    rz = torch.dot(r.view(-1), z.view(-1))
    stop = 1e-13 * float(r.norm())
    for it in range(6000):
        _neighbour_sum(p, q).neg_().addcmul_(diag, p).mul_(act)
        alpha = rz / torch.dot(p.view(-1), q.view(-1))
        phi.addcmul_(alpha, p)
        r.addcmul_(-alpha, q)
        if it % 20 == 19 and float(r.norm()) <= stop:
            break
        torch.mul(inv, r, out=z)
        rz, old = torch.dot(r.view(-1), z.view(-1)), rz
        p.mul_(rz / old).add_(z)
    return phi


def _exact_unet(case, w):
    """The network in 64 bits on unrounded weights; the gradients of sum(g pred) in parameter order."""
    levels = case["levels"]
    params, at, train = [], 0, case["kind"] == "unet_train"
    for ci, co in _unet_channels(levels) + [(None, None)]:
        for shape in (((co, ci, 3, 3, 3), (co,)) if ci else ((1, 16, 1, 1, 1), (1,))):
            n = math.prod(shape)
            params.append(w["params"][at:at + n].reshape(shape).clone().requires_grad_(train))
            at += n

    def pair(i, t):
        for j in (i, i + 1):
            t = F.relu(F.conv3d(t, params[2 * j], params[2 * j + 1], padding=1))
        return t

    with torch.set_grad_enabled(train):
        t, skips = w["x"].double()[None], []
        for l in range(levels):
            t = pair(2 * l, F.avg_pool3d(t, 2) if l else t)
            skips.append(t)
        for l in range(levels - 2, -1, -1):
            t = pair(2 * levels + 2 * l, torch.cat([skips[l], F.interpolate(t, scale_factor=2, mode="nearest")], 1))
        pred = F.conv3d(t, params[-2], params[-1])[0, 0] * (w["x"][1] > 0)
        if not train:
            return {"pred": pred}
        grads = torch.autograd.grad((pred * w["g"].double()).sum(), params)
    return {"pred": pred.detach(), "grads": torch.cat([g.reshape(-1) for g in grads])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        shape = _shape(case)
        h = 1.0 / max(shape)
        w = DOMAINS[case["domain"]](_Draws(seed), shape, h)
        faces = _coarse_faces(w["phi_c"], shape) if "phi_c" in w else w.get("faces")
        return {"phi": _exact_solution(w["mask"], w["rho"], h, faces), "status": None}
    if kind == "batch":
        phis = [_exact_solution(w["mask"], w["rho"], 1.0 / 512, _coarse_faces(w["phi_c"], tuple(w["mask"].shape)))
                for w in _patches(case, seed)]
        return {"phi": torch.cat([p.reshape(-1) for p in phis]), "status": None}
    if kind == "norm":
        w = _norm_inputs(case, seed)
        h = 1.0 / max(_shape(case))
        act, diag, bc = _operator(w["mask"], w["faces"])
        phi = act * w["phi"]
        r = act * (_neighbour_sum(phi, torch.empty_like(phi)) - diag * phi + bc - h * h * w["rho"])
        return {"norm": r.norm().reshape(1) / (h * h)}
    return _exact_unet(case, _unet_inputs(case, seed))
