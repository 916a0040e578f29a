"""Timed workloads of the renderer, as its users run it.

Every case goes through the package's public entry points (``render``,
``BatchRenderer``, ``ScanConverter``, ``hu_to_z``) with the defaults a user
gets.  Sizes are those of the package's own named workloads and of its
benchmark, and ``draw`` spreads further cases over the ranges these stand
for.  ``exact`` restates the method in plain 64-bit torch.

Volumes are seeded synthetic tissue: a smooth impedance field with lesions
and texture, and, where a case says ``bone``, a thin 7.8 MRayl shell.  The
literal reading of Eq. 1 (``mode`` 0, the default) has poles behind bone,
where rows are ill-posed and users drop them; so soft tissue is rendered with
mode 0; volumes with bone and the lossless depth-gain reading with the signed
coefficients (``mode`` 1).  So are gradients through BF16 volumes, whose
rounding makes many neighbouring voxels equal: |Z2 - Z1| has no derivative
there.  Every output of a case is then well-posed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_06768_gb300 import binding as B
from paper_2508_06768_gb300.inputs import Fan, Params
from paper_2508_06768_gb300.render import BatchRenderer, ScanConverter, render

# ------------------------------------------------------------------ the cases


def _fan_case(name, shape, spacing, rays, rows, depth, fov, f_mhz, grad, **kw):
    c = {"name": name, "kind": "fan", "nx": shape[0], "ny": shape[1], "nz": shape[2], "spacing": spacing,
         "rays": rays, "rows": rows, "depth": depth, "fov": fov, "f_mhz": f_mhz, "grad": grad, "bf16": False,
         "bone": False, "texture": 0.01, "refine": 0, "atten": 0}
    c.update(kw)
    return c


def _batch_case(name, shape, spacing, poses, rays, rows, step_mm, f_mhz, grad, **kw):
    c = {"name": name, "kind": "batch", "nx": shape[0], "ny": shape[1], "nz": shape[2], "spacing": spacing,
         "poses": poses, "rays_lo": rays[0], "rays_hi": rays[1], "rows_lo": rows[0], "rows_hi": rows[1],
         "step_mm": step_mm, "fov": 60.0, "f_mhz": f_mhz, "grad": grad, "bf16": False, "bone": False,
         "texture": 0.0, "refine": 0, "atten": 0}
    c.update(kw)
    return c


def listed():
    small, brain = (64, 64, 64), (256, 256, 192)
    return [
        # an interactive preview: one small frame, nothing else in flight
        _fan_case("frame_small", small, 1.0, 64, 256, 60.0, 60.0, 5.0, "none"),
        # one step of pose registration: a frame and its 6-DoF gradient
        _fan_case("register_step", small, 1.0, 64, 256, 60.0, 60.0, 5.0, "pose", bone=True),
        # one step of fitting a small volume: frame, volume and pose gradients
        _fan_case("fit_small", small, 1.0, 64, 256, 60.0, 60.0, 5.0, "both"),
        # a full-size frame of a brain volume, rendered once
        _fan_case("frame_brain", brain, 1.0, 256, 1024, 120.0, 70.0, 7.0, "none", bone=True),
        # the same frame with odd sizes inside a reconstruction loop
        _fan_case("fit_brain", brain, 1.0, 251, 1021, 120.0, 70.0, 7.0, "both", bone=True, texture=0.0),
        # reconstruction from a handful of small odd frames, depth-gain attenuation
        _batch_case("fit_few_odd", (48, 44, 40), 1.0, 9, (17, 70), (90, 333), 0.12, 5.0, True, bone=True, atten=1),
        # a freehand sweep of equal frames rendered for display from a BF16 volume
        _batch_case("sweep_serve", (256, 256, 256), 1.0, 100, (192, 192), (1000, 1000), 0.1, 5.0, False, bf16=True,
                    texture=0.01),
        # many uneven frames and all gradients: the training step
        _batch_case("fit_batch", (256, 256, 256), 1.0, 512, (64, 512), (256, 2048), 0.1, 5.0, True, bone=True),
        # high-resolution BF16 volume, deep frames: images with the refined solve
        # (at this texture the solve's conditioning gets low enough at depth
        # that some rays need the refined pass, and none meets a pole)
        _batch_case("fine_refined", (512, 512, 512), 0.5, 64, (1024, 1024), (4096, 4096), 0.05, 7.0, False,
                    bf16=True, refine=1, texture=0.052),
        # the same volume and frames inside a reconstruction loop
        _batch_case("fit_fine_bf16", (512, 512, 512), 0.5, 64, (1024, 1024), (4096, 4096), 0.05, 7.0, True,
                    bf16=True, bone=True, texture=0.02),
        # polar frames to display images, and the gradient through that step
        {"name": "scan_convert", "kind": "scan", "count": 64, "rays": 256, "rows": 1024, "width": 1024,
         "height": 1024, "depth": 120.0, "fov": 70.0, "grad": True},
        # a CT volume turned into impedance before rendering
        {"name": "ct_volume", "kind": "hu", "n": 256 ** 3, "points": 7, "bf16": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case, its sizes spread over the ranges of the listed ones."""
    kind = rng.choice(("fan", "fan", "fan", "batch", "batch", "batch", "scan", "hu"))
    if kind == "hu":
        return {"kind": "hu", "n": _log_int(rng, 64 ** 3, 256 ** 3), "points": rng.randint(2, 40),
                "bf16": rng.random() < 0.5}
    if kind == "scan":
        return {"kind": "scan", "count": _log_int(rng, 1, 64), "rays": _log_int(rng, 64, 256),
                "rows": _log_int(rng, 256, 1024), "width": _log_int(rng, 256, 1024),
                "height": _log_int(rng, 256, 1024), "depth": 120.0, "fov": rng.uniform(40.0, 90.0),
                "grad": rng.random() < 0.5}
    bone = rng.random() < 0.5
    shape = tuple(_log_int(rng, 40, 256) for _ in range(3))
    kw = {"bone": bone, "bf16": rng.random() < 0.3, "texture": 0.0 if bone else rng.choice((0.0, 0.01)),
          "atten": int(rng.random() < 0.2)}
    if kind == "fan":
        rows = _log_int(rng, 200, 2048)
        c = _fan_case("", shape, 1.0, _log_int(rng, 48, 512), rows, round(rng.uniform(0.06, 0.15) * rows, 3),
                      rng.uniform(40.0, 80.0), rng.uniform(3.0, 8.0), rng.choice(("none", "pose", "both")), **kw)
    else:
        poses = _log_int(rng, 2, 256)
        rays = sorted((_log_int(rng, 17, 512), _log_int(rng, 17, 512)))
        rows = sorted((_log_int(rng, 90, 2048), _log_int(rng, 90, 2048)))
        c = _batch_case("", shape, 1.0, poses, rays, rows, round(rng.uniform(0.08, 0.12), 4), rng.uniform(3.0, 8.0),
                        rng.random() < 0.6, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _volume(case, seed, dev):
    """Seeded tissue volume [nz][ny][nx] (MRayl), float32 or bfloat16."""
    g = _generator(seed, dev)
    h = float(case["spacing"])
    shape = (case["nz"], case["ny"], case["nx"])
    ext = [(n - 1) * h for n in shape]
    # smooth field over 24 mm cells and two finer octaves, 1.45 to 1.65 MRayl
    v = torch.zeros((1, 1) + shape, device=dev)
    for o in range(3):
        cells = [max(2, math.ceil(e / (24.0 / 2 ** o)) + 1) for e in ext]
        lattice = torch.randn((1, 1, *cells), generator=g, device=dev) * 0.5 ** o
        v += torch.nn.functional.interpolate(lattice, size=shape, mode="trilinear", align_corners=True)
    v = v[0, 0]
    lo, hi = v.min(), v.max()
    v = 1.45 + 0.20 * (v - lo) / (hi - lo)
    z, y, x = (torch.arange(n, device=dev, dtype=torch.float32) * h for n in shape)

    def level(c, a):
        return (((z - c[0]) / a[0]) ** 2)[:, None, None] + (((y - c[1]) / a[1]) ** 2)[None, :, None] + \
            (((x - c[2]) / a[2]) ** 2)[None, None, :]

    r = np.random.default_rng(seed)
    for _ in range(6):      # lesions at +-5 %
        c = [0.5 * e + r.uniform(-0.25, 0.25) * e for e in ext]
        inside = level(c, [r.uniform(0.04, 0.09) * e for e in ext]) <= 1.0
        v = torch.where(inside, v * (1.0 + float(r.choice((-0.05, 0.05)))), v)
    if case["bone"]:        # a thin closed shell
        c, outer = [0.5 * e for e in ext], [0.45 * e for e in ext]
        shell = (level(c, outer) <= 1.0) & (level(c, [max(o - 1.5, 0.5) for o in outer]) > 1.0)
        v = torch.where(shell, 7.8, v)
    if case["texture"]:
        v = v + float(case["texture"]) * torch.randn(shape, generator=g, device=dev)
    return v.to(torch.bfloat16 if case["bf16"] else torch.float32).contiguous()


def _params(case, seed):
    fit16 = case["bf16"] and case["grad"] not in (False, "none")
    return Params(seed=int(seed), mode=1 if case["bone"] or case["atten"] or fit16 else 0, refine=case["refine"],
                  atten=case["atten"])


def _poses(case, seed):
    """Seeded probe poses (float32 [P][6]): one near the top face looking
    down, or many on the upper hemisphere looking at the centre."""
    r = np.random.default_rng([int(seed), 1])
    h = case["spacing"]
    ext = np.array([(case[k] - 1) * h for k in ("nx", "ny", "nz")])
    if case["kind"] == "fan":
        p = np.array([[0.5 * ext[0], 0.5 * ext[1], 0.0, 0.0, 0.0, 0.0]])
        p[:, :3] += r.uniform(-2.0, 2.0, 3)
        p[:, 3:] += np.deg2rad(r.uniform(-3.0, 3.0, 3))
        return p.astype(np.float32)
    out = np.zeros((case["poses"], 6), dtype=np.float32)
    rad = 0.45 * ext.max()
    for i in range(case["poses"]):
        d = r.normal(size=3)
        d /= np.linalg.norm(d)
        d[2] = -abs(d[2])
        ax = -d
        u = np.cross([1.0, 0.0, 0.0] if abs(ax[0]) < 0.9 else [0.0, 1.0, 0.0], ax)
        u /= np.linalg.norm(u)
        w = np.cross(ax, u)
        roll = r.uniform(0.0, 2.0 * math.pi)
        xr = math.cos(roll) * u + math.sin(roll) * w
        yr = np.cross(ax, xr)
        R = np.stack([xr, yr, ax], axis=1)
        out[i, :3] = 0.5 * ext + rad * d
        out[i, 3:] = (math.atan2(R[2, 1], R[2, 2]), -math.asin(max(-1.0, min(1.0, R[2, 0]))),
                      math.atan2(R[1, 0], R[0, 0]))
    return out


def _fans(case):
    """(rays, rows, depth) of every pose: fixed by the case, whatever the seed."""
    if case["kind"] == "fan":
        return [(case["rays"], case["rows"], case["depth"])]
    r = np.random.default_rng(case["poses"])
    out = []
    for _ in range(case["poses"]):
        n = int(r.integers(case["rays_lo"], case["rays_hi"] + 1))
        s = int(r.integers(case["rows_lo"], case["rows_hi"] + 1))
        out.append((n, s, s * case["step_mm"]))
    return out


def _fan_objects(case):
    return [Fan(n, s, math.radians(case["fov"]), d, case["f_mhz"], 0.5) for n, s, d in _fans(case)]


def _cotangent(case, seed, dev):
    """dL/dimage of a user's loss: seeded normal weights."""
    n = sum(a * b for a, b, _ in _fans(case))
    return torch.randn(n, generator=_generator(seed + 1000003, dev), device=dev)


def _scan_input(case, seed, dev):
    g = _generator(seed, dev)
    img = torch.randn((case["count"], case["rays"], case["rows"]), generator=g, device=dev)
    cot = torch.randn((case["count"], case["height"], case["width"]), generator=g, device=dev)
    return img, cot


def _hu_input(case, seed, dev):
    g = _generator(seed, dev)
    hu = (torch.randn(case["n"], generator=g, device=dev) * 300.0 + 40.0).clamp(-1024, 3071).to(torch.int16)
    pts = np.round(np.linspace(-1000, 2000, case["points"]))
    z = np.linspace(0.4, 7.8, case["points"]) ** 1.2
    return hu, pts, z


def prepare(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "hu":
        hu, pts, z = _hu_input(case, seed, dev)
        return {"case": case, "hu": hu, "pts": pts, "z": z}
    if kind == "scan":
        img, cot = _scan_input(case, seed, dev)
        fan = Fan(case["rays"], case["rows"], math.radians(case["fov"]), case["depth"])
        return {"case": case, "img": img.requires_grad_(case["grad"]), "cot": cot,
                "conv": ScanConverter(fan, case["width"], case["height"], device=dev)}
    s = {"case": case, "vol": _volume(case, seed, dev), "spacing": (case["spacing"],) * 3,
         "params": _params(case, seed), "poses": torch.from_numpy(_poses(case, seed)).to(dev)}
    if case["grad"] not in (False, "none"):
        s["cot"] = _cotangent(case, seed, dev)
    if kind == "fan":
        s["fan"] = _fan_objects(case)[0]
        s["pose"] = s["poses"][0].clone()
        if case["grad"] != "none":
            s["pose"].requires_grad_()
            s["cot"] = s["cot"].view(case["rays"], case["rows"])
        if case["grad"] == "both":
            s["vol"].requires_grad_()
    else:
        s["renderer"] = BatchRenderer(s["vol"], s["spacing"], (0.0, 0.0, 0.0), _fan_objects(case), s["params"],
                                      with_bwd=case["grad"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "hu":
        return {"z": B.hu_to_z(s["hu"], s["pts"], s["z"], dtype=torch.bfloat16 if case["bf16"] else torch.float32)}
    if kind == "scan":
        out = s["conv"](s["img"])
        if not case["grad"]:
            return {"display": out}
        return {"display": out.detach(), "grad": torch.autograd.grad(out, s["img"], s["cot"])[0]}
    if kind == "fan":
        img, valid = render(s["vol"], s["pose"], s["fan"], s["params"], spacing=s["spacing"])
        if case["grad"] == "none":
            return {"image": img, "valid": valid}
        wrt = [s["pose"], s["vol"]] if case["grad"] == "both" else [s["pose"]]
        grads = torch.autograd.grad(img, wrt, s["cot"])
        return {"image": img.detach(), "valid": valid, "grads": list(grads)}
    r = s["renderer"]
    if case["grad"]:
        r.run(s["poses"], s["cot"])
        return {"images": r.images, "valid": r.ray_valid, "grad_poses": r.grad_poses, "grad_vol": r.grad_vol}
    r.run(s["poses"])
    return {"images": r.images, "valid": r.ray_valid}


def work(case):
    kind = case["kind"]
    if kind == "hu":
        return {"bytes": case["n"] * (2 + (2 if case["bf16"] else 4)), "flops": 2.0 * case["n"]}
    if kind == "scan":
        polar, disp = case["count"] * case["rays"] * case["rows"], case["count"] * case["width"] * case["height"]
        passes = 2 if case["grad"] else 1
        return {"bytes": 4.0 * passes * (polar + disp), "flops": 8.0 * passes * disp}
    fans = _fans(case)
    n = sum(a * b for a, b, _ in fans)
    el = 2 if case["bf16"] else 4
    vox = case["nx"] * case["ny"] * case["nz"]
    # voxels the fans pass through: two layers around each fan's plane, at most all
    fov = math.radians(case["fov"])
    plane = sum(0.5 * fov * (d / case["spacing"]) ** 2 for _, _, d in fans)
    touched = min(vox, 2.0 * plane)
    # per sample: trilinear 20, coefficient and transfer 9, state 6, scan 2,
    # echo 7, speckle 58, blur 22; adjoint 57, its blur 22
    nbytes, flops = touched * el + 4.0 * n, 124.0 * n
    if case["grad"] not in (False, "none"):
        nbytes += 4.0 * n
        flops += (57.0 + 22.0 + 44.0) * n     # with the sampled gradient and pose terms
    if case["grad"] in (True, "both"):
        nbytes += vox * (el if kind == "fan" else 4)
        flops += 30.0 * n                      # scatter of dL/dZ to eight corners
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------ the method in 64 bits


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(m, a):
        lo, hi = (a & 0xFFFF) * m, (a >> 16) * m
        return (hi + (lo >> 16)) >> 16, (((hi & 0xFFFF) << 16) + lo) & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return torch.stack((c0, c1, c2, c3), dim=-1)


def _normals(words):
    s = (words & 255) + ((words >> 8) & 255) + ((words >> 16) & 255) + (words >> 24)
    return (s - 510).double() * (math.sqrt(3.0) / 256.0)


def _speckle(prm, pose, n, S, dev):
    key = int(prm.seed)
    k0, k1 = key & 0xFFFFFFFF, key >> 32
    ray = torch.arange(n, device=dev)[:, None]

    def words(group, stream):
        g = (group & 0xFFFFFFFF)[None, :].expand(n, -1)
        return _philox(g, ray.expand_as(g), torch.full_like(g, pose), torch.full_like(g, stream), k0, k1)

    L = prm.Lr
    groups = torch.arange(-1, (S + 3) // 4 + 1, device=dev)
    nu = _normals(words(groups, 0)).reshape(n, -1)                   # row k at column k + 4
    c = torch.nn.functional.pad(nu.cumsum(1), (1, 0))
    k = torch.arange(S, device=dev)
    n_r = (c[:, k + 4 + L + 1] - c[:, k + 4 - L]) / math.sqrt(2 * L + 1)
    band = (4 * k) // S
    idx = (k - (band * S + 3) // 4) >> (prm.gshift + band)
    cell = (band << 24) | idx
    grp, where = torch.unique(cell >> 2, return_inverse=True)
    n_g = _normals(words(grp, 1))[:, where, cell & 3]
    z = (k + 1).double() / S
    return (1.0 + prm.Ar * z ** prm.pr * n_r + prm.Ag * z ** prm.pg * n_g).clamp_min(0.0)


def _blurred(prm, y):
    n, S = y.shape
    W = math.ceil(3 * (prm.sigma0 + prm.sigma1))
    s = prm.sigma0 + prm.sigma1 * torch.arange(1, S + 1, device=y.device, dtype=torch.float64) / S
    yp = torch.nn.functional.pad(y, (0, 0, W, W))
    ones = torch.nn.functional.pad(torch.ones(n, 1, device=y.device, dtype=torch.float64), (0, 0, W, W))
    acc = norm = 0.0
    for m in range(-W, W + 1):
        w = torch.exp(-m * m / (2.0 * s * s))
        acc = acc + w * yp[W + m:W + m + n]
        norm = norm + w * ones[W + m:W + m + n]
    return acc / norm


def _rotation(r):
    (sx, sy, sz), (cx, cy, cz) = torch.sin(r).unbind(1), torch.cos(r).unbind(1)
    o, i = torch.zeros_like(sx), torch.ones_like(sx)
    mat = lambda *v: torch.stack(v, 1).view(-1, 3, 3)   # noqa: E731
    rx = mat(i, o, o, o, cx, -sx, o, sx, cx)
    ry = mat(cy, o, sy, o, i, o, -sy, o, cy)
    rz = mat(cz, -sz, o, sz, cz, o, o, o, i)
    return rz @ ry @ rx


def _cells(vol, pos):
    """Flat indices and corner weights of the trilinear cells at voxel
    coordinates pos [..., 3] (clamped), with the strictly-inside flags."""
    nz, ny, nx = vol.shape
    idx, frac, inside = [], [], []
    for a, n in enumerate((nx, ny, nz)):
        p = pos[..., a]
        q = p.clamp(0.0, n - 1.0)
        i = q.floor().clamp_max(n - 2.0)
        idx.append(i.long())
        frac.append(q - i)
        inside.append((p > 0.0) & (p < n - 1.0))
    return (idx[2] * ny + idx[1]) * nx + idx[0], frac, inside


def _corner_offsets(vol):
    nz, ny, nx = vol.shape
    return [(i, j, k, (k * ny + j) * nx + i) for k in (0, 1) for j in (0, 1) for i in (0, 1)]


def _weight(frac, i, j, k):
    fx, fy, fz = frac
    return (fx if i else 1.0 - fx) * (fy if j else 1.0 - fy) * (fz if k else 1.0 - fz)


def _exact_frames(case, seed):
    dev = _device()
    vol = _volume(case, seed, dev).double()
    flat = vol.reshape(-1)
    prm, fans = _params(case, seed), _fans(case)
    poses = torch.from_numpy(_poses(case, seed)).double().to(dev).requires_grad_()
    h = float(case["spacing"])
    S = max(f[1] for f in fans)
    # unit directions of all rays, differentiable in the poses
    R = _rotation(poses[:, 3:])
    half = 0.5 * math.radians(case["fov"])
    dirs, org, step, att = [], [], [], []
    for p, (n, s, d) in enumerate(fans):
        th = torch.linspace(-half, half, n, dtype=torch.float64, device=dev) if n > 1 else \
            torch.zeros(1, dtype=torch.float64, device=dev)
        dirs.append(torch.stack((torch.sin(th), torch.zeros_like(th), torch.cos(th)), 1) @ R[p].T)
        org.append(poses[p, :3].expand(n, 3))
        step.append(torch.full((n,), d / s, dtype=torch.float64, device=dev))
        att.append(torch.full((n,), 10.0 ** (-2.0 * 0.5 * case["f_mhz"] * (d / s / 10.0) / 20.0), dtype=torch.float64,
                              device=dev))
    dirs, org, step, att = torch.cat(dirs), torch.cat(org), torch.cat(step), torch.cat(att)
    n_rays = dirs.shape[0]
    k = torch.arange(S + 1, device=dev, dtype=torch.float64) + 0.5
    chunk = max(1, (1 << 22) // (S + 1))

    def positions(a, b):
        depth = k[None, :] * step[a:b, None]
        return (org[a:b, None, :] + depth[..., None] * dirs[a:b, None, :]).detach() / h, depth

    Z = torch.empty((n_rays, S + 1), dtype=torch.float64, device=dev)
    for a in range(0, n_rays, chunk):
        pos, _ = positions(a, a + chunk)
        base, frac, _ = _cells(vol, pos)
        z = 0.0
        for i, j, m, off in _corner_offsets(vol):
            z = z + _weight(frac, i, j, m) * flat[base + off]
        Z[a:a + chunk] = z
    grad = case["grad"] not in (False, "none")
    Z = Z.T.contiguous().requires_grad_(grad)          # [S + 1][rays]
    r = (Z[1:] - Z[:-1]) / (Z[1:] + Z[:-1])
    a2 = torch.ones_like(att) if case["atten"] else att
    if prm.mode == 0:
        r = r.abs()
        m00, m10 = a2 * (1.0 - 2.0 * r * r), -r
    else:
        m00, m10 = a2.expand_as(r), r
    x = a2 * r
    delta = a2 * (1.0 - r * r)
    b0, b1, D = torch.zeros_like(att), torch.ones_like(att), torch.ones_like(att)
    rows = []
    for xi, mi, ni, di in zip(x.unbind(0), m00.unbind(0), m10.unbind(0), delta.unbind(0)):
        q = b0 * xi + b1
        rows.append(xi * D / (b1 * q))
        b0, b1, D = b0 * mi + b1 * ni, q, D * di
    e = torch.stack(rows, 0)
    del rows
    images, j0 = [], 0
    for p, (n, s, d) in enumerate(fans):
        y = e[:s, j0:j0 + n].T
        if prm.speckle:
            y = y * _speckle(prm, p, n, s, dev)
        if prm.blur:
            y = _blurred(prm, y)
        if case["atten"]:
            y = y * att[j0] ** torch.arange(1, s + 1, device=dev, dtype=torch.float64)
        images.append(y.reshape(-1))
        j0 += n
    image = torch.cat(images)
    if not grad:
        return image, None, None
    (gZ,) = torch.autograd.grad(image, Z, _cotangent(case, seed, dev).double())
    image = image.detach()
    del e, images, r, m00, m10, x, delta
    gZ = gZ.T
    gvol = torch.zeros_like(flat)
    T, U = torch.zeros_like(dirs), torch.zeros_like(dirs)
    for a in range(0, n_rays, chunk):
        pos, depth = positions(a, a + chunk)
        base, frac, inside = _cells(vol, pos)
        g = gZ[a:a + chunk]
        dz = [0.0, 0.0, 0.0]
        for i, j, m, off in _corner_offsets(vol):
            at = base + off
            gvol.index_add_(0, at.reshape(-1), (g * _weight(frac, i, j, m)).reshape(-1))
            v = flat[at]
            fx, fy, fz = frac
            wx, wy, wz = (fx if i else 1.0 - fx), (fy if j else 1.0 - fy), (fz if m else 1.0 - fz)
            dz[0] = dz[0] + (v if i else -v) * wy * wz
            dz[1] = dz[1] + (v if j else -v) * wx * wz
            dz[2] = dz[2] + (v if m else -v) * wx * wy
        for c in range(3):
            gp = torch.where(inside[c], g * dz[c], 0.0) / h
            T[a:a + chunk, c] = gp.sum(1)
            U[a:a + chunk, c] = (gp * depth).sum(1)
    (gpose,) = torch.autograd.grad((org * T).sum() + (dirs * U).sum(), poses)
    return image, gpose, gvol.view(vol.shape)


def exact(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "hu":
        hu, pts, z = _hu_input(case, seed, dev)
        p, v = (torch.as_tensor(a, dtype=torch.float64, device=dev) for a in (pts, z))
        x = hu.double().clamp(p[0], p[-1])
        i = (torch.searchsorted(p, x, right=True) - 1).clamp(0, len(pts) - 2)
        return {"z": v[i] + (x - p[i]) * (v[i + 1] - v[i]) / (p[i + 1] - p[i])}
    if kind == "scan":
        return _exact_scan(case, seed, dev)
    image, gpose, gvol = _exact_frames(case, seed)
    if kind == "fan":
        out = {"image": image.view(case["rays"], case["rows"]), "valid": None}
        if case["grad"] != "none":
            out["grads"] = [gpose[0], gvol] if case["grad"] == "both" else [gpose[0]]
        return out
    out = {"images": image, "valid": None}
    if case["grad"]:
        out.update(grad_poses=gpose, grad_vol=gvol)
    return out


def _exact_scan(case, seed, dev):
    img, cot = _scan_input(case, seed, dev)
    n, S, W, H = case["rays"], case["rows"], case["width"], case["height"]
    fov, depth = math.radians(case["fov"]), case["depth"]
    half = depth * math.sin(0.5 * fov)
    px = -half + (torch.arange(W, device=dev, dtype=torch.float64) + 0.5) * (2.0 * half / W)
    pz = (torch.arange(H, device=dev, dtype=torch.float64) + 0.5) * (depth / H)
    z, x = torch.meshgrid(pz, px, indexing="ij")
    v = (torch.atan2(x, z) + 0.5 * fov) * (n - 1) / fov
    u = torch.sqrt(x * x + z * z) / (depth / S) - 1.0
    ok = (v >= 0) & (v <= n - 1) & (u >= 0) & (u <= S - 1)
    j, k = v.floor().clamp(0, n - 2).long(), u.floor().clamp(0, S - 2).long()
    fv, fu = v - j, u - k
    taps = [(dj, dk, torch.where(ok, (fv if dj else 1.0 - fv) * (fu if dk else 1.0 - fu), 0.0).reshape(-1),
             ((j + dj) * S + (k + dk)).reshape(-1)) for dj in (0, 1) for dk in (0, 1)]
    src = img.reshape(case["count"], -1)
    out = torch.zeros((case["count"], H * W), dtype=torch.float64, device=dev)
    for c in range(case["count"]):
        s = src[c].double()
        for _, _, w, at in taps:
            out[c] += w * s[at]
    res = {"display": out.view(case["count"], H, W)}
    if case["grad"]:
        g = torch.zeros((case["count"], n * S), dtype=torch.float64, device=dev)
        for c in range(case["count"]):
            for _, _, w, at in taps:
                g[c].index_add_(0, at, w * cot[c].reshape(-1).double())
        res["grad"] = g.view(case["count"], n, S)
    return res
