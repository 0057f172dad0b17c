"""The calls a user of the rasterizer makes, as measurable cases.

Sizes are those of the repository's own workloads (synth.py, bench.py, the tests): avatars of
2,000 to 100,000 Gaussians with 5 to 40 blendshapes, frames of 64 to 1,024 pixels a side (512 x 512
in training), batches of 1 to 64 frames of one or several avatars. Inputs follow the recipe of
synth.py (ellipsoidal head, log-scales N(log 3 mm, 0.3), opacity logits N(0, 1), weights N(0, 0.3),
cameras within 20 degrees), drawn on the GPU from the seed. Targets are smooth head-shaped
pictures in front of the frame's background, as a matted video has them.

A case's fields: kind (the entry point), n and k (Gaussians and blendshapes of the largest
avatar), avatars, frames, w and h (pixels; `mixed` scales them by 1/2, 1, 2 from frame group to
frame group), mask (the blended channels), bound (a tangent-space avatar on a deforming mesh),
tile and stage (the binning tile and the staging size an autotuner picks from), loss.
"""
import math
import random

import torch

from paper_2503_12886_gb300 import api, synth
from paper_2503_12886_gb300.autograd import rasterize
from paper_2503_12886_gb300.batching import GraphStep
from paper_2503_12886_gb300.optim import PAPER_DELTA_SCALE, PAPER_LR, Adam
from paper_2503_12886_gb300.rasterizer import DeviceBatch, DeviceBinding, DeviceModel, Renderer

# blended channels: mean + log-scale + colour, and mean + rotation + colour
MASKS = {"scale": (0, 1, 2, 7, 8, 9, 11, 12, 13), "rotation": (0, 1, 2, 3, 4, 5, 6, 11, 12, 13)}
RADII = (0.09, 0.12, 0.10)
NEAR = 0.2


def _case(name, kind, **kw):
    c = {"name": name, "kind": kind, "n": 60000, "k": 32, "avatars": 1, "frames": 1, "w": 512, "h": 512,
         "mixed": False, "mask": "scale", "bound": False, "tile": "16x16", "stage": 64, "loss": "l1"}
    c.update(kw)
    return c


def listed():
    return [
        # a small avatar drawn alone: a preview or thumbnail, where latency is everything
        _case("render_small", "render", n=10000, k=20, w=128, h=128),
        # animation: one frame of one avatar per call, as a viewer draws it
        _case("render_frame", "render"),
        # a server's batch: several resident avatars, frames of 256 to 1,024 pixels in one call
        _case("render_mixed", "render", n=100000, avatars=5, frames=15, mixed=True),
        # one training sample per step on a small frame, the host waiting for each loss
        _case("step_small", "step", n=10000, k=20, w=128, h=128),
        # training at odd sizes: few blendshapes, ragged frames, the tall tile, rotations blended
        _case("step_ragged", "step", n=35001, k=7, frames=3, w=499, h=377, mask="rotation", tile="8x32",
              loss="l2"),
        # the batch-parallel training step, replayed from its graph
        _case("train_batch", "graph", frames=16),
        # the paper's own setting: batches of 10, 20 blendshapes on position, rotation and colour
        _case("train_ten", "graph", k=20, frames=10, mask="rotation"),
        # avatars bound to a tracked mesh that deforms with every frame
        _case("train_tangent", "graph", frames=16, bound=True),
        # many avatars of different sizes and resolutions trained together: the largest batch
        _case("train_uneven", "graph", n=100000, avatars=8, frames=64, mixed=True),
        # differentiable rendering inside a user's own torch loss
        _case("autograd", "autograd", n=30000, k=16, frames=4, w=256, h=256),
        # colour initialisation of a new avatar from its first frames
        _case("color_init", "color", k=20, frames=10),
        # the optimiser's update of every base Gaussian and blendshape
        _case("adam", "adam"),
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["render", "render", "step", "step", "graph", "graph", "graph", "autograd", "color", "adam"])
    n, k = logu(2000, 100000), rng.randint(5, 40)
    avatars = rng.choice([1, 1, 1, 2, 3, 4])
    w = logu(64, 1024)
    h = max(64, min(1024, w if rng.random() < 0.5 else int(w * rng.uniform(0.6, 1.6))))
    # no more pixels than 16 frames of 640 x 640 and no more splats than 1,200,000
    frames = min(logu(1, 24), max(1, 16 * 640 * 640 // (w * h)), max(1, 1200000 // n))
    case = _case("", kind, n=n, k=k, avatars=min(avatars, frames), frames=frames, w=w, h=h,
                 mixed=frames > 2 and w <= 512 and h <= 512 and rng.random() < 0.25,
                 mask=rng.choice(["scale", "rotation"]), bound=kind != "adam" and rng.random() < 0.2,
                 tile=rng.choice(["16x16", "16x16", "8x32"]), stage=rng.choice([64, 64, 128, 256]),
                 loss=rng.choice(["l1", "l2"]))
    del case["name"]
    return case


# ------------------------------------------------------------------------------------------- sizes

def _avatar_sizes(case):
    a = case["avatars"]
    return [(max(64, int(case["n"] * (1.0 - 0.7 * j / max(1, a - 1)))), max(1, case["k"] - (case["k"] // 4) * (j % 3)))
            for j in range(a)]


def _frame_sizes(case):
    out = []
    for f in range(case["frames"]):
        s = (0.5, 1, 2)[(f // case["avatars"]) % 3] if case["mixed"] else 1
        out.append((f % case["avatars"], max(1, int(case["w"] * s)), max(1, int(case["h"] * s))))
    return out


def work(case):
    sizes, frames, A = _avatar_sizes(case), _frame_sizes(case), len(MASKS[case["mask"]])
    params = sum(4.0 * n * (14 + k * A) for n, k in sizes)
    if case["kind"] == "adam":  # parameter, moments: read and written; gradient: read
        return {"bytes": 7 * params, "flops": 14 * params / 4}
    used = {m for m, _, _ in frames}
    params = sum(4.0 * n * (14 + k * A) for m, (n, k) in enumerate(sizes) if m in used)
    pix = sum(w * h for _, w, h in frames)
    # blend 2 K A and projection about 450 operations per (frame, Gaussian); a splat of the usual
    # size blends at about 25 pixels of a 512 x 512 frame, about 30 operations each (70 backwards)
    splat = sum(sizes[m][0] * (2.0 * sizes[m][1] * A + 450) for m, _, _ in frames)
    pairs = sum(sizes[m][0] * (4.0 + 21.0 * (w / 512) * (h / 512)) for m, w, h in frames)
    flops = splat + 30 * pairs
    if case["kind"] == "render":
        return {"bytes": params + 20.0 * pix, "flops": flops}
    if case["kind"] == "color":
        return {"bytes": params + 12.0 * pix + sum(12.0 * n for n, _ in sizes), "flops": flops}
    return {"bytes": 2 * params + 24.0 * pix, "flops": flops + 2.5 * splat + 70 * pairs}


# ------------------------------------------------------------------------------------------ inputs

def _camera(w, h, yaw, pitch, bg):
    cy, sy, cp, sp = math.cos(yaw), math.sin(yaw), math.cos(pitch), math.sin(pitch)
    # the transpose of R_y(yaw) R_x(pitch), one metre from the origin
    view = [cy, 0.0, -sy, 0.0, sy * sp, cp, cy * sp, 0.0, sy * cp, -sp, cy * cp, 1.0]
    f = 150.0 * w / 128.0
    return view + [f, f, w / 2.0, h / 2.0, NEAR] + list(bg)


def _mesh(r, n_lat=48, n_lon=96, n_expr=10):
    """An ellipsoid head mesh with a latitude-longitude atlas and smooth normal displacements."""
    th = 0.06 * math.pi + 0.88 * math.pi * torch.arange(n_lat, dtype=torch.float64) / (n_lat - 1)
    ph = 2 * math.pi * torch.arange(n_lon + 1, dtype=torch.float64) / n_lon
    T, P = torch.meshgrid(th, ph, indexing="ij")
    pos = torch.stack([RADII[0] * T.sin() * P.cos(), RADII[1] * T.cos(), RADII[2] * T.sin() * P.sin()], -1).reshape(-1, 3)
    uv = torch.stack([P / (2 * math.pi), (T - th[0]) / (th[-1] - th[0])], -1).reshape(-1, 2)
    a = (torch.arange(n_lat - 1)[:, None] * (n_lon + 1) + torch.arange(n_lon)[None]).reshape(-1)
    b, c = a + 1, a + n_lon + 1
    faces = torch.stack([torch.stack([a, c, b], -1), torch.stack([b, c, c + 1], -1)], 1).reshape(-1, 3)
    nrm = pos / torch.tensor(RADII, dtype=torch.float64) ** 2
    nrm = nrm / nrm.norm(dim=1, keepdim=True)
    dv = []
    for _ in range(n_expr):
        d = torch.tensor([r.gauss(0, 1) for _ in range(3)], dtype=torch.float64)
        k = d / d.norm() * r.uniform(20, 60)
        dv.append(4e-3 * torch.cos(pos @ k + r.uniform(0, 2 * math.pi))[:, None] * nrm)
    return pos, faces.to(torch.int32), uv[faces].reshape(-1, 6).float(), torch.stack(dv)


def _inputs(case, seed):
    """Plain tensors on the GPU: avatars, frames, weights, cameras, targets."""
    dev, r = "cuda", random.Random(seed)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    rn = lambda *s: torch.randn(*s, device=dev, generator=g)  # noqa: E731
    ru = lambda *s: torch.rand(*s, device=dev, generator=g)  # noqa: E731
    chans = MASKS[case["mask"]]
    mesh = _mesh(r) if case["bound"] else None
    sd = torch.tensor([1e-3] * 3 + [1e-2] * 4 + [1e-3] * 3 + [0.0] + [0.05] * 3, device=dev)[list(chans)]
    avatars = []
    for n, k in _avatar_sizes(case):
        pad = max(4, (n + 3) // 4 * 4)
        g0 = torch.zeros(14, pad, device=dev)
        if mesh is None:  # means uniform in the head's ellipsoid
            d = rn(3, n)
            d = d / d.norm(dim=0) * ru(n) ** (1 / 3)
            g0[0:3, :n] = d * torch.tensor(RADII, device=dev)[:, None]
        else:             # offsets in the triangle's tangent space
            g0[0:3, :n] = rn(3, n) * torch.tensor([2e-3, 3e-3, 1e-3], device=dev)[:, None]
        q = rn(4, n)
        g0[3:7, :n] = q / q.norm(dim=0)
        g0[7:10, :n] = math.log(4e-3 if mesh else 3e-3) + 0.3 * rn(3, n)
        g0[10, :n] = rn(n)
        g0[11:14, :n] = ru(3, n)
        dg = torch.zeros(k, len(chans), pad, device=dev)
        dg[:, :, :n] = rn(k, len(chans), n) * sd[None, :, None]
        av = {"n": n, "k": k, "g0": g0, "dg": dg, "mesh": None}
        if mesh is not None:
            r1, r2 = ru(n).sqrt(), ru(n)
            bary = torch.zeros(3, pad, device=dev)
            bary[:, :n] = torch.stack([1 - r1, r1 * (1 - r2), r1 * r2])
            av["mesh"] = {"faces": mesh[1].to(dev), "face_uv": mesh[2].to(dev), "verts": mesh[0].shape[0],
                          "face_of": (ru(n) * mesh[1].shape[0]).to(torch.int32).clamp_(max=mesh[1].shape[0] - 1),
                          "bary": bary}
        avatars.append(av)
    frames, kmax = _frame_sizes(case), max(a["k"] for a in avatars)
    psi = 0.3 * rn(len(frames), kmax)
    fp, verts, targets = [], [], []
    for m, w, h in frames:
        psi[len(fp), avatars[m]["k"]:] = 0
        bg = [r.random() for _ in range(3)]
        j = math.radians(20.0)
        fp.append(_camera(w, h, r.uniform(-j, j), r.uniform(-j, j), bg))
        if mesh is not None:
            wts = torch.tensor([r.gauss(0, 1) for _ in range(mesh[3].shape[0])], dtype=torch.float64)
            verts.append((mesh[0] + torch.tensordot(wts, mesh[3], 1)).float().contiguous().to(dev))
        y = (torch.arange(h, device=dev) + 0.5 - h / 2)[:, None] / (RADII[1] * 150 * w / 128)
        x = (torch.arange(w, device=dev) + 0.5 - w / 2)[None] / (RADII[0] * 150 * w / 128)
        head = torch.nn.functional.interpolate(ru(1, 3, 8, 8), size=(h, w), mode="bilinear", align_corners=True)[0]
        targets.append(torch.where(x * x + y * y < 1, head, torch.tensor(bg, device=dev)[:, None, None]))
    return {"avatars": avatars, "frames": frames, "psi": psi, "fparams": torch.tensor(fp, dtype=torch.float32, device=dev),
            "verts": verts or [None] * len(frames), "targets": targets}


def prepare(case, seed):
    x = _inputs(case, seed)
    bits = sum(1 << c for c in MASKS[case["mask"]])
    tile = tuple(int(v) for v in case["tile"].split("x"))
    s = {"kind": case["kind"], "r": Renderer(0), "in": x}
    bind = [a["mesh"] and DeviceBinding(a["mesh"]["faces"], a["mesh"]["face_uv"], a["mesh"]["face_of"], a["mesh"]["bary"],
                                        a["mesh"]["verts"]) for a in x["avatars"]]
    if case["kind"] == "autograd":
        s["psi"] = x["psi"].requires_grad_()
        s["models"] = [(a["n"], a["k"], bits, a["g0"].requires_grad_(), a["dg"].requires_grad_()) for a in x["avatars"]]
        s["bind"], s["tile"], s["stage"] = bind, tile, case["stage"]
        return s
    models = [DeviceModel(a["n"], a["k"], bits, a["g0"], a["dg"], binding=b) for a, b in zip(x["avatars"], bind)]
    batch = synth.Batch([], [synth.Frame(m, w, h) for m, w, h in x["frames"]], x["psi"].cpu().numpy(),
                        x["fparams"].cpu().numpy(), x["psi"].shape[1])
    db = DeviceBatch(batch, "cuda", tile=tile, smem_batch=case["stage"], models=models,
                     grads=case["kind"] in ("step", "graph", "adam"))
    db.verts = x["verts"]
    s["db"] = db
    s["target"] = torch.cat([t.reshape(-1) for t in x["targets"]])
    kind = api.RGBA_LOSS_L1 if case["loss"] == "l1" else api.RGBA_LOSS_L2
    s["loss"] = kind
    s["img"] = torch.empty(3 * db.total_pix, device="cuda")
    if case["kind"] == "render":  # a viewer or server has rendered the avatar before
        s["r"].forward(db)
    elif case["kind"] == "step":
        s["r"].step(db, s["target"], kind, s["img"])
    elif case["kind"] == "color":
        s["r"].color_init(db, s["target"], [torch.zeros(m.n_pad, dtype=torch.uint8, device="cuda") for m in models])
    elif case["kind"] == "graph":
        s["graph"] = GraphStep(s["r"], db, s["target"], kind, s["img"])
    elif case["kind"] == "adam":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        for m in models:  # gradients of the size a training step leaves
            m.grad_g0.normal_(0, 1e-5, generator=g)
            m.grad_dg.normal_(0, 3e-6, generator=g)
        s["opt"] = Adam(s["r"], db)
    return s


# --------------------------------------------------------------------------------------------- run

def _grads(db):
    return {"psi": db.grad_psi, "g0": [m.grad_g0 for m in db.models], "dg": [m.grad_dg for m in db.models]}


def run(s):
    kind = s["kind"]
    if kind == "render":
        img, T, n = s["r"].forward(s["db"])
        return {"img": img, "T": T, "n": n}
    if kind == "step":
        out = s["r"].step(s["db"], s["target"], s["loss"], s["img"])
        return {"loss": out.loss, "pairs": out.pairs, "img": s["img"], "grad": _grads(s["db"])}
    if kind == "graph":
        loss, pairs = s["graph"].replay()
        return {"loss": loss, "pairs": pairs, "img": s["img"], "grad": _grads(s["db"])}
    if kind == "color":
        done = [torch.zeros(m.n_pad, dtype=torch.uint8, device="cuda") for m in s["db"].models]
        pairs = s["r"].color_init(s["db"], s["target"], done)
        return {"pairs": pairs, "done": done, "g0": [m.g0 for m in s["db"].models]}
    if kind == "adam":
        s["opt"].step()
        return {"p": [[m.g0, m.dg] for m in s["db"].models], "m": s["opt"].m, "v": s["opt"].v}
    x = s["in"]
    imgs = rasterize(s["r"], x["frames"], s["psi"], x["fparams"], s["models"], s["tile"], s["stage"], s["bind"], x["verts"])
    loss = sum(((i - t) ** 2).mean() for i, t in zip(imgs, x["targets"])) / len(imgs)
    leaves = [s["psi"]] + [m[3] for m in s["models"]] + [m[4] for m in s["models"]]
    gr, a = torch.autograd.grad(loss, leaves), len(s["models"])
    return {"loss": loss, "img": torch.cat([i.reshape(-1) for i in imgs]),
            "grad": {"psi": gr[0], "g0": list(gr[1: 1 + a]), "dg": list(gr[1 + a:])}}


# ------------------------------------------------------------------------- the same in 64-bit torch

def _tangent(av, verts):
    """Per Gaussian the frame [T B N] and the surface point of its triangle."""
    me, n = av["mesh"], av["n"]
    f = me["face_of"].long()
    v0, v1, v2 = (verts.double()[me["faces"].long()[f, c]] for c in range(3))
    uv = me["face_uv"].double()[f].reshape(-1, 3, 2)
    e1, e2, d1, d2 = v1 - v0, v2 - v0, uv[:, 1] - uv[:, 0], uv[:, 2] - uv[:, 0]
    det = (d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0])[:, None]
    t = (d2[:, 1:] * e1 - d1[:, 1:] * e2) / det
    b = (d1[:, :1] * e2 - d2[:, :1] * e1) / det
    nn = torch.linalg.cross(e1, e2)
    w = me["bary"][:, :n].double()[:, :, None]
    return torch.stack([t, b, nn / nn.norm(dim=1, keepdim=True)], -1), w[0] * v0 + w[1] * v1 + w[2] * v2


def _project(v, fp, w, h, tangent, tile):
    """Blended channels [14][n] -> per splat (u, v, conic, opacity, colour), depth and tile rectangle."""
    V = fp[:12].reshape(3, 4)
    x, q, s = v[0:3].t(), v[3:7] / v[3:7].norm(dim=0), v[7:10].exp()
    qw, qx, qy, qz = q
    R = torch.stack([1 - 2 * (qy * qy + qz * qz), 2 * (qx * qy - qw * qz), 2 * (qx * qz + qw * qy),
                     2 * (qx * qy + qw * qz), 1 - 2 * (qx * qx + qz * qz), 2 * (qy * qz - qw * qx),
                     2 * (qx * qz - qw * qy), 2 * (qy * qz + qw * qx), 1 - 2 * (qx * qx + qy * qy)], -1).reshape(-1, 3, 3)
    M = R * s.t()[:, None, :]
    if tangent is not None:
        x, M = (tangent[0] @ x[:, :, None])[:, :, 0] + tangent[1], tangent[0] @ M
    p, M = x @ V[:, :3].t() + V[:, 3], V[:, :3] @ M
    fx, fy, z = fp[12], fp[13], p[:, 2]
    lx, ly = 1.3 * 0.5 * w / fx, 1.3 * 0.5 * h / fy
    rx, ry, zero = (p[:, 0] / z).clamp(-lx, lx), (p[:, 1] / z).clamp(-ly, ly), torch.zeros_like(z)
    J = torch.stack([fx / z, zero, -fx * rx / z, zero, fy / z, -fy * ry / z], -1).reshape(-1, 2, 3)
    K = J @ M
    S = K @ K.transpose(1, 2)
    A, B, C = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = A * C - B * B
    mid = 0.5 * (A + C)
    rad = (3 * (mid + (mid * mid - det).clamp(min=0.1).sqrt()).sqrt()).ceil()
    u, vv = fx * p[:, 0] / z + fp[14], fy * p[:, 1] / z + fp[15]
    tw, th = tile
    tx, ty = -(-w // tw), -(-h // th)
    rect = torch.stack([((u - rad) / tw).floor().clamp(0, tx), ((vv - rad) / th).floor().clamp(0, ty),
                        ((u + rad + tw - 1) / tw).floor().clamp(0, tx), ((vv + rad + th - 1) / th).floor().clamp(0, ty)], -1)
    kept = (z > fp[16]) & (det > 0) & (rect[:, 2] > rect[:, 0]) & (rect[:, 3] > rect[:, 1])
    splat = torch.stack([u, vv, C / det, -B / det, A / det, torch.sigmoid(v[10]), v[11], v[12], v[13]])
    return splat, z.detach(), rect.detach() * kept[:, None]


def _composite(P, px, py):
    """Weights [L][pixels] of the depth-ordered splats P [9][L] and the remaining transmittance."""
    dx, dy = px[None] - P[0][:, None], py[None] - P[1][:, None]
    power = -0.5 * (P[2][:, None] * dx * dx + P[4][:, None] * dy * dy) - P[3][:, None] * dx * dy
    alpha = (P[5][:, None] * power.exp()).clamp(max=0.99)
    alpha = torch.where((power <= 0) & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
    live = torch.cumprod(1 - alpha.detach(), 0) >= 1e-4
    alpha = torch.where(live, alpha, torch.zeros_like(alpha))
    cum = torch.cumprod(1 - alpha, 0)
    return alpha * torch.cat([torch.ones_like(cum[:1]), cum[:-1]]), cum[-1]


def exact(case, seed):
    frames, kind = _frame_sizes(case), case["kind"]
    x, chans = _inputs(case, seed), list(MASKS[case["mask"]])
    if kind == "adam":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        p, ms, vs = [], [], []
        for a in x["avatars"]:
            g0 = torch.empty_like(a["g0"]).normal_(0, 1e-5, generator=g).double()
            dg = torch.empty_like(a["dg"]).normal_(0, 3e-6, generator=g).double()
            b1, b2, eps = (float(torch.tensor(v, dtype=torch.float32)) for v in (0.9, 0.999, 1e-8))
            lr = torch.tensor(PAPER_LR, device="cuda").double()[:, None]
            lrd = torch.tensor([l * q for l, q in zip(PAPER_LR, PAPER_DELTA_SCALE)], device="cuda").double()[chans][None, :, None]
            p.append([a["g0"].double() - lr * g0 / (g0.abs() + eps), a["dg"].double() - lrd * dg / (dg.abs() + eps)])
            ms.append([(1 - b1) * g0, (1 - b1) * dg])
            vs.append([(1 - b2) * g0 * g0, (1 - b2) * dg * dg])
        return {"p": p, "m": ms, "v": vs}
    # about 4 ms a tile forwards and 12 ms with gradients: within some twenty seconds
    area = sum((w / 512) * (h / 512) + 0.2 for _, w, h in frames)
    if area > (40 if kind in ("render", "color") else 20):
        return None
    train = kind in ("step", "graph", "autograd")
    tw, th = (int(v) for v in case["tile"].split("x"))
    psi = x["psi"].double().requires_grad_(train)
    G = [a["g0"][:, : a["n"]].double().requires_grad_(train) for a in x["avatars"]]
    D = [a["dg"][:, :, : a["n"]].double().requires_grad_(train) for a in x["avatars"]]
    W = [torch.zeros(4, a["n"], dtype=torch.float64, device="cuda") for a in x["avatars"]]
    imgs, Ts, loss = [], [], 0.0
    for b, (m, w, h) in enumerate(frames):
        av, fp = x["avatars"][m], x["fparams"][b].double()
        with torch.set_grad_enabled(train):
            v = G[m].index_add(0, torch.tensor(chans, device="cuda"), torch.einsum("k,kan->an", psi[b, : av["k"]], D[m]))
            tan = _tangent(av, x["verts"][b]) if av["mesh"] else None
            splat, z, rect = _project(v, fp, w, h, tan, (tw, th))
        order = torch.argsort(z, stable=True)
        rect = rect[order].long()
        leaf = splat.detach()
        grad = torch.zeros_like(leaf)
        img = fp[17:20][:, None, None].expand(3, h, w).clone()
        T = torch.ones(h, w, dtype=torch.float64, device="cuda")
        tgt = x["targets"][b].double()
        scale = 1.0 / (3.0 * w * h * len(frames))
        for ty in range(int(rect[:, 1].min()), int(rect[:, 3].max())):
            row = ((rect[:, 1] <= ty) & (ty < rect[:, 3])).nonzero()[:, 0]
            rr = rect[row]
            for tx in range(-(-w // tw)):
                idx = order[row[(rr[:, 0] <= tx) & (tx < rr[:, 2])]]
                if not idx.numel():
                    continue
                ys = torch.arange(ty * th, min(h, ty * th + th), device="cuda")
                xs = torch.arange(tx * tw, min(w, tx * tw + tw), device="cuda")
                py, px = (t.reshape(-1) for t in torch.meshgrid(ys, xs, indexing="ij"))
                at = (slice(None), py, px)
                with torch.set_grad_enabled(train):
                    P = leaf[:, idx].requires_grad_(train)
                    wt, Tf = _composite(P, px + 0.5, py + 0.5)
                    c = P[6:9] @ wt + Tf * fp[17:20][:, None]
                    if train:
                        d = c - tgt[at]
                        part = scale * (d.abs().sum() if case["loss"] == "l1" and kind != "autograd" else
                                        (d * d).sum() * (1.0 if kind == "autograd" else 0.5))
                        grad.index_add_(1, idx, torch.autograd.grad(part, P)[0])
                img[at], T[py, px] = c.detach(), Tf.detach()
                if kind == "color":
                    W[m].index_add_(1, idx, torch.cat([wt.sum(1)[None], tgt[at] @ wt.t()]))
        if train:
            splat.backward(grad)
            d = img - tgt
            loss += scale * float(d.abs().sum() if case["loss"] == "l1" and kind != "autograd" else
                                  (d * d).sum() * (1.0 if kind == "autograd" else 0.5))
        imgs.append(img.reshape(-1))
        Ts.append(T.reshape(-1))
    if kind == "render":
        return {"img": torch.cat(imgs), "T": torch.cat(Ts), "n": None}
    if kind == "color":
        for a, s in zip(x["avatars"], W):
            ok = s[0] > 0.1
            a["g0"] = a["g0"].double()
            a["g0"][11:14, : a["n"]] = torch.where(ok, s[1:] / s[0].clamp(min=1e-30), a["g0"][11:14, : a["n"]])
        return {"pairs": None, "done": None, "g0": [a["g0"] for a in x["avatars"]]}
    fill = lambda t, like: torch.nn.functional.pad(t, (0, like.shape[-1] - t.shape[-1]))  # noqa: E731
    out = {"loss": loss, "img": torch.cat(imgs),
           "grad": {"psi": psi.grad, "g0": [fill(t.grad if t.grad is not None else torch.zeros_like(t), a["g0"]) for t, a in zip(G, x["avatars"])],
                    "dg": [fill(t.grad if t.grad is not None else torch.zeros_like(t), a["dg"]) for t, a in zip(D, x["avatars"])]}}
    if kind != "autograd":
        out["pairs"] = None
    return out
