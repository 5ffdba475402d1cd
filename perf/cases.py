"""What a user of this library has it do, as measurable cases: frames of one
avatar to a 10,000-character crowd, host-to-host frames, contribution
statistics, training steps of the differentiable render and of the ranking
network.  Everything goes through ``paper_2501_17792_gb300.binding``.

``listed()`` names the cases, ``draw(rng)`` gives another one of the same
ranges, ``prepare(case, seed)`` makes its inputs and handles on the GPU,
``run(state)`` is one pass, ``work(case)`` the bytes and operations a pass
cannot do without, ``exact(case, seed)`` the pass's results in FP64 from plain
torch operations.
"""
import math

import numpy as np
import torch

from paper_2501_17792_gb300 import binding
from paper_2501_17792_gb300 import scene as S

# Capsule radius (m) of the body segment that ends in each joint.
RADIUS = (0.11, 0.09, 0.09, 0.13, 0.06, 0.06, 0.14, 0.045, 0.045, 0.15, 0.04, 0.04, 0.05, 0.06, 0.06, 0.10, 0.05,
          0.05, 0.045, 0.045, 0.04, 0.04, 0.04, 0.04)
# Levels of detail: (thresholds m, fractions, scale multipliers).
_F = (1.0, 0.25, 0.06)
LODS = {
    "full": ((), (1.0,), (1.0,)),
    # the distance bands of the benchmark crowd
    "paper": ((10.0, 30.0), _F, tuple(f ** -0.5 for f in _F)),
    # level sizes of the learned ranking at equal image quality
    "budget": ((10.0, 30.0), (1.0, 0.02, 0.0048), (1.0, 1.0, 1.0)),
}
FRAME = dict(kind="frame", templates=1, gauss=16384, sh=3, cols=1, rows=1, spacing=1.2, first=3.0, width=256,
             height=256, lod="full", store="fp32", skin="full", world_sh=False, host=False)


def listed():
    f = FRAME
    return [
        # one avatar in a small view, new pose per frame: the smallest call, all latency
        dict(f, name="avatar_16k_256", sh=0, first=2.5),
        # one full-size reconstructed avatar filling a 720p view
        dict(f, name="avatar_202k_720p", gauss=202738, width=1280, height=720),
        # a room of 100 characters of the middle template size
        dict(f, name="chars_100_12k_720p", gauss=12661, cols=10, rows=10, width=1280, height=720),
        # 5,000 characters of the smallest template size, one level of detail
        dict(f, name="chars_5000_3k_720p", gauss=3176, cols=50, rows=100, width=1280, height=720),
        # the benchmark crowd: 3,500 animated characters, three levels of detail
        dict(f, name="crowd_3500_1080p", templates=14, gauss=65536, cols=50, rows=70, width=1920, height=1080,
             lod="paper"),
        # the same with its inputs and its image in pinned host memory
        dict(f, name="crowd_3500_1080p_host", templates=14, gauss=65536, cols=50, rows=70, width=1920, height=1080,
             lod="paper", host=True),
        # the largest crowd and image: 10,000 characters at the ranked levels' sizes, 4K
        dict(f, name="crowd_10000_4k", templates=14, gauss=65536, cols=100, rows=100, width=3840, height=2160,
             lod="budget"),
        # ragged sizes with the other options: 16-bit storage, degree 2, means-only skinning, world-frame colour
        dict(f, name="crowd_609_bf16_odd", templates=5, gauss=7001, sh=2, cols=29, rows=21, width=1366, height=743,
             lod="paper", store="bf16", skin="means", world_sh=True),
        # contribution statistics of one training view of the ranking: 100 full-detail characters, 4K
        dict(f, name="contrib_100_4k", kind="contrib", templates=14, gauss=65536, cols=10, rows=10, first=10.0,
             spacing=2.0, width=3840, height=2160),
        # forward and backward of the differentiable render: the template-fitting step
        dict(f, name="train_64_65k_512", kind="train", gauss=65536, cols=8, rows=8, spacing=0.9, width=512, height=512),
        # the same for a small odd-sized fit
        dict(f, name="train_3_4k_odd", kind="train", gauss=4097, cols=3, rows=1, spacing=0.9, width=145, height=131),
        # one full-batch step of the ranking network over every (band, Gaussian) row
        dict(kind="mlp", name="mlp_train_2750k", rows=2752512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["contrib"] + ["train"] * 2 + ["mlp"])
    if kind == "mlp":
        return dict(kind="mlp", rows=_log(rng, 3000, 2752512))
    while True:
        c = dict(FRAME, kind=kind, templates=rng.choice([1, 1, 2, 5, 14]), gauss=_log(rng, 1000, 202738),
                 sh=rng.choice([0, 1, 2, 3, 3, 3]))
        if kind == "train":
            c.update(cols=rng.randint(1, 8), rows=rng.randint(1, 8), spacing=0.9, width=_log(rng, 96, 512))
            c["height"] = max(64, int(c["width"] * rng.uniform(0.6, 1.0)))
            c["gauss"] = min(c["gauss"], 65536)
            c["templates"] = 1
        else:
            n = _log(rng, 1, 10000 if kind == "frame" else 100)
            c["cols"] = max(1, int(math.sqrt(n) * rng.uniform(0.7, 1.3)))
            c["rows"] = max(1, n // c["cols"])
            c["width"] = _log(rng, 160, 3840)
            c["height"] = max(90, int(c["width"] * rng.uniform(0.5, 0.75)))
            if kind == "contrib":
                c.update(first=10.0, spacing=2.0)
            else:
                c["lod"] = rng.choice(["full", "paper", "paper", "budget"])
                c["store"] = rng.choice(["fp32", "fp32", "fp32", "bf16"])
                c["skin"] = rng.choice(["full", "full", "full", "means"])
                c["world_sh"] = rng.random() < 0.2
                c["host"] = rng.random() < 0.15
        most = {"frame": 12e6, "contrib": 5e6, "train": 3e6}[kind]
        if c["templates"] * c["gauss"] <= 917504 and _splats(c) <= most:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _camera(case):
    w, h = case["width"], case["height"]
    if case["kind"] == "train":
        return S.look_camera((0.0, 1.4, 0.0), 12.0, w, h)
    if case["cols"] * case["rows"] == 1:
        return S.look_camera((0.0, 0.95, 0.0), 0.0, w, h)
    return S.look_camera((0.0, 1.6, 0.0), 10.0, w, h)


def _grid(case):
    k = np.arange(case["cols"] * case["rows"])
    x = (k % case["cols"] - (case["cols"] - 1) / 2) * case["spacing"]
    return x, case["first"] + k // case["cols"] * case["spacing"]


def _splats(case):
    """Gaussian-instances in view, from the unjittered layout."""
    cam, (x, z) = _camera(case), _grid(case)
    seen = np.abs(x) <= z * case["width"] / (2 * cam.fx) + 1.0
    thr, frac, _ = LODS[case["lod"]]
    lvl = sum((np.hypot(x, z) >= t).astype(int) for t in thr) + np.zeros(len(x), int)
    return float((np.asarray(frac)[lvl] * case["gauss"] * seen).sum())


def _templates(case, g, dev):
    """Avatars on the GPU: Gaussians on the surface of a capsule body, top-4
    distance skinning weights, log-normal scales (mean 1 cm), random
    rotations, sigmoid-normal opacity, normal SH coefficients."""
    n, out = case["gauss"], []
    rest0 = S.make_template(0, 1, 0).rest_joints
    par = S.PARENTS
    radius = torch.tensor(RADIUS, device=dev)
    for _ in range(case["templates"]):
        rest = torch.from_numpy(rest0).to(dev) * (0.9 + 0.2 * torch.rand(1, generator=g, device=dev))
        a = rest[torch.from_numpy(np.maximum(par, 0)).long().to(dev)]
        b = rest + torch.tensor([0.0, 1e-3, 0.0], device=dev)
        axis = b - a
        length = axis.norm(dim=1)
        seg = torch.multinomial(length * radius + radius ** 2, n, replacement=True, generator=g)
        d = torch.randn((n, 3), generator=g, device=dev)
        t = torch.rand((n, 1), generator=g, device=dev)
        dir_ = axis[seg] / length[seg, None]
        side = d - (d * dir_).sum(1, keepdim=True) * dir_
        means = a[seg] + t * axis[seg] + radius[seg, None] * side / side.norm(dim=1, keepdim=True)
        near = ((means[:, None] - a) * axis).sum(2) / length ** 2
        dist = (means[:, None] - a - near.clamp(0, 1)[..., None] * axis).norm(dim=2)
        d4, idx = dist.topk(4, dim=1, largest=False)
        w = (d4 + 1e-3) ** -2
        q = torch.randn((n, 4), generator=g, device=dev)
        s = torch.exp(math.log(0.01) - 0.125 + 0.5 * torch.randn((n, 3), generator=g, device=dev))
        out.append(dict(
            means=means, scales=s, quats=q / q.norm(dim=1, keepdim=True),
            opacity=torch.sigmoid(torch.randn(n, generator=g, device=dev)),
            sh=0.3 * torch.randn((n, (case["sh"] + 1) ** 2, 3), generator=g, device=dev),
            skin_idx=idx.to(torch.uint8), skin_w=w / w.sum(1, keepdim=True), rest_joints=rest))
    return out


def _instances(case, g, dev):
    x, z = _grid(case)
    n = len(x)
    jit = 0.3 * (2 * torch.rand((n, 2), generator=g, device=dev) - 1) * (n > 1)
    yaw = 2 * math.pi * torch.rand(n, generator=g, device=dev)
    root = torch.zeros((n, 3, 4), device=dev)
    root[:, 0, 0] = root[:, 2, 2] = torch.cos(yaw)
    root[:, 0, 2], root[:, 2, 0] = torch.sin(yaw), -torch.sin(yaw)
    root[:, 1, 1] = 1.0
    root[:, 0, 3] = torch.from_numpy(x).float().to(dev) + jit[:, 0]
    root[:, 2, 3] = torch.from_numpy(z).float().to(dev) + jit[:, 1]
    tid = torch.randint(0, case["templates"], (n,), generator=g, device=dev, dtype=torch.int32)
    pose = 0.3 * torch.randn((n, 24, 3), generator=g, device=dev)
    return tid, root, pose


def _inputs(case, seed):
    dev = torch.device("cuda", 0)
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) * 7919 + 13)
    if case["kind"] == "mlp":
        n = case["rows"]
        return dict(feat=torch.randn((n, 32), generator=g, device=dev),
                    band=torch.randint(0, 3, (n,), generator=g, device=dev, dtype=torch.int32),
                    target=torch.randn(n, generator=g, device=dev) - 1.0)
    tpls = _templates(case, g, dev)
    tid, root, pose = _instances(case, g, dev)
    grad = torch.randn((case["height"], case["width"], 4), generator=g, device=dev) if case["kind"] == "train" else None
    return dict(tpls=tpls, tid=tid, root=root, pose=pose, grad=grad)


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "mlp":
        return dict(s, case=case, mlp=binding.Mlp(device=0, seed=int(seed)))
    r = binding.Renderer(device=0, skin_mode=binding.CS_SKIN_MEANS_ONLY if case["skin"] == "means" else binding.CS_SKIN_FULL,
                         sh_frame=binding.CS_SH_WORLD_FRAME if case["world_sh"] else binding.CS_SH_ROOT_FRAME,
                         template_storage=binding.CS_STORE_BF16 if case["store"] == "bf16" else binding.CS_STORE_FP32)
    r.upload_templates([S.Template(parents=S.PARENTS, sh_degree=case["sh"], **{k: v.cpu().numpy() for k, v in t.items()})
                        for t in s["tpls"]])
    thr, frac, mult = LODS[case["lod"]]
    r.set_lod(S.LodConfig(thresholds=np.array(thr, np.float32), fractions=np.array(frac, np.float32),
                          scale_mult=np.array(mult, np.float32)))
    dev, size = s["tid"].device, (case["height"], case["width"], 4)
    st = dict(case=case, r=r, cam=_camera(case), tid=s["tid"], root=s["root"], pose=s["pose"], grad=s["grad"],
              n=len(s["tid"]))
    if case["host"]:
        for k in ("tid", "root", "pose"):
            st[k] = st[k].cpu().pin_memory()
        st["pinned"] = torch.empty(size, dtype=torch.float32).pin_memory()
        st["out"] = st["pinned"].numpy()
    else:
        st["out"] = torch.empty(size, device=dev)
    if case["kind"] == "contrib":
        st["contrib"] = torch.zeros(r.n_gauss_total, device=dev)
    if case["kind"] == "train":
        shapes = dict(means=(3,), scales=(3,), quats=(4,), opacity=(), sh=(16, 3))
        st["grads"] = {k: torch.zeros((r.n_gauss_total,) + v, device=dev) for k, v in shapes.items()}
        st["grads"]["pose"] = torch.zeros((st["n"], 24, 3), device=dev)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    case = state["case"]
    if case["kind"] == "mlp":
        m = state["mlp"]
        loss = m.train_step(state["feat"], state["band"], state["target"], 1e-3)
        return dict(loss=loss, grad=m.grad())
    r = state["r"]
    r.set_instances(state["tid"], state["root"], state["pose"])
    if case["kind"] == "train":
        img = r.render_train(state["cam"], out=state["out"])
        for v in state["grads"].values():
            v.zero_()
        return dict(img=img, **r.backward(state["grad"], state["n"], state["grads"]))
    if case["kind"] == "contrib":
        state["contrib"].zero_()
        return dict(img=r.render_contrib(state["cam"], state["contrib"], out=state["out"]), contrib=state["contrib"])
    if case["host"]:
        return r.render_to_host(state["cam"], out=state["out"])
    return r.render(state["cam"], out=state["out"])


def work(case):
    if case["kind"] == "mlp":
        n = case["rows"]
        return dict(bytes=n * (32 * 4 + 4 + 4), flops=6.0 * n * (36 * 64 + 64 * 64 + 64))
    k = 3 * (case["sh"] + 1) ** 2
    attr = 60 + 4 * k if case["store"] == "fp32" else 32 + 2 * k
    frac = max(LODS[case["lod"]][1])
    total, pixels, n = case["templates"] * case["gauss"], case["width"] * case["height"], case["cols"] * case["rows"]
    by = total * frac * attr + n * (4 + 48 + 288) + pixels * 16
    # skinning 96, covariance and projection 200, colour 2 per coefficient plus its basis
    fl = _splats(case) * (300 + 2 * k + k)
    if case["kind"] == "contrib":
        by += 8 * total
    if case["kind"] == "train":
        by += pixels * 16 + total * (attr + 4 * 59) + n * 288
        fl *= 3
    return dict(bytes=float(by), flops=float(fl))


# ---------------------------------------------------------------------------
# FP64
# ---------------------------------------------------------------------------

def _basis(deg, d):
    """Real spherical harmonics to degree 3 (degree 1: -y, z, -x)."""
    x, y, z = d.unbind(-1)
    p = math.pi
    xx, yy, zz = x * x, y * y, z * z
    c0, c1 = 0.5 / math.sqrt(p), math.sqrt(3 / (4 * p))
    a2, b2, e2 = math.sqrt(15 / p) / 2, math.sqrt(5 / p) / 4, math.sqrt(15 / p) / 4
    k0, k1, k2 = math.sqrt(35 / (2 * p)) / 4, math.sqrt(105 / p) / 2, math.sqrt(21 / (2 * p)) / 4
    k3, k5 = math.sqrt(7 / p) / 4, math.sqrt(105 / p) / 4
    y_ = [c0 * torch.ones_like(x), -c1 * y, c1 * z, -c1 * x, a2 * x * y, -a2 * y * z, b2 * (2 * zz - xx - yy),
          -a2 * x * z, e2 * (xx - yy), -k0 * y * (3 * xx - yy), k1 * x * y * z, -k2 * y * (4 * zz - xx - yy),
          k3 * z * (2 * zz - 3 * xx - 3 * yy), -k2 * x * (4 * zz - xx - yy), k5 * z * (xx - yy),
          -k0 * x * (xx - 3 * yy)]
    return torch.stack(y_[:(deg + 1) ** 2], -1)


def _skin(pose, rest):
    """Joint transforms [24, 3, 4] relative to the rest pose: R(v) = exp([v]x), parents first."""
    zero = torch.zeros_like(pose[:, 0])
    v0, v1, v2 = pose.unbind(1)
    K = torch.stack([zero, -v2, v1, v2, zero, -v0, -v1, v0, zero], 1).reshape(-1, 3, 3)
    R = torch.linalg.matrix_exp(K)
    GR, Gt = [], []
    for j, p in enumerate(S.PARENTS.tolist()):
        if p < 0:
            GR.append(R[j])
            Gt.append(rest[j])
        else:
            GR.append(GR[p] @ R[j])
            Gt.append(GR[p] @ (rest[j] - rest[p]) + Gt[p])
    GR, Gt = torch.stack(GR), torch.stack(Gt)
    return torch.cat([GR, (Gt - (GR @ rest[..., None])[..., 0])[..., None]], 2)


def _project(case, cam, t, pose, root, m, count):
    """The instance's first `count` Gaussians as splats (depth, u, v, conic, opacity, rgb, radius)."""
    f64 = dict(dtype=torch.float64, device=pose.device)
    Rc, tc = torch.tensor(cam.R, **f64), torch.tensor(cam.t, **f64)
    mu, w = t["means"][:count], t["skin_w"][:count]
    B = _skin(pose, t["rest_joints"].double())[t["skin_idx"][:count].long()]
    M = (w[..., None, None] * B).sum(1)
    pl = (M[:, :, :3] @ mu[..., None])[..., 0] + M[:, :, 3]
    Rr, tr = root[:, :3], root[:, 3]
    cam_p = (pl @ Rr.T + tr) @ Rc.T + tc
    W = Rc @ Rr
    W = W.expand(len(mu), 3, 3) if case["skin"] == "means" else W @ M[:, :, :3]
    q = t["quats"][:count]
    q = q / q.norm(dim=1, keepdim=True)
    a, b, c, d = q.unbind(1)
    R = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c), 2 * (b * c + a * d),
                     1 - 2 * (b * b + d * d), 2 * (c * d - a * b), 2 * (b * d - a * c), 2 * (c * d + a * b),
                     1 - 2 * (b * b + c * c)], 1).reshape(-1, 3, 3)
    L = W @ (R * (m * t["scales"][:count])[:, None])
    x, y, z = cam_p.unbind(1)
    lx, ly = 1.3 * cam.width / (2 * cam.fx), 1.3 * cam.height / (2 * cam.fy)
    zero = torch.zeros_like(z)
    cx, cy = (x / z).clamp(-lx, lx), (y / z).clamp(-ly, ly)
    J = torch.stack([cam.fx / z, zero, -cam.fx * cx / z, zero, cam.fy / z, -cam.fy * cy / z], 1).reshape(-1, 2, 3)
    T = J @ L
    C = T @ T.transpose(1, 2)
    A0, B0, C0 = C[:, 0, 0] + 0.3, C[:, 0, 1], C[:, 1, 1] + 0.3
    det = A0 * C0 - B0 * B0
    mid = 0.5 * (A0 + C0)
    rad = torch.ceil(3 * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
    centre = -Rc.T @ tc
    view = pl - Rr.T @ (centre - tr)
    view = view @ Rr.T if case["world_sh"] else view
    Y = _basis(case["sh"], view / view.norm(dim=1, keepdim=True))
    rgb = ((Y[..., None] * t["sh"][:count]).sum(1) + 0.5).clamp(min=0)
    u, v = cam.fx * x / z + cam.cx, cam.fy * y / z + cam.cy
    sp = torch.stack([z, u, v, C0 / det, -B0 / det, A0 / det, t["opacity"][:count], *rgb.unbind(1), rad], 1)
    return sp, (z > cam.near).detach()


def _composite(sp, cam, backward=None):
    """RGBA [H, W, 4] of splats [n, 11] (depth first); with `backward`
    (dL/dRGBA) also dL/d(splats)."""
    W, H, dev = cam.width, cam.height, sp.device
    sp = sp[sp[:, 0].argsort(stable=True)] if backward is None else sp
    at = sp.detach()
    lo = [((at[:, k] - at[:, 10] - 0.5).ceil().clamp(min=0) / 16).floor().long() for k in (1, 2)]
    hi = [((at[:, k] + at[:, 10] - 0.5).floor().clamp(max=n - 1) / 16).floor().long() for k, n in ((1, W), (2, H))]
    nx, ny = [(h - l + 1).clamp(min=0) for l, h in zip(lo, hi)]
    cnt = nx * ny
    who = torch.repeat_interleave(torch.arange(len(sp), device=dev), cnt)
    k = torch.arange(len(who), device=dev) - (cnt.cumsum(0) - cnt)[who]
    tx, step = (W + 15) // 16, nx[who].clamp(min=1)
    tile = (lo[1][who] + k // step) * tx + lo[0][who] + k % step
    order = tile.argsort(stable=True)
    who, ends = who[order], tile.bincount(minlength=tx * ((H + 15) // 16)).cumsum(0).tolist()
    out = torch.zeros((H, W, 4), dtype=torch.float64, device=dev)
    grad = None if backward is None else torch.zeros_like(at)
    for i, e in enumerate(ends):
        b = ends[i - 1] if i else 0
        if e == b:
            continue
        x0, y0 = i % tx * 16, i // tx * 16
        px = torch.arange(x0, min(x0 + 16, W), device=dev, dtype=torch.float64) + 0.5
        py = torch.arange(y0, min(y0 + 16, H), device=dev, dtype=torch.float64) + 0.5
        gx, gy = [g.reshape(-1) for g in torch.meshgrid(px, py, indexing="xy")]
        T0, rgba, s, first = torch.ones_like(gx), torch.zeros((len(gx), 4), dtype=torch.float64, device=dev), None, True
        for c in range(b, e, 16384 if backward is None else e - b):
            ids = who[c:min(e, c + 16384) if backward is None else e]
            s = at[ids].requires_grad_(backward is not None)
            dx, dy = gx - s[:, 1:2], gy - s[:, 2:3]
            p = -0.5 * (s[:, 3:4] * dx * dx + s[:, 5:6] * dy * dy) - s[:, 4:5] * dx * dy
            al = (s[:, 6:7] * torch.exp(p.clamp(max=0))).clamp(max=0.99)
            on = (torch.maximum(dx.abs(), dy.abs()) <= s[:, 10:11]) & (p <= 0) & (al >= 1 / 255)
            al = torch.where(on, al, torch.zeros_like(al))
            Ti = T0 * torch.cumprod(1 - al, 0)
            keep = Ti.detach() >= 1e-4
            al = torch.where(keep, al, torch.zeros_like(al))
            Ti = T0 * torch.cumprod(1 - al, 0)
            w = al * torch.cat([T0[None], Ti[:-1]])
            # a stopped pixel stays stopped: everything behind it is hidden
            T0 = torch.where(keep[-1], Ti[-1], torch.zeros_like(T0)) if backward is None else Ti[-1]
            rgba = rgba + torch.cat([w.T @ s[:, 7:10], w.sum(0)[:, None]], 1)
        if backward is not None:
            g = backward[y0:y0 + len(py), x0:x0 + len(px)].reshape(-1, 4)
            grad.index_add_(0, ids, torch.autograd.grad((rgba * g).sum(), s)[0])
        out[y0:y0 + len(py), x0:x0 + len(px)] = rgba.detach().reshape(len(py), len(px), 4)
    return out if backward is None else (out, grad)


def _exact_mlp(case, seed):
    s = _inputs(case, seed)
    p = torch.from_numpy(binding.Mlp(device=0, seed=int(seed)).params()).double().cuda().requires_grad_(True)
    i1, i2 = 48 * 64, 48 * 64 + 64
    W1, b1, W2, b2 = p[:i1].view(48, 64), p[i1:i2], p[i2:i2 + 4096].view(64, 64), p[i2 + 4096:i2 + 4160]
    w3, b3 = p[i2 + 4160:i2 + 4224], p[i2 + 4224]
    n, loss, grad = case["rows"], 0.0, torch.zeros_like(p)
    for c in range(0, n, 1 << 18):
        x = torch.zeros((min(n, c + (1 << 18)) - c, 48), dtype=torch.float64, device=p.device)
        x[:, :32] = s["feat"][c:c + len(x)]
        x[:, 32:36] = torch.nn.functional.one_hot(s["band"][c:c + len(x)].long(), 4)
        y = torch.relu(torch.relu(x @ W1 + b1) @ W2 + b2) @ w3 + b3
        part = ((y - s["target"][c:c + len(x)]) ** 2).sum() / n
        grad += torch.autograd.grad(part, p, retain_graph=True)[0]
        loss += float(part)
    return dict(loss=loss, grad=grad)


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "contrib" or _splats(case) > (1.5e6 if case["kind"] == "frame" else 3e4):
        return None
    s, cam = _inputs(case, seed), _camera(case)
    train = case["kind"] == "train"
    tpls = [{k: v.double() if v.dtype == torch.float32 else v for k, v in t.items()} for t in s["tpls"]]
    leaves = {k: tpls[0][k].requires_grad_(True) for k in ("means", "scales", "quats", "opacity", "sh")} if train else {}
    pose, root = s["pose"].double().requires_grad_(train), s["root"].double()
    thr, frac, mult = LODS[case["lod"]]
    centre = torch.from_numpy(-cam.R.astype(np.float64).T @ cam.t.astype(np.float64)).to(root.device)
    dist = (root[:, :, 3] - centre).norm(dim=1).tolist()
    parts = []
    for i, t in enumerate(s["tid"].tolist()):
        lvl = sum(dist[i] >= np.float32(x) for x in thr)
        count = int(math.floor(float(np.float32(frac[lvl])) * case["gauss"] + 0.5))
        sp, live = _project(case, cam, tpls[t], pose[i], root[i], float(np.float32(mult[lvl])), count)
        at = sp.detach()
        live &= (at[:, 1] > -at[:, 10] - 1) & (at[:, 1] < cam.width + at[:, 10] + 1)
        live &= (at[:, 2] > -at[:, 10] - 1) & (at[:, 2] < cam.height + at[:, 10] + 1)
        parts.append(sp[live])
    sp = torch.cat(parts)
    if not train:
        return _composite(sp, cam)
    sp = sp[sp[:, 0].detach().argsort(stable=True)]
    img, g = _composite(sp, cam, backward=s["grad"].double())
    names = list(leaves) + ["pose"]
    got = dict(zip(names, torch.autograd.grad(sp, list(leaves.values()) + [pose], g)))
    sh = torch.zeros((case["gauss"], 16, 3), dtype=torch.float64, device=sp.device)
    sh[:, :got["sh"].shape[1]] = got["sh"]
    return dict(got, img=img, sh=sh)
