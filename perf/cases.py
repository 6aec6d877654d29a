"""Performance cases of the RayGS renderer: what its users run, through its public entry points.

A case is a dict of plain values:

  kind     "frame"        one forward pass, preprocess + binning + rasteriser, launched directly
           "loop"         one frame of a display loop: new poses, then the captured graph's replay
           "train"        one forward + backward through the autograd function (L1 loss)
           "supersample"  a forward pass at `factor` times the resolution, then the box resolve
           "noalloc"      the allocation-free entry point (it waits for its own result)
  scene    "uniform" (the small test scene) or "blobs" (the reconstructed-capture shape), n
           primitives, sh_degree, a fraction `flat` of near-degenerate disks
  storage  "f32"; "sh16" (SH alone in FP16), "f16" / "bf16" (SH, log-scales; logits in FP16)
  cameras  "front" (one view at the origin), "ragged" (views of uneven size on a sphere around
           the scene), "stereo" (pairs at width x height per eye, then `extra` smaller uneven
           views) or "4k" (four poses at width x height, and the same at a quarter with MIP)
  mip, divergence   the anti-aliasing mode of the views and the divergence of the plan

Scenes follow scenes.py's recipes but are drawn on the GPU, so that preparing them is quick.
The outputs are what a program shows or optimises: the image, the final transmittance and the
gradients.  (n_contrib indexes the plan's own lists; it is asked for where the backward needs
it.)
"""
import math

import numpy as np
import torch

from paper_2503_18682_gb300 import raygs, scenes

_BASE = dict(kind="frame", scene="blobs", n=1000, sh_degree=3, flat=0.0, storage="f32", cameras="front", views=1,
             extra=0, width=64, height=64, focal=64.0, mip="off", divergence="ray", factor=1)


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one thumbnail of a thousand primitives (latency, launches)
        _case("thumbnail_64", scene="uniform", n=1000, sh_degree=0),
        # a plug-in drawing a small overlay out of the library's own array; odd size
        _case("noalloc_overlay", kind="noalloc", scene="uniform", n=5000, sh_degree=0, width=253, height=187,
              focal=200.0, mip="approx"),
        # the smallest training step: gradient checks, fitting a tiny scene
        _case("train_tiny_128", kind="train", scene="blobs", n=2000, sh_degree=3, width=128, height=128, focal=100.0),
        # a training batch of a few uneven low-resolution views
        _case("train_batch_ragged", kind="train", n=200_000, sh_degree=2, cameras="ragged", views=4, width=640,
              height=480, focal=500.0),
        # the forward + backward benchmark view: 1.5M primitives at 1280x720
        _case("train_720p_1p5m", kind="train", n=1_500_000, width=1280, height=720, focal=1000.0),
        # an ordinary frame: 500k primitives at 1280x720 with the pixel-invariant anti-aliasing
        _case("frame_720p_mip", n=500_000, width=1280, height=720, focal=1000.0, mip="approx"),
        # the same frame with the exact, pixel-dependent anti-aliasing
        _case("frame_720p_mip_exact", n=500_000, width=1280, height=720, focal=1000.0, mip="exact"),
        # the same frame rendered with the GS divergence
        _case("frame_720p_gs", n=500_000, width=1280, height=720, focal=1000.0, divergence="gs"),
        # the same frame, 2x2 supersampled
        _case("supersample_720p", kind="supersample", n=500_000, width=1280, height=720, focal=1000.0, factor=2),
        # one headset frame: a stereo pair of a mid-sized scene stored with FP16 colour
        _case("vr_pair_1m_sh16", kind="loop", n=1_000_000, flat=0.1, storage="sh16", cameras="stereo", views=2,
              width=2064, height=2208, focal=1100.0),
        # the headline batch: 3M primitives, four stereo pairs and eight smaller uneven views
        _case("vr_batch_3m", kind="loop", n=3_000_000, flat=0.1, cameras="stereo", views=8, extra=8, width=2064,
              height=2208, focal=1100.0),
        # the largest: 6M primitives in FP16 storage, four 3840x2160 views and four quarter-size MIP ones
        _case("4k_6m_f16", n=6_000_000, storage="f16", cameras="4k", views=8, width=3840, height=2160, focal=2000.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tiny", "noalloc", "train_tiny", "train", "train", "frame", "frame", "supersample", "loop", "loop", "4k"])
    deg = rng.choice([0, 1, 2, 3, 3])
    if kind == "tiny":
        w, h = _log(rng, 33, 256), _log(rng, 33, 256)
        return _case(scene="uniform", n=_log(rng, 500, 20_000), sh_degree=0, width=w, height=h, focal=float(w))
    if kind == "noalloc":
        w, h = _log(rng, 64, 400), _log(rng, 64, 300)
        return _case(kind="noalloc", scene="uniform", n=_log(rng, 1000, 10_000), sh_degree=0, width=w, height=h,
                     focal=0.8 * w, mip=rng.choice(["off", "approx"]))
    if kind == "train_tiny":
        w, h = rng.randint(48, 160), rng.randint(48, 160)
        return _case(kind="train", n=_log(rng, 300, 4000), sh_degree=deg, width=w, height=h, focal=0.8 * w)
    if kind == "train":
        w, h = rng.randint(320, 1280), rng.randint(240, 720)
        if rng.random() < 0.5:
            return _case(kind="train", n=_log(rng, 50_000, 400_000), sh_degree=deg, cameras="ragged",
                         views=rng.randint(2, 6), width=w, height=h, focal=0.8 * w, flat=rng.choice([0.0, 0.1]))
        return _case(kind="train", n=_log(rng, 100_000, 1_500_000), sh_degree=deg, width=w, height=h, focal=0.8 * w)
    if kind in ("frame", "supersample"):
        w, h = rng.randint(400, 1920), rng.randint(300, 1080)
        c = dict(n=_log(rng, 50_000, 2_000_000), sh_degree=deg, width=w, height=h, focal=0.8 * w,
                 storage=rng.choice(["f32", "f32", "sh16", "f16", "bf16"]))
        if kind == "supersample":
            return _case(kind="supersample", factor=rng.choice([2, 2, 3]), **dict(c, width=w // 2, height=h // 2,
                                                                                 focal=0.4 * w))
        mode = rng.choice(["off", "approx", "approx", "exact", "gs"])
        return _case(mip="off" if mode == "gs" else mode, divergence="gs" if mode == "gs" else "ray", **c)
    if kind == "loop":
        w, h = rng.randint(1000, 2064), rng.randint(1000, 2208)
        return _case(kind="loop", n=_log(rng, 300_000, 3_000_000), sh_degree=deg, flat=rng.choice([0.0, 0.1]),
                     storage=rng.choice(["f32", "sh16", "bf16"]), cameras="stereo", views=2 * rng.randint(1, 4),
                     extra=rng.randint(0, 8), width=w, height=h, focal=0.53 * w)
    w, h = rng.randint(1920, 3840), rng.randint(1080, 2160)
    return _case(n=_log(rng, 1_000_000, 6_000_000), storage=rng.choice(["f32", "f16", "bf16"]), cameras="4k", views=8,
                 width=w, height=h, focal=0.52 * w)


# ------------------------------------------------------------------------------- inputs

def _scene(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    n, dev = case["n"], "cuda"
    k = (case["sh_degree"] + 1) ** 2

    def u(*shape, lo=0.0, hi=1.0):
        return torch.rand(shape, generator=g, device=dev) * (hi - lo) + lo

    def z(*shape):
        return torch.randn(shape, generator=g, device=dev)

    quats = torch.nn.functional.normalize(z(n, 4), dim=1)
    if case["scene"] == "uniform":
        means = torch.stack([u(n, lo=-1, hi=1), u(n, lo=-1, hi=1), u(n, lo=2, hi=4)], dim=1)
        log_scales = u(n, 3, lo=math.log(0.01), hi=math.log(0.1))
        logits = z(n)
    else:
        centres = torch.cat([u(64, 2, lo=-5, hi=5), u(64, 1, lo=1, hi=11)], dim=1)
        which = torch.randint(0, 64, (n,), generator=g, device=dev)
        means = centres[which] + 0.3 * z(n, 3)
        log_scales = math.log(0.02) + 0.8 * z(n, 3)
        if case["flat"] > 0:
            thin = u(n) < case["flat"]
            amin = log_scales.argmin(dim=1, keepdim=True)
            flat = log_scales.amax(dim=1, keepdim=True) - u(n, 1, lo=3, hi=4) * math.log(10.0)
            log_scales = torch.where(thin[:, None], log_scales.scatter(1, amin, flat), log_scales)
        logits = 1.5 * z(n)
    sh = torch.empty((n, k, 3), device=dev)
    sh[:, 0] = u(n, 3)
    if k > 1:
        sh[:, 1:] = 0.05 * z(n, k - 1, 3)
    st = dict(means=means.contiguous(), log_scales=log_scales.contiguous(), quats=quats.contiguous(),
              opacity_logits=logits.contiguous(), sh=sh, sh_degree=case["sh_degree"])
    if case["storage"] != "f32":
        half = torch.bfloat16 if case["storage"] == "bf16" else torch.float16
        st["sh"] = st["sh"].to(half)
        if case["storage"] != "sh16":
            st["log_scales"] = st["log_scales"].to(half)
            st["opacity_logits"] = st["opacity_logits"].to(torch.float16)
    return st


def _cameras(case, seed):
    rng = np.random.default_rng(int(seed) + 1000)
    centre = np.array([0.0, 0.0, 6.0])
    w, h, f = case["width"], case["height"], case["focal"]
    mip = {"off": False, "approx": True, "exact": "exact"}[case["mip"]]

    def pose():
        v = rng.standard_normal(3)
        return centre + 3.0 * v / np.linalg.norm(v)

    if case["cameras"] == "front":
        return [scenes.make_camera(w, h, f, f, mip=mip)]
    cams = []
    if case["cameras"] == "ragged":
        size = np.random.default_rng(w * 65537 + h * 31 + case["views"])   # sizes belong to the case
        for _ in range(case["views"]):
            s = size.uniform(0.6, 1.0, 2)
            R, t = scenes.look_at(pose(), centre)
            cams.append(scenes.make_camera(int(w * s[0]), int(h * s[1]), f, f, R=R, t=t, mip=mip))
    elif case["cameras"] == "stereo":
        for _ in range(case["views"] // 2):
            eye = pose()
            R, _ = scenes.look_at(eye, centre)
            for side in (-0.5, 0.5):
                e = eye + side * 0.064 * R[0].astype(np.float64)
                cams.append(scenes.make_camera(w, h, f, f, R=R, t=-(R.astype(np.float64) @ e), mip=mip))
        size = np.random.default_rng(w * 65537 + h * 31 + case["extra"])
        for _ in range(case["extra"]):
            ew, eh = int(size.uniform(0.31, 0.93) * w), int(size.uniform(0.22, 0.49) * h)
            R, t = scenes.look_at(pose(), centre)
            cams.append(scenes.make_camera(ew, eh, f * ew / w, f * ew / w, R=R, t=t, mip=mip))
    else:
        low = []
        for _ in range(case["views"] // 2):
            R, t = scenes.look_at(pose(), centre)
            cams.append(scenes.make_camera(w, h, f, f, R=R, t=t))
            low.append(scenes.make_camera(w // 4, h // 4, f / 4, f / 4, R=R, t=t, mip=True))
        cams += low
    return cams


def prepare(case, seed):
    scene, cams = _scene(case, seed), _cameras(case, seed)
    s = dict(case=case, scene=scene, cams=cams)
    kind = case["kind"]
    px = sum(c["width"] * c["height"] for c in cams)
    if kind == "noalloc":
        s.update(sc=raygs.make_scene(scene), cfg=raygs.make_config(), rgb=torch.empty((px, 3), device="cuda"),
                 T=torch.empty(px, device="cuda"))
        return s
    if kind == "train":
        r = raygs.Renderer(cams, case["n"], enable_backward=1)
        leaves = {k: v.requires_grad_(True) for k, v in scene.items() if k != "sh_degree"}
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 3)
        s.update(r=r, leaves=leaves, target=torch.rand((px, 3), generator=g, device="cuda"))
        with torch.no_grad():   # a first pass sizes the plan
            raygs.render(r, dict(leaves, sh_degree=case["sh_degree"]))
        return s
    if kind == "supersample":
        r = raygs.Renderer(raygs.supersampled_cameras(cams, case["factor"]), case["n"])
        s.update(lo_rgb=torch.empty((px, 3), device="cuda"), lo_T=torch.empty(px, device="cuda"))
    else:
        r = raygs.Renderer(cams, case["n"], divergence=1 if case["divergence"] == "gs" else 0)
    rgb, T, _ = r.alloc_outputs()
    r.forward(scene, rgb, T)    # a first pass sizes the plan
    s.update(r=r, rgb=rgb, T=T)
    if kind == "loop":
        s.update(sc=raygs.make_scene(scene), poses=raygs.make_cameras(cams))
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        raygs.raygs_graph_capture(r.plan, s["sc"], rgb, T, stream=side)
        side.synchronize()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "noalloc":
        raygs.raygs_render_noalloc(s["cams"], s["sc"], s["cfg"], s["rgb"], s["T"])
        return s["rgb"], s["T"]
    if kind == "train":
        leaves = s["leaves"]
        rgb, T, _ = raygs.render(s["r"], dict(leaves, sh_degree=case["sh_degree"]))
        loss = (rgb - s["target"]).abs().sum()
        grads = torch.autograd.grad(loss, list(leaves.values()))
        return dict(rgb=rgb.detach(), T=T.detach(), grads=dict(zip(leaves, grads)))
    r = s["r"]
    if kind == "loop":
        raygs.raygs_plan_set_poses(r.plan, s["poses"])
        raygs.raygs_graph_launch(r.plan)
        return s["rgb"], s["T"]
    r.forward(s["scene"], s["rgb"], s["T"], check=False)
    if kind == "supersample":
        raygs.raygs_resolve_supersampled(r.plan, case["factor"], s["rgb"], s["T"], s["lo_rgb"], s["lo_T"])
        return s["lo_rgb"], s["lo_T"]
    return s["rgb"], s["T"]


def work(case):
    """Attributes read and images (and gradients) written once; the arithmetic of the vertex
    stage per (primitive, view).  What the compositing costs depends on the scene's content
    and is not in these figures."""
    n, k3 = case["n"], 3 * (case["sh_degree"] + 1) ** 2
    sh_b = 4 if case["storage"] == "f32" else 2
    ls_b = 2 if case["storage"] in ("f16", "bf16") else 4
    attr = n * (12 + 16 + 3 * ls_b + ls_b + k3 * sh_b)
    cams = _cameras(case, 0)
    px = sum(c["width"] * c["height"] for c in cams)
    out = 16 * px
    if case["kind"] == "train":     # target and image gradient read, gradients written
        out += 12 * px + 4 * n * (11 + k3)
    flops = n * len(cams) * (300 + 2 * k3) * (3 if case["kind"] == "train" else 1)
    return dict(bytes=attr + out, flops=flops)


# ------------------------------------------------------------- the same image in 64 bits

_SH = (
    lambda x, y, z: 1.0 + 0 * x,
    lambda x, y, z: math.sqrt(3 / (4 * math.pi)) * y,
    lambda x, y, z: math.sqrt(3 / (4 * math.pi)) * z,
    lambda x, y, z: math.sqrt(3 / (4 * math.pi)) * x,
    lambda x, y, z: math.sqrt(15 / (4 * math.pi)) * x * y,
    lambda x, y, z: math.sqrt(15 / (4 * math.pi)) * y * z,
    lambda x, y, z: math.sqrt(5 / (16 * math.pi)) * (3 * z * z - 1),
    lambda x, y, z: math.sqrt(15 / (4 * math.pi)) * x * z,
    lambda x, y, z: math.sqrt(15 / (16 * math.pi)) * (x * x - y * y),
    lambda x, y, z: math.sqrt(35 / (32 * math.pi)) * y * (3 * x * x - y * y),
    lambda x, y, z: math.sqrt(105 / (4 * math.pi)) * x * y * z,
    lambda x, y, z: math.sqrt(21 / (32 * math.pi)) * y * (5 * z * z - 1),
    lambda x, y, z: math.sqrt(7 / (16 * math.pi)) * z * (5 * z * z - 3),
    lambda x, y, z: math.sqrt(21 / (32 * math.pi)) * x * (5 * z * z - 1),
    lambda x, y, z: math.sqrt(105 / (16 * math.pi)) * z * (x * x - y * y),
    lambda x, y, z: math.sqrt(35 / (32 * math.pi)) * x * (x * x - 3 * y * y),
)


def _dense(p, cam, x0, x1):
    """Colour and final transmittance of the pixels [x0, x1) of one view, every pixel against
    every primitive, in float64: the ray's maximum density, cut off at 1/255, clamped at 0.99,
    composited in depth order until the transmittance would fall below 1e-4."""
    f64 = dict(dtype=torch.float64, device="cuda")
    R, t = torch.as_tensor(cam["R"], **f64), torch.as_tensor(cam["t"], **f64)
    fx, fy, cx, cy = (float(cam[k]) for k in ("fx", "fy", "cx", "cy"))
    mu = p["means"] @ R.T + t
    q = p["quats"] / p["quats"].norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    Rp = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                      1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                      1 - 2 * (x * x + y * y)], dim=1).view(-1, 3, 3)
    N = R @ Rp                                                  # columns: axes in the camera frame
    s2 = torch.exp(2 * p["log_scales"])
    o = torch.sigmoid(p["opacity_logits"])
    proj = torch.einsum("nik,ni->nk", N, mu)
    c2 = (proj * proj / s2).sum(1)
    if cam["mip"] == 1:
        lam = (0.1 * (mu * mu).sum(1) / (fx * fy))[:, None]
        h2 = s2 + lam
        ch2 = (proj * proj / h2).sum(1)
        o = o * torch.sqrt((s2 / h2).prod(1) * c2 / ch2)
        s2, c2 = h2, ch2
    kappa = 2 * torch.log(o * 255)
    keep = (mu[:, 2] > float(cam["near"])) & (kappa > 0) & (c2 > kappa)
    order = torch.argsort(mu[:, 2].detach().float(), stable=True)
    order = order[keep[order]]
    mu, N, s2, o, kappa = mu[order], N[order], s2[order], o[order], kappa[order]
    centre = -(R.T @ t)
    d = p["means"][order] - centre
    d = d / d.norm(dim=1, keepdim=True)
    sh = p["sh"][order]
    rgb = sum(_SH[k](*d.unbind(1))[:, None] * sh[:, k] for k in range(sh.shape[1])).clamp(min=0)
    pix = torch.arange(x0, x1, device="cuda")
    ray = torch.stack([((pix % cam["width"]).double() + 0.5 - cx) / fx,
                       (torch.div(pix, cam["width"], rounding_mode="floor").double() + 0.5 - cy) / fy,
                       torch.ones(x1 - x0, **f64)], dim=1)
    sr = torch.sqrt(s2)
    ry = [(ray @ N[:, :, k].T) / sr[:, k] for k in range(3)]   # whitened rays and means, [pixel, primitive]
    rm = [(N[:, :, k] * mu).sum(1) / sr[:, k] for k in range(3)]
    yy = ry[0] ** 2 + ry[1] ** 2 + ry[2] ** 2
    my = rm[0] * ry[0] + rm[1] * ry[1] + rm[2] * ry[2]
    e = [rm[1] * ry[2] - rm[2] * ry[1], rm[2] * ry[0] - rm[0] * ry[2], rm[0] * ry[1] - rm[1] * ry[0]]
    D = (e[0] ** 2 + e[1] ** 2 + e[2] ** 2) / yy               # |m x y|^2 / |y|^2: no cancellation
    om = torch.where((my > 0) & (D <= kappa), (o * torch.exp(-0.5 * D)).clamp(max=0.99), torch.zeros((), **f64))
    after = torch.cumprod(1 - om, dim=1)
    om = torch.where(after >= 1e-4, om, torch.zeros((), **f64))
    T = torch.cumprod(1 - om, dim=1)
    before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], dim=1)
    return (om * before) @ rgb, T[:, -1] if T.shape[1] else torch.ones(x1 - x0, **f64)


def exact(case, seed):
    cams = _cameras(case, seed)
    px = sum(c["width"] * c["height"] for c in cams)
    train = case["kind"] == "train"
    if case["kind"] == "supersample" or case["mip"] == "exact" or case["divergence"] == "gs":
        return None
    if case["n"] * px > (1e8 if train else 6e8):
        return None     # every pixel against every primitive: too long
    scene = _scene(case, seed)
    p = {k: v.double().requires_grad_(train) for k, v in scene.items() if k != "sh_degree"}
    target = None
    if train:
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 3)
        target = torch.rand((px, 3), generator=g, device="cuda").double()
    step = max(1, int(8e6) // max(1, case["n"]))
    rgbs, Ts, done = [], [], 0
    with torch.set_grad_enabled(train):
        for cam in cams:
            n_px = cam["width"] * cam["height"]
            for a in range(0, n_px, step):
                b = min(n_px, a + step)
                rgb, T = _dense(p, cam, a, b)
                if train:
                    (rgb - target[done + a:done + b]).abs().sum().backward()
                rgbs.append(rgb.detach())
                Ts.append(T.detach())
            done += n_px
    rgb, T = torch.cat(rgbs), torch.cat(Ts)
    if train:
        return dict(rgb=rgb, T=T, grads={k: v.grad for k, v in p.items()})
    return rgb, T
