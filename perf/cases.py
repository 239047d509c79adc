"""Timed cases of the fisheye stereo library, through its public entry points.

A case is what a program of this library does again and again: one frame of
a rig (cold, from a host buffer, or continued from the last one), a batch of
pairs, a pose change, the primal-dual iterations alone.  Sizes and solver
settings are those of the repository's workloads, tests and benchmark.

Inputs are rendered here from a seed: a stereo pair of a fisheye rig in a
sphere with textured planes and balls (the value range and texture spectrum
the method meets), images in [0, 1] with Gaussian noise of 0.01, as float32.
``exact`` is the method in 64 bits, written with plain torch operations.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_1909_07545_gb300 as fsb

DEV = "cuda"
F64 = torch.float64
LAM, EPS, DU, BETA, ETA = 50.0, 0.01, 0.2, 9.0, 0.85
ALPHA0, ALPHA1 = 17.0, 1.2


# ------------------------------------------------------------------ the cases

def _frame(name, W, H, levels, warps, iters, **kw):
    c = dict(name=name, kind="frame", W=W, H=H, levels=levels, warps=warps, iters=iters,
             model="kb", reg="huber_tv", storage="f32", deriv="forward", accel=0.0, graph=1,
             tune=0, start="cold")
    c.update(kw)
    return c


def listed():
    return [
        # the iterations alone on a caller's buffers (a host that may not
        # allocate device memory): the smallest call
        dict(name="iterate_160x120", kind="iterate", W=160, H=120, iters=20),
        # a thumbnail-sized rig, launched directly: latency and launches
        _frame("small_128", 128, 128, 3, 3, 20, model="equidistant", graph=0),
        # the small equidistant workload of the tests, replayed
        _frame("plain_256", 256, 256, 3, 5, 50, model="equidistant"),
        # a ragged size, the accelerated steps and the central derivative
        _frame("ragged_333x257_accel", 333, 257, 4, 5, 40, accel=0.4, deriv="central"),
        # a rig whose pose is re-estimated per frame: fields and pre-rotation
        dict(name="repose_1024", kind="repose", W=1024, H=1024, levels=5),
        # the paper's timing setup (Fig. 4): 20 warps of 10 iterations
        _frame("paper_800", 800, 800, 5, 20, 10, model="equidistant"),
        # one frame from pinned host buffers and back, the size of a tracking
        # camera's fisheye pair
        _frame("host_848x800", 848, 800, 5, 5, 50, start="host"),
        # the next frame of a video stream from the rig's last result, as the
        # server runs it: 3 warps of 50 on the finest level
        _frame("video_640", 640, 640, 5, 3, 50, start="continue", tune=1),
        # the benchmark's frame, tuned and replayed
        _frame("kb_1024", 1024, 1024, 5, 10, 100, tune=1),
        # the paper's TGV-L1 energy
        _frame("tgv_800", 800, 800, 5, 5, 30, reg="tgv"),
        # the largest single frame of the workloads
        _frame("equidistant_2048", 2048, 2048, 6, 10, 100, model="equidistant"),
        # many rigs of uneven sizes in one call, 16-bit storage
        dict(name="batch_uneven_8", kind="batch", sizes="512,800,1024,1280", pairs=8, warps=10,
             iters=100, storage="f16", finest=2),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _levels(W, H):
    # every level at least 40 pixels wide, as the workloads have it
    n = 1
    while min(W, H) / 2 ** n >= 40 and n < 7:
        n += 1
    return n


def draw(rng):
    kind = rng.choice(["frame"] * 6 + ["iterate", "repose", "batch"])
    if kind == "iterate":
        W = _log_size(rng, 48, 512)
        return dict(kind=kind, W=W, H=min(_log_size(rng, 48, 512), 512 * 512 // W),
                    iters=rng.randint(5, 100))
    W = _log_size(rng, 96, 1900)
    H = max(96, min(1900, int(W * rng.choice([1.0, 1.0, 0.75, rng.uniform(0.5, 1.5)]))))
    if kind == "repose":
        return dict(kind=kind, W=W, H=H, levels=_levels(W, H))
    if kind == "batch":
        sizes = [str(_log_size(rng, 200, 1100)) for _ in range(rng.randint(2, 4))]
        return dict(kind=kind, sizes=",".join(sizes), pairs=rng.randint(2, 6),
                    warps=rng.randint(2, 8), iters=rng.randint(20, 80),
                    storage=rng.choice(["f32", "f16", "bf16"]), finest=rng.choice([0, 1, 2]))
    reg = rng.choice(["huber_tv"] * 4 + ["tgv"])
    storage = rng.choice(["f32", "f32", "f16", "bf16"]) if reg == "huber_tv" else "f32"
    accel = rng.choice([0.0, 0.0, 0.0, 0.4]) if reg == "huber_tv" and storage == "f32" else 0.0
    c = _frame("", W, H, _levels(W, H), rng.randint(2, 12), rng.randint(10, 100),
               model=rng.choice(["kb", "equidistant", "ucm", "eucm"]), reg=reg, storage=storage,
               accel=accel, deriv=rng.choice(["forward", "central"]), graph=rng.choice([0, 1, 1]),
               start=rng.choice(["cold", "cold", "host", "continue", "init"]))
    del c["name"]
    if reg == "tgv":                           # no more than the largest listed case
        c["warps"] = min(c["warps"], 6)
        c["iters"] = min(c["iters"], 50)
    return c


def _batch_sizes(case):
    s = [int(v) for v in case["sizes"].split(",")]
    return [s[i % len(s)] for i in range(case["pairs"])]


def _level_pixels(W, H, levels):
    n = 0
    for _ in range(levels):
        n += W * H
        W, H = (W + 1) // 2, (H + 1) // 2
    return n


def work(case):
    """Inputs read once and outputs written once; the arithmetic of the
    iterations (41 operations per pixel for Huber-TV, 95 for TGV)."""
    k = case["kind"]
    if k == "iterate":
        n = case["W"] * case["H"]
        # I0, mask, I_u, rho0, u_w in; u, p in and out
        return dict(bytes=n * (4 * 4 + 1 + 2 * 3 * 4), flops=41 * n * case["iters"])
    if k == "repose":
        n = case["W"] * case["H"]
        # I1 in; the pre-rotated image and gamma' out; about 1000 operations
        # for the three camera maps of a pixel
        return dict(bytes=n * (4 + 4 + 8), flops=1000 * n)
    if k == "batch":
        sizes = _batch_sizes(case)
        px = sum(s * s for s in sizes)
        it = sum(_level_pixels(s, s, _levels(s, s)) for s in sizes) * case["warps"] * case["iters"]
        return dict(bytes=16 * px, flops=41 * it)
    n = case["W"] * case["H"]
    lv = case["levels"] if case["start"] in ("cold", "host") else 1
    it = _level_pixels(case["W"], case["H"], lv) * case["warps"] * case["iters"]
    extra = {"init": 4, "continue": 12}.get(case["start"], 0)
    return dict(bytes=(16 + extra) * n, flops=(95 if case["reg"] == "tgv" else 41) * it)


# ------------------------------------------------------------------ cameras (64 bits)

def _radius(cam, th):
    m, k = cam["model"], cam["k"]
    if m == "equidistant":
        return th
    if m == "ucm":
        return torch.sin(th) / (torch.cos(th) + k[0])
    if m == "eucm":
        s, c = torch.sin(th), torch.cos(th)
        return s / (k[0] * torch.sqrt(k[1] * s * s + c * c) + (1.0 - k[0]) * c)
    t2 = th * th
    return th * (1 + t2 * (k[0] + t2 * (k[1] + t2 * (k[2] + t2 * k[3]))))


def _radius_slope(cam, th):
    m, k = cam["model"], cam["k"]
    if m == "equidistant":
        return torch.ones_like(th)
    if m == "ucm":
        c = torch.cos(th)
        return (1 + k[0] * c) / (c + k[0]) ** 2
    if m == "eucm":
        s, c = torch.sin(th), torch.cos(th)
        q = torch.sqrt(k[1] * s * s + c * c)
        den = k[0] * q + (1 - k[0]) * c
        dden = k[0] * s * c * (k[1] - 1) / q - (1 - k[0]) * s
        return (c * den - s * dden) / den ** 2
    t2 = th * th
    return 1 + t2 * (3 * k[0] + t2 * (5 * k[1] + t2 * (7 * k[2] + t2 * 9 * k[3])))


def _half(cam):
    return math.radians(cam["fov_deg"]) / 2


def _rmax(cam):
    return float(_radius(cam, torch.tensor(_half(cam), dtype=F64)))


def _grid(W, H):
    y, x = torch.meshgrid(torch.arange(H, dtype=F64, device=DEV),
                          torch.arange(W, dtype=F64, device=DEV), indexing="ij")
    return x, y


def _unproject(cam, x, y):
    """Unit rays of pixel positions and theta; radii beyond the FOV clamp."""
    mx, my = (x - cam["cx"]) / cam["fx"], (y - cam["cy"]) / cam["fy"]
    rn = torch.sqrt(mx * mx + my * my)
    if cam["model"] == "equidistant":
        th = rn
    else:
        lo, hi = torch.zeros_like(rn), torch.full_like(rn, _half(cam))
        for _ in range(56):
            mid = 0.5 * (lo + hi)
            below = _radius(cam, mid) < rn
            lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
        th = 0.5 * (lo + hi)
    safe = torch.where(rn > 0, rn, torch.ones_like(rn))
    s = torch.sin(th)
    ray = torch.stack([torch.where(rn > 0, s * mx / safe, 0 * s),
                       torch.where(rn > 0, s * my / safe, 0 * s), torch.cos(th)], -1)
    return ray, th, rn


def _project(cam, X):
    rho = torch.hypot(X[..., 0], X[..., 1])
    r = _radius(cam, torch.atan2(rho, X[..., 2]))
    safe = torch.where(rho > 0, rho, torch.ones_like(rho))
    q = torch.where(rho > 0, r / safe, 0 * r)
    return cam["fx"] * q * X[..., 0] + cam["cx"], cam["fy"] * q * X[..., 1] + cam["cy"]


def _mask(cam, W, H):
    x, y = _grid(W, H)
    return torch.hypot((x - cam["cx"]) / cam["fx"], (y - cam["cy"]) / cam["fy"]) <= _rmax(cam)


def _level_cam(cam, l):
    s = 0.5 ** l
    return dict(cam, fx=cam["fx"] * s, fy=cam["fy"] * s, cx=(cam["cx"] + 0.5) * s - 0.5,
                cy=(cam["cy"] + 0.5) * s - 0.5)


# ------------------------------------------------------------------ rigs and scenes

def _rotation(axis, angle):
    a = np.asarray(axis, dtype=np.float64)
    a = a / np.linalg.norm(a)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    return np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * K @ K


def _rig(rng, model, W, H):
    """A lens whose FOV circle about fills the image, and a second camera 0.1
    m to the right (turned by up to 2 degrees except for the plain lens)."""
    n = min(W, H)
    if model == "equidistant":
        k, fov, f = [0.0] * 4, 180.0, n * 80.0 / 256.0
    elif model == "kb":
        fov, f = 190.0, n * 320.0 / 1024.0
        while True:                              # r(theta) has to increase
            k = rng.uniform(-0.05, 0.05, 4).tolist()
            th = torch.linspace(0.0, math.radians(fov) / 2, 10000, dtype=F64)
            if bool((torch.diff(_radius(dict(model=model, k=k), th)) > 0).all()):
                break
    else:
        k = [rng.uniform(0.7, 0.95), 0, 0, 0] if model == "ucm" else \
            [rng.uniform(0.5, 0.65), rng.uniform(1.0, 1.2), 0, 0]
        fov = 190.0
        f = 0.47 * n / _rmax(dict(model=model, k=k, fov_deg=fov))
    cam = dict(model=model, fx=f, fy=f, cx=(W - 1) / 2.0, cy=(H - 1) / 2.0,
               k=[float(v) for v in k], fov_deg=fov)
    R = np.eye(3) if model == "equidistant" else \
        _rotation(rng.normal(size=3), math.radians(rng.uniform(0.2, 2.0)))
    return cam, R, np.array([0.1, 0.0, 0.0])


def _waves(rng, fmax):
    d = rng.normal(size=(16, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    freq = fmax * 2.0 ** (-6 * rng.uniform(0, 1, 16))
    return dict(k=torch.tensor(2 * math.pi * d * freq[:, None], device=DEV),
                amp=torch.tensor(rng.uniform(0.5, 1.0, 16) * np.sqrt(fmax / freq), device=DEV),
                phase=torch.tensor(rng.uniform(0, 2 * math.pi, 16), device=DEV),
                base=float(rng.uniform(0.35, 0.65)))


def _texture(t, P):
    s = torch.sin(P @ t["k"].T + t["phase"]) @ t["amp"] / t["amp"].sum()
    return (t["base"] + 0.45 * s).clamp(0, 1)


def _scene(rng, f, n=12, far=8.0):
    objs = []
    for i in range(n):
        cz, ph = rng.uniform(math.cos(math.radians(70)), 1.0), rng.uniform(0, 2 * math.pi)
        sz = math.sqrt(1 - cz * cz)
        view = np.array([sz * math.cos(ph), sz * math.sin(ph), cz])
        dist = rng.uniform(0.8, far)
        tex = _waves(rng, 0.25 * f / dist)
        if i % 2:
            objs.append(("ball", dist * view, rng.uniform(0.15, 0.45) * min(dist, 2.0), tex))
        else:
            tilt = rng.normal(size=3) * 0.25
            nrm = -(view + tilt) / np.linalg.norm(view + tilt)
            u = np.cross(nrm, [0.0, 1.0, 0.0])
            u /= np.linalg.norm(u)
            objs.append(("plane", dist * view, (nrm, u, np.cross(nrm, u), rng.uniform(0.5, 1.5, 2)),
                         tex))
    return objs, far, _waves(rng, 0.25 * f / far)


def _render(scene, cam, R, C, W, H, gen):
    """The image of a camera at C with world-to-camera rotation R."""
    objs, far, bg = scene
    x, y = _grid(W, H)
    ray, _, rn = _unproject(cam, x, y)
    inside = rn <= _rmax(cam)
    d = (ray @ torch.tensor(R, dtype=F64, device=DEV)).reshape(-1, 3)
    o = torch.tensor(np.asarray(C, dtype=np.float64), device=DEV)
    od = d @ o
    best = -od + torch.sqrt(od * od - (o @ o - far * far))
    which = torch.full(best.shape, -1, dtype=torch.int32, device=DEV)
    for i, (kind, c, a, _) in enumerate(objs):
        c = torch.tensor(c, device=DEV)
        if kind == "ball":
            oc = o - c
            b = d @ oc
            disc = b * b - (oc @ oc - a * a)
            s = -b - torch.sqrt(disc.clamp(min=0))
            hit = (disc >= 0) & (s > 1e-6) & (s < best)
        else:
            nrm, u, v, half = (torch.tensor(np.asarray(q), device=DEV) for q in a)
            den = d @ nrm
            s = ((c - o) @ nrm) / torch.where(den.abs() > 1e-12, den, torch.full_like(den, 1e-12))
            rel = o + s[:, None] * d - c
            hit = ((rel @ u).abs() <= half[0]) & ((rel @ v).abs() <= half[1]) & (s > 1e-6) & (s < best)
        best = torch.where(hit, s, best)
        which = torch.where(hit, torch.full_like(which, i), which)
    img = _texture(bg, o + best[:, None] * d)
    for i, (_, _, _, tex) in enumerate(objs):
        at = (which == i).nonzero()[:, 0]
        img[at] = _texture(tex, o + best[at, None] * d[at])
    img = img.reshape(H, W)
    noise = 0.01 * torch.randn(H, W, generator=gen, dtype=F64, device=DEV)
    return torch.where(inside, (img + noise).clamp(0, 1), 0 * img).float().contiguous()


def _inputs(model, W, H, seed, frames=1):
    """cam, R, t (X1 = R X0 + t) and the pairs of `frames` frames of the rig
    moving at walking speed."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    cam, R, C1 = _rig(rng, model, W, H)
    scene = _scene(rng, cam["fx"])
    v, wv = rng.normal(size=3) * 0.008, rng.normal(size=3) * 0.002
    pairs = []
    for k in range(frames):
        o, ang = k * v, k * float(np.linalg.norm(wv))
        R0 = _rotation(wv, ang) if k else np.eye(3)
        pairs.append((_render(scene, cam, R0, o, W, H, gen),
                      _render(scene, cam, R @ R0, o + R0.T @ C1, W, H, gen)))
    return cam, R, -R @ C1, pairs


# ------------------------------------------------------------------ prepare, run

def _params(case):
    p = dict(lam=LAM, huber_eps=EPS, use_graph=case.get("graph", 1), storage=case["storage"],
             regularizer=case.get("reg", "huber_tv"), deriv=case.get("deriv", "forward"))
    if case.get("accel", 0.0) > 0:
        p.update(accel_gamma=case["accel"], precond=0)
    return p


def _init_disparity(cam, W, H):
    """A smooth disparity of a few pixels, as a coarser sensor would give."""
    x, y = _grid(W, H)
    d = 2.0 + 1.5 * torch.sin(x * (4.0 / W)) * torch.cos(y * (3.0 / H))
    return torch.where(_mask(cam, W, H), d, 0 * d).float().contiguous()


def _iterate_inputs(case, seed):
    """The linearisation of one warp: I_u about an image derivative, the
    residual of a smooth true disparity of up to 0.3 px plus noise."""
    W, H = case["W"], case["H"]
    cam, _, _, ((I0, _),) = _inputs("equidistant", W, H, seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 1)
    x, y = _grid(W, H)
    Iu = torch.roll(I0, -1, 1) - I0
    true = 0.2 + 0.1 * torch.sin(x * (5.0 / W) + y * (3.0 / H))
    rho0 = (-Iu.double() * true + 0.01 * torch.randn(H, W, generator=gen, dtype=F64, device=DEV))
    m = _mask(cam, W, H)
    z = torch.zeros(H, W, device=DEV)
    return (I0, m.to(torch.uint8).contiguous(), torch.where(m, Iu, z).contiguous(),
            torch.where(m, rho0.float(), z).contiguous(), z)


def _fresh(W, H):
    return torch.empty(H, W, device=DEV), torch.empty(H, W, device=DEV)


def prepare(case, seed):
    k = case["kind"]
    if k == "iterate":
        I0, m, Iu, rho0, uw = _iterate_inputs(case, seed)
        prm = fsb.default_params(lam=LAM, huber_eps=EPS)
        return dict(case=case, I0=I0, m=m, Iu=Iu, rho0=rho0, uw=uw, prm=prm,
                    u=torch.zeros_like(I0), p=torch.zeros(2, case["H"], case["W"], device=DEV),
                    lib=fsb.load_library())
    if k == "batch":
        sizes, solvers, I0, I1 = _batch_sizes(case), [], [], []
        for i, s in enumerate(sizes):
            cam, R, t, ((a, b),) = _inputs("kb", s, s, seed * 1000 + i)
            solvers.append(fsb.Solver(cam, cam, R, t, s, s, _levels(s, s), **_params(case)))
            I0.append(a)
            I1.append(b)
        out = [_fresh(s, s) for s in sizes]
        return dict(case=case, batch=fsb.Batch(solvers, finest_limit=case["finest"]), I0=I0, I1=I1,
                    disp=[o[0] for o in out], depth=[o[1] for o in out])
    W, H = case["W"], case["H"]
    if k == "repose":
        cam, R, t, ((_, I1),) = _inputs("kb", W, H, seed)
        s = fsb.Solver(cam, cam, np.eye(3), np.array([-0.1, 0.0, 0.0]), W, H, case["levels"])
        return dict(case=case, s=s, R=R, t=t, I1=I1)
    start = case["start"]
    cam, R, t, pairs = _inputs(case["model"], W, H, seed, 2 if start == "continue" else 1)
    s = fsb.Solver(cam, cam, R, t, W, H, case["levels"], **_params(case))
    if case["tune"]:
        s.autotune(case["iters"])
    disp, depth = _fresh(W, H)
    st = dict(case=case, s=s, I0=pairs[-1][0], I1=pairs[-1][1], disp=disp, depth=depth)
    if start == "init":
        st["init"] = _init_disparity(cam, W, H)
    elif start == "continue":
        st["first"] = pairs[0]
        s.solve(*pairs[0], 4, 20, disp=disp, depth=depth)
    elif start == "host":
        for key in ("I0", "I1", "disp", "depth"):
            st[key] = torch.empty(H, W).pin_memory().copy_(st[key])
    return st


def run(st):
    case = st["case"]
    k = case["kind"]
    if k == "iterate":
        st["u"].zero_()
        st["p"].zero_()
        ptr = lambda a: ctypes.c_void_p(a.data_ptr())
        code = st["lib"].fs_pd_iterate_noalloc(
            ptr(st["I0"]), ptr(st["m"]), ptr(st["Iu"]), ptr(st["rho0"]), ptr(st["uw"]),
            ptr(st["u"]), ptr(st["p"]), case["W"], case["H"], case["iters"],
            ctypes.byref(st["prm"]), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if code != 0:
            raise RuntimeError(st["lib"].fs_last_error().decode())
        return st["u"], st["p"]
    if k == "batch":
        return st["batch"].solve(st["I0"], st["I1"], case["warps"], case["iters"],
                                 disps=st["disp"], depths=st["depth"])
    s = st["s"]
    if k == "repose":
        s.set_pose(st["R"], st["t"])
        s.prerotate(st["I1"])
        return s.trajectory_field(0), s.read(0, "I1")
    args = (st["I0"], st["I1"], case["warps"], case["iters"])
    if case["start"] == "host":
        return s.solve_host(*args, disp=st["disp"], depth=st["depth"])
    if case["start"] == "continue":
        return s.solve_continue(*args, disp=st["disp"], depth=st["depth"])
    return s.solve(*args, init=st.get("init"), disp=st["disp"], depth=st["depth"])


# ------------------------------------------------------------------ the method in 64 bits

def _tap(img, yi, xi):
    return img[yi, xi] if img.dim() == 2 else img[:, yi, xi]


def _bilinear(img, x, y):
    H, W = img.shape
    x, y = x.clamp(0, W - 1), y.clamp(0, H - 1)
    x0 = x.floor().clamp(max=max(W - 2, 0)).long()
    y0 = y.floor().clamp(max=max(H - 2, 0)).long()
    x1, y1 = (x0 + 1).clamp(max=W - 1), (y0 + 1).clamp(max=H - 1)
    ax, ay = x - x0, y - y0
    top = img[y0, x0] + ax * (img[y0, x1] - img[y0, x0])
    bot = img[y1, x0] + ax * (img[y1, x1] - img[y1, x0])
    return top + ay * (bot - top)


def _keys(s):
    s, a = s.abs(), -0.5
    inner = ((a + 2) * s - (a + 3)) * s * s + 1
    outer = ((a * s - 5 * a) * s + 8 * a) * s - 4 * a
    return torch.where(s <= 1, inner, torch.where(s < 2, outer, 0 * s))


def _bicubic(f, x, y):
    """A (2, H, W) field at (x, y), Keys' kernel with a = -1/2."""
    _, H, W = f.shape
    x, y = x.clamp(0, W - 1), y.clamp(0, H - 1)
    xi, yi = x.floor().long(), y.floor().long()
    out = 0.0
    for j in range(-1, 3):
        wy, row = _keys(y - (yi + j)), 0.0
        for i in range(-1, 3):
            row = row + _keys(x - (xi + i)) * _tap(f, (yi + j).clamp(0, H - 1), (xi + i).clamp(0, W - 1))
        out = out + wy * row
    return out


def _trajectory(cam, tp, W, H, M):
    """The image velocity of a point on each pixel's ray moving along tp,
    normalised; by the chain rule through theta and the azimuth."""
    x, y = _grid(W, H)
    ray, th, rn = _unproject(cam, x, y)
    t = tp / np.linalg.norm(tp)
    mx, my = (x - cam["cx"]) / cam["fx"], (y - cam["cy"]) / cam["fy"]
    safe = torch.where(rn > 0, rn, torch.ones_like(rn))
    ux = torch.where(rn > 0, mx / safe, torch.ones_like(rn))
    uy = torch.where(rn > 0, my / safe, torch.zeros_like(rn))
    rho, z = torch.sin(th), torch.cos(th)
    rad = _radius_slope(cam, th) * (z * (ux * t[0] + uy * t[1]) - rho * t[2])
    cross = ux * t[1] - uy * t[0]
    scale = torch.where(rho > 1e-12, _radius(cam, th) / torch.where(rho > 1e-12, rho, 1 + 0 * rho),
                        1.0 / z)
    slope0 = float(_radius_slope(cam, torch.zeros(1, dtype=F64)))
    scale = torch.where(rho > 1e-12, scale, torch.full_like(rho, slope0))
    vx = cam["fx"] * (rad * ux - scale * uy * cross)
    vy = cam["fy"] * (rad * uy + scale * ux * cross)
    n = torch.hypot(vx, vy)
    ok = M & (n >= 1e-3)
    n = torch.where(ok, n, torch.ones_like(n))
    return torch.stack([torch.where(ok, vx / n, 0 * n), torch.where(ok, vy / n, 0 * n)])


def _prerotated(cam, R, W, H, M, I1):
    x, y = _grid(W, H)
    ray, _, _ = _unproject(cam, x, y)
    qx, qy = _project(cam, ray @ torch.tensor(R.T.copy(), device=DEV))
    return _bilinear(I1, torch.where(M, qx, x), torch.where(M, qy, y))


def _down(img, M):
    H, W = img.shape
    h, w = (H + 1) // 2, (W + 1) // 2
    pad = (0, 2 * w - W, 0, 2 * h - H)
    f = torch.nn.functional.pad

    def cells(a):
        return f(a, pad).reshape(h, 2, w, 2).sum((1, 3))
    m = M.double()
    n_in, n_all = cells(m), cells(torch.ones_like(img))
    return torch.where(n_in > 0, cells(img * m) / n_in.clamp(min=1), cells(img) / n_all)


def _up(v, Mc, M):
    H, W = M.shape
    h, w = v.shape
    x, y = _grid(W, H)
    X, Y = ((x + 0.5) / 2 - 0.5).clamp(0, w - 1), ((y + 0.5) / 2 - 0.5).clamp(0, h - 1)
    x0, y0 = X.floor().clamp(max=max(w - 2, 0)).long(), Y.floor().clamp(max=max(h - 2, 0)).long()
    x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
    ax, ay = X - x0, Y - y0
    num, den = 0.0, 0.0
    for g, yy, xx in (((1 - ax) * (1 - ay), y0, x0), (ax * (1 - ay), y0, x1),
                      ((1 - ax) * ay, y1, x0), (ax * ay, y1, x1)):
        g = g * Mc[yy, xx]
        num, den = num + g * v[yy, xx], den + g
    ok = M & (den > 0)
    return torch.where(ok, 2 * num / torch.where(ok, den, torch.ones_like(den)), 0 * num)


def _grad(u, m1, m2):
    return (torch.nn.functional.pad(u[:, 1:] - u[:, :-1], (0, 1)) * m1,
            torch.nn.functional.pad(u[1:] - u[:-1], (0, 0, 0, 1)) * m2)


def _div(a, b, m1, m2):
    a, b = a * m1, b * m2
    d = a + b
    d[:, 1:] -= a[:, :-1]
    d[1:] -= b[:-1]
    return d


def _tensor_steps(I0, M, precond):
    """T^1/2 = [[a, b], [b, c]], the difference masks and the diagonal steps."""
    m1, m2 = torch.zeros_like(I0), torch.zeros_like(I0)
    m1[:, :-1] = (M[:, :-1] & M[:, 1:]).double()
    m2[:-1] = (M[:-1] & M[1:]).double()
    g1, g2 = _grad(I0, m1, m2)
    l1, l2 = torch.zeros_like(I0), torch.zeros_like(I0)
    l1[:, 1:], l2[1:] = m1[:, :-1], m2[:-1]
    b1, b2 = torch.zeros_like(I0), torch.zeros_like(I0)
    b1[:, 1:], b2[1:] = g1[:, :-1], g2[:-1]
    gx, gy = (g1 + b1) / (m1 + l1).clamp(min=1), (g2 + b2) / (m2 + l2).clamp(min=1)
    mag = torch.hypot(gx, gy)
    big = mag >= 1e-12
    safe = torch.where(big, mag, torch.ones_like(mag))
    nx, ny = torch.where(big, gx / safe, 1 + 0 * mag), torch.where(big, gy / safe, 0 * mag)
    e = torch.exp(-BETA * mag ** ETA)
    one, zero = torch.ones_like(e), torch.zeros_like(e)
    a = torch.where(M, 1 - (1 - e) * nx * nx, one)
    b = torch.where(M, -(1 - e) * nx * ny, zero)
    c = torch.where(M, 1 - (1 - e) * ny * ny, one)
    row = torch.maximum(2 * (a.abs() * m1 + b.abs() * m2), 2 * (b.abs() * m1 + c.abs() * m2))
    if not precond:
        s = torch.full_like(a, 8.0 ** -0.5)
        return a, b, c, m1, m2, torch.where(M, s, zero), s, row
    left, upper = (a.abs() + b.abs()) * m1, (b.abs() + c.abs()) * m2
    col = left + upper
    col[:, 1:] += left[:, :-1]
    col[1:] += upper[:-1]
    tau = torch.where(M & (col > 0), 1 / torch.where(col > 0, col, one), zero)
    sig = torch.where(row > 0, 1 / torch.where(row > 0, row, one), zero)
    return a, b, c, m1, m2, tau, sig, row


def _shrink(uh, Iu, rho0, uw, tau):
    safe = torch.where(Iu != 0, Iu, torch.ones_like(Iu))
    step = (tau * LAM * Iu).abs()
    r = torch.where(Iu != 0, -(rho0 + Iu * (uh - uw)) / safe, 0 * Iu)
    return uh + torch.minimum(torch.maximum(r, -step), step)


def _huber_iterations(st, lv, Iu, rho0, uw, iters, accel):
    a, b, c, m1, m2, tau, sig, _ = lv
    u, p1, p2 = st["u"], st["p1"], st["p2"]
    ub, t, s, theta = u, 8.0 ** -0.5, 8.0 ** -0.5, 1.0
    for _ in range(iters):
        if accel > 0:
            theta = 1 / math.sqrt(1 + 2 * accel * t)
            tau, sig = torch.where(tau > 0, torch.full_like(tau, t), 0 * tau), torch.full_like(sig, s)
            t, s = theta * t, s / theta
        g1, g2 = _grad(ub, m1, m2)
        q1 = (p1 + sig * (a * g1 + b * g2)) / (1 + sig * EPS)
        q2 = (p2 + sig * (b * g1 + c * g2)) / (1 + sig * EPS)
        n = torch.hypot(q1, q2).clamp(min=1)
        p1, p2 = q1 / n, q2 / n
        uh = u + tau * _div(a * p1 + b * p2, b * p1 + c * p2, m1, m2)
        un = _shrink(uh, Iu, rho0, uw, tau)
        ub, u = un + theta * (un - u), un
    st.update(u=u, p1=p1, p2=p2)


def _tgv_iterations(st, lv, Iu, rho0, uw, iters, M):
    a, b, c, m1, m2, tau, _, row = lv
    m = M.double()
    sp, sq = m / (row + 1), 0.5 * m
    col = m1 + m2
    col[:, 1:] += m1[:, :-1]
    col[1:] += m2[:-1]
    tv = m / (1 + col)
    u, v1, v2 = st["u"], st["v1"], st["v2"]
    ub, w1, w2 = u, v1, v2
    p1, p2, q = st["p1"], st["p2"], st["q"]
    for _ in range(iters):
        g1, g2 = _grad(ub, m1, m2)
        r1, r2 = p1 + sp * (a * g1 + b * g2 - w1), p2 + sp * (b * g1 + c * g2 - w2)
        n = (torch.hypot(r1, r2) / ALPHA1).clamp(min=1)
        p1, p2 = r1 / n, r2 / n
        q = [x + sq * j for x, j in zip(q, _grad(w1, m1, m2) + _grad(w2, m1, m2))]
        n = ((q[0] ** 2 + q[1] ** 2 + q[2] ** 2 + q[3] ** 2).sqrt() / ALPHA0).clamp(min=1)
        q = [x / n for x in q]
        un = _shrink(u + tau * _div(a * p1 + b * p2, b * p1 + c * p2, m1, m2), Iu, rho0, uw, tau)
        ub, u = 2 * un - u, un
        n1, n2 = v1 + tv * (p1 + _div(q[0], q[1], m1, m2)), v2 + tv * (p2 + _div(q[2], q[3], m1, m2))
        w1, v1, w2, v2 = 2 * n1 - v1, n1, 2 * n2 - v2, n2
    st.update(u=u, v1=v1, v2=v2, p1=p1, p2=p2, q=q)


def _level(case, I0, I1, cam, tp, M, u, w, warps, iters):
    """The warps of one level; returns u and w."""
    H, W = I0.shape
    x, y = _grid(W, H)
    gamma = _trajectory(cam, tp, W, H, M)
    accel, tgv = case.get("accel", 0.0), case.get("reg") == "tgv"
    lv = _tensor_steps(I0, M, not accel > 0)
    z = torch.zeros_like(u)
    st = dict(u=u, p1=z, p2=z, v1=z, v2=z, q=[z] * 4)
    for _ in range(warps):
        g = _bicubic(gamma, x + w[0], y + w[1])
        n = torch.hypot(g[0], g[1])
        ok = M & (n >= 1e-6)
        g = torch.where(ok, g / torch.where(ok, n, torch.ones_like(n)), 0 * g)
        Iw = _bilinear(I1, x + w[0], y + w[1])
        ahead = _bilinear(I1, x + w[0] + g[0], y + w[1] + g[1])
        Iu = ahead - Iw if case.get("deriv", "forward") == "forward" else \
            0.5 * (ahead - _bilinear(I1, x + w[0] - g[0], y + w[1] - g[1]))
        Iu, rho0, uw = torch.where(M, Iu, z), torch.where(M, Iw - I0, z), st["u"]
        if tgv:
            _tgv_iterations(st, lv, Iu, rho0, uw, iters, M)
        else:
            _huber_iterations(st, lv, Iu, rho0, uw, iters, accel)
        du = torch.where(M, (st["u"] - uw).clamp(-DU, DU), z)
        st["u"] = uw + du
        w = w + du * g
    return st["u"], w


def _walk(cam, tp, M, d):
    """w of a given disparity: equal steps of at most DU along gamma'."""
    H, W = d.shape
    x, y = _grid(W, H)
    gamma = _trajectory(cam, tp, W, H, M)
    n = torch.ceil(d.float().abs() / torch.tensor(DU, dtype=torch.float32)).double()
    step = d / n.clamp(min=1)
    w = torch.zeros(2, H, W, dtype=F64, device=DEV)
    for k in range(int(n.max())):
        g = _bicubic(gamma, x + w[0], y + w[1])
        r = torch.hypot(g[0], g[1])
        ok = (n > k) & (r >= 1e-6)
        w = w + torch.where(ok, step * g / torch.where(ok, r, torch.ones_like(r)), 0 * g)
    return w


def _solve(case, cam, R, t, I0, I1, levels, warps, iters, start=None):
    """Disparity and warp field of one pair; start: (u, w) of the finest
    level, which then runs alone."""
    H, W = I0.shape
    I0 = I0.to(DEV).double()
    tp = R.T @ t
    cams = [_level_cam(cam, l) for l in range(levels)]
    sizes = [(W, H)]
    for _ in range(1, levels):
        sizes.append(((sizes[-1][0] + 1) // 2, (sizes[-1][1] + 1) // 2))
    M = [_mask(cams[l], *sizes[l]) for l in range(levels)]
    A, B = [I0], [_prerotated(cam, R, W, H, M[0], I1.to(DEV).double())]
    if start is not None:
        return _level(case, A[0], B[0], cam, tp, M[0], *start, warps, iters)
    for l in range(1, levels):
        A.append(_down(A[-1], M[l - 1]))
        B.append(_down(B[-1], M[l - 1]))
    u = torch.zeros_like(A[-1])
    w = torch.zeros(2, *u.shape, dtype=F64, device=DEV)
    for l in range(levels - 1, -1, -1):
        if l < levels - 1:
            u, w = _up(u, M[l + 1], M[l]), torch.stack([_up(v, M[l + 1], M[l]) for v in w])
        u, w = _level(case, A[l], B[l], cams[l], tp, M[l], u, w, warps, iters)
    return u, w


def exact(case, seed):
    """Disparities, fields and states.  The range has no value to hold to: it
    is unbounded where the parallax passes through 0."""
    k = case["kind"]
    if k == "iterate":
        I0, m, Iu, rho0, uw = _iterate_inputs(case, seed)
        lv = _tensor_steps(I0.double(), m > 0, True)
        z = torch.zeros_like(uw, dtype=F64)
        st = dict(u=z, p1=z, p2=z)
        _huber_iterations(st, lv, Iu.double(), rho0.double(), uw.double(), case["iters"], 0.0)
        return st["u"], torch.stack([st["p1"], st["p2"]])
    if k == "batch":
        out = []
        for i, s in enumerate(_batch_sizes(case)):
            cam, R, t, ((a, b),) = _inputs("kb", s, s, seed * 1000 + i)
            out.append(_solve(case, cam, R, t, a, b, _levels(s, s), case["warps"], case["iters"])[0])
        return out, None
    W, H = case["W"], case["H"]
    if k == "repose":
        cam, R, t, ((_, I1),) = _inputs("kb", W, H, seed)
        M = _mask(cam, W, H)
        return _trajectory(cam, R.T @ t, W, H, M), _prerotated(cam, R, W, H, M, I1.double())
    start = case["start"]
    cam, R, t, pairs = _inputs(case["model"], W, H, seed, 2 if start == "continue" else 1)
    begin = None
    if start == "init":
        d = _init_disparity(cam, W, H).double()
        begin = (d, _walk(cam, R.T @ t, _mask(cam, W, H), d))
    elif start == "continue":
        begin = _solve(case, cam, R, t, *pairs[0], case["levels"], 4, 20)
    u, _ = _solve(case, cam, R, t, *pairs[-1], case["levels"], case["warps"], case["iters"], begin)
    return u, None
