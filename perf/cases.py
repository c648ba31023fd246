"""Performance cases of the scene-space gather-and-filter library, through its public Python entry points.

listed() names the fixed cases, draw(rng) gives more of the same ranges, prepare(case, seed) loads
the clips a user's program has loaded, run(state) is one call such a program makes (gather and read
back, superres, plan launch, reload, gradient of a training batch), work(case) is what one pass has
to read, write and compute, and exact(case, seed) is the same result in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_2102_03011_gb300 as ss

RADIUS_REL = 0.005  # of the clip's median depth, the library's default
SIGMA_RGB = 40.0 / 255.0
SIGMA_F = 6.0


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the tiny workload: a whole 160 x 90 clip, every frame over all frames; a preview, where latency and launches count
        dict(name="tiny_clip", op="window", mode="denoise", scene="planes", W=160, H=90, F=16, T=15, k=5, O=0, n=16, f16=False),
        # an ordinary 720p denoising call over +-15 frames
        dict(name="hd_denoise", op="window", mode="denoise", scene="room", W=1280, H=720, F=34, T=15, k=7, O=15, n=4, f16=False),
        # the headline: 1080p denoising over +-30 frames
        dict(name="fhd_denoise", op="window", mode="denoise", scene="room", W=1920, H=1080, F=64, T=30, k=7, O=30, n=4, f16=False),
        # deblurring of a ragged frame size with FP16 colour and a 5 x 5 window
        dict(name="ragged_deblur", op="window", mode="deblur", scene="room", W=853, H=479, F=23, T=10, k=5, O=10, n=3, f16=True),
        # 1080p virtual aperture over +-30 frames with FP16 colour, one refocused frame
        dict(name="fhd_aperture", op="aperture", scene="room", W=1920, H=1080, F=61, T=30, k=7, O=30, n=1, f16=True),
        # uneven clips, all their frames, in one captured plan
        dict(name="mixed_plan", op="plan", scene="room", shapes="640x360x30,854x480x20,1280x720x8", T=15, k=7, f16=True),
        # 1080p learned weighting over +-6 frames (the learned filter's fast operating point)
        dict(name="fhd_learned", op="learned", scene="room", W=1920, H=1080, F=14, T=6, k=7, O=6, n=2, f16=False),
        # the paper's own frustum gather at 720p over +-15 frames
        dict(name="hd_frustum", op="frustum", mode="denoise", scene="room", W=1280, H=720, F=31, T=15, O=15, n=1, f16=False),
        # super-resolution of a 640 x 360 clip to 1080p over +-30 frames
        dict(name="superres_x3", op="superres", scene="room", W=640, H=360, F=61, T=30, O=30, n=1, scale=3, f16=False),
        # inpainting: one box of the scene removed from a 720p frame over +-15 frames
        dict(name="hd_inpaint", op="frustum", mode="inpaint", scene="room", W=1280, H=720, F=31, T=15, O=15, n=1, f16=False),
        # the next shot: a new clip of the same size from device tensors, its cameras, one denoised frame
        dict(name="hd_reload", op="reload", mode="denoise", scene="room", W=1280, H=720, F=31, T=15, k=7, O=15, n=1, f16=False),
        # training: loss and gradient of a 16,384-pixel batch of one 640 x 360 frame
        dict(name="train_grad", op="grad", scene="room", W=640, H=360, F=31, T=15, k=7, O=15, batch=16384, f16=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any operation, sizes over the range of the listed ones (odd ones among them)."""
    op = rng.choice(["window"] * 6 + ["aperture", "plan", "learned", "learned", "frustum", "frustum", "superres", "reload", "grad"])
    f16 = rng.random() < 0.4
    if op == "plan":
        shapes = []
        for _ in range(rng.randint(2, 4)):
            W = _log_int(rng, 96, 1024)
            shapes.append("%dx%dx%d" % (W, max(48, W * 9 // 16 + rng.randint(-9, 9)), rng.randint(6, 20)))
        return dict(op=op, scene="room", shapes=",".join(shapes), T=rng.randint(5, 15), k=rng.choice([5, 7]), f16=f16)
    W = _log_int(rng, 128, 1920 if op in ("window", "learned") else 1280)
    H = max(64, W * 9 // 16 + rng.randint(-12, 12))
    H = min(H, 1080)
    T = _log_int(rng, 3, 30 if op != "learned" else 10)
    c = dict(op=op, scene="room", W=W, H=H, F=0, T=T, O=T, n=1, f16=f16)
    if op in ("window", "reload"):
        c["mode"] = rng.choice(["denoise", "denoise", "denoise", "mean", "deblur", "shutter"]) if op == "window" else "denoise"
        c["k"] = rng.choice([3, 5, 7, 7, 7, 9])
        cap = 1920 * 1080 * 4 * 61 * 49 // 2
        c["n"] = max(1, min(rng.randint(1, 6) if op == "window" else 1, cap // (W * H * (2 * T + 1) * c["k"] ** 2)))
    elif op == "aperture":
        c["k"] = 7
    elif op == "learned":
        c["k"], c["n"] = rng.choice([5, 7, 7]), rng.randint(1, 2)
    elif op == "frustum":
        c["mode"] = rng.choice(["denoise", "mean", "inpaint", "semi"])
        c["T"] = c["O"] = min(T, 15)
    elif op == "superres":
        c["scale"] = rng.choice([2, 3])
        c["W"], c["H"] = max(96, W // 2), max(54, H // 2)
    elif op == "grad":
        c["k"], c["batch"] = 7, _log_int(rng, 1024, 16384)
        c["W"], c["H"] = max(96, W // 2), max(54, H // 2)
    c["F"] = 2 * c["T"] + c["n"]
    return c


# ---------------------------------------------------------------- inputs

def _rot(w):
    th = float(np.linalg.norm(w))
    if th < 1e-12:
        return np.eye(3)
    k = np.asarray(w) / th
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    return np.eye(3) + math.sin(th) * K + (1 - math.cos(th)) * (K @ K)


def _scene(kind, rng):
    """Surfaces: (point, rows of axes, half sizes or None for an unbounded plane / third half 0 for a rectangle)."""
    I = np.eye(3)
    if kind == "planes":
        tilt = _rot([0, math.radians(30), 0])
        return [((0, 0, 7.5), I, None), ((0, 1.2, 0), I[[0, 2, 1]], None), ((0.4, -0.1, 4.0), tilt.T, (1.0, 0.7, 0.0))]
    tilt = _rot([0, math.radians(40), 0])
    objs = [((0, 0, 12.0 + rng.uniform(-1, 1)), I, None), ((0, 1.5, 0), I[[0, 2, 1]], None), ((0, -2.2, 0), I[[0, 2, 1]], None),
            ((-4.5, 0, 0), I[[2, 1, 0]], None), ((5.0, 0, 0), I[[2, 1, 0]], None), ((-1.8, 0.2, 6.5), tilt.T, (1.0, 1.2, 0.0))]
    for b in range(4):
        half = rng.uniform(0.3, 0.8, 3)
        c = (rng.uniform(-2.5, 2.5), 1.5 - half[1] if b % 2 == 0 else rng.uniform(-1.0, 0.5), rng.uniform(3.5, 9.0))
        objs.append((c, _rot([0, rng.uniform(0, math.pi / 2), 0]).T, tuple(half)))
    return objs


def _cameras(kind, F, rng):
    """True and measured world->camera poses: a steady walk (planes) or a hand-held path, with jitter."""
    true, given = np.empty((F, 3, 4)), np.empty((F, 3, 4))
    ph = rng.uniform(0, 2 * math.pi, 3)
    for f in range(F):
        if kind == "planes":
            C, R = np.array([-0.15 + 0.02 * f, 0.0, 0.0]), _rot(np.radians(0.5) * rng.normal(size=3))
        else:
            s = f / 60.0
            C = np.array([1.2, 0.25, 0.5]) * (np.sin(np.array([1.0, 0.7, 0.5]) * s + ph) - np.sin(ph))
            R = _rot([0, -0.12 * C[0], 0]) @ _rot(np.radians(0.3) * rng.normal(size=3))
        true[f] = np.concatenate([R.T, (-R.T @ C)[:, None]], 1)
        R2, C2 = _rot(0.002 * rng.normal(size=3)) @ R, C + 0.002 * rng.normal(size=3)
        given[f] = np.concatenate([R2.T, (-R2.T @ C2)[:, None]], 1)
    return true, given


def _render(objs, K, w2c, W, H, dev):
    """One frame: colour (H, W, 3) and camera depth (H, W) of the nearest surface."""
    f32 = dict(dtype=torch.float32, device=dev)
    y, x = torch.meshgrid(torch.arange(H, **f32), torch.arange(W, **f32), indexing="ij")
    R, t = w2c[:, :3], w2c[:, 3]
    C = -R.T @ t
    dc = torch.stack([(x - K[0, 2]) / K[0, 0], (y - K[1, 2]) / K[1, 1], torch.ones_like(x)], -1)
    d = dc @ torch.tensor(R, **f32)  # camera -> world directions, unit camera z
    best = torch.full((H, W), 60.0, **f32)
    col = torch.full((H, W, 3), 0.5, **f32)
    for i, (c, A, half) in enumerate(objs):
        At = torch.tensor(np.asarray(A), **f32)
        o = torch.tensor(np.asarray(A) @ (C - np.asarray(c)), **f32)
        q = d @ At.T
        if half is None or half[2] == 0.0:
            s = -o[2] / q[..., 2]
            p = o + s[..., None] * q
            hit = s > 0.05
            if half is not None:
                hit &= (p[..., 0].abs() < half[0]) & (p[..., 1].abs() < half[1])
        else:
            h = torch.tensor(half, **f32)
            a, b = (-h - o) / q, (h - o) / q
            s, far = torch.minimum(a, b).amax(-1), torch.maximum(a, b).amin(-1)
            p = o + s[..., None] * q
            hit = (s < far) & (s > 0.05)
        hit &= s < best
        ph = p * (2.0 + 0.35 * i)
        g = torch.sin(ph[..., 0] * 1.7 + i) * torch.sin(ph[..., 1] * 2.3 + 0.5 * i) + 0.5 * torch.sin(ph.sum(-1) * 5.1) * torch.cos(ph[..., 2] * 3.7)
        tex = torch.stack([0.5 + 0.22 * g, 0.45 + 0.2 * torch.sin(3.1 * g + i), 0.5 + 0.2 * torch.cos(2.3 * g - i)], -1)
        best = torch.where(hit, s, best)
        col = torch.where(hit[..., None], tex, col)
    return col, best


class _Clip:
    """A noisy clip: rgb (F, H, W, 3) and depth (F, H, W) on the GPU, clean colours where asked, cameras on the host."""

    def __init__(self, scene, W, H, F, seed, clean=False):
        dev = torch.device("cuda")
        rng = np.random.default_rng(seed)
        g = torch.Generator(device=dev).manual_seed(seed)
        self.W, self.H, self.F = W, H, F
        self.objs = _scene(scene, rng)
        f = 0.75 * W
        self.K = np.array([[f, 0, (W - 1) / 2], [0, f, (H - 1) / 2], [0, 0, 1.0]])
        true, self.w2c = _cameras(scene, F, rng)
        sd, si = (0.01, 0.03) if scene == "planes" else (0.02, 0.05)
        self.rgb = torch.empty(F, H, W, 3, device=dev)
        self.depth = torch.empty(F, H, W, device=dev)
        self.clean = torch.empty(F, H, W, 3, device=dev) if clean else None
        for j in range(F):
            c, z = _render(self.objs, self.K, true[j], W, H, dev)
            if clean:
                self.clean[j] = c
            self.rgb[j] = c + si * torch.randn(H, W, 3, generator=g, device=dev)
            z = z * (1 + sd * torch.randn(H, W, generator=g, device=dev))
            hole = torch.rand(H, W, generator=g, device=dev) < 0.001  # depth estimates have holes
            self.depth[j] = torch.where(hole, torch.zeros_like(z), z)

    def box(self):
        """World box of one of the scene's boxes, the object that inpainting removes."""
        c, A, half = self.objs[-1]
        ext = np.abs(np.asarray(A)).T @ np.asarray(half) + 0.05
        return tuple(np.asarray(c) - ext) + tuple(np.asarray(c) + ext)


def _mlp(seed):
    rng = np.random.default_rng(seed + 77)
    return (rng.normal(size=(64, 16)) * math.sqrt(2 / 15), 0.1 * rng.normal(size=64), rng.normal(size=(2, 64)) * math.sqrt(2 / 64),
            np.array([0.2, 1.0]))


def _batch(case, seed):
    return np.random.default_rng(seed + 99).integers(0, case["W"] * case["H"], case["batch"]).astype(np.int32)


def _shutter(T):
    return np.exp2(-np.abs(np.arange(-T, T + 1)) / max(1.0, T / 3)).astype(np.float32)


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


# ---------------------------------------------------------------- the library's side

class _State:
    def __init__(self, case):
        self.case, self.ctx, self.plan = case, ss.ssvp_create(torch.cuda.current_device(), torch.cuda.current_stream()), None

    def __del__(self):
        if self.plan is not None:
            ss.ssvp_plan_destroy(self.plan)
        ss.ssvp_destroy(self.ctx)


MODES = dict(denoise=ss.SSVP_MODE_DENOISE, mean=ss.SSVP_MODE_MEAN, deblur=ss.SSVP_MODE_DEBLUR, shutter=ss.SSVP_MODE_SHUTTER,
             inpaint=ss.SSVP_MODE_INPAINT, semi=ss.SSVP_MODE_SEMI)


def _params(case):
    p = ss.ssvp_params_default()
    p.half_window, p.k, p.radius, p.sigma_rgb, p.sigma_f = case["T"], case.get("k", 7), -RADIUS_REL, SIGMA_RGB, SIGMA_F
    op = case["op"]
    if "O" in case:
        p.frame_begin, p.frame_end = case["O"], case["O"] + case.get("n", 1)
    if op in ("window", "reload", "frustum"):
        p.mode = MODES[case["mode"]]
    if op == "frustum":
        p.gather = ss.SSVP_GATHER_FRUSTUM
    if op == "aperture":
        p.mode = ss.SSVP_MODE_APERTURE
    if op == "learned":
        p.mode = ss.SSVP_MODE_LEARNED
    return p


def prepare(case, seed):
    s = _State(case)
    s.p = _params(case)
    fmt = ss.SSVP_COLOUR_F16 if case["f16"] else ss.SSVP_COLOUR_F32
    op = case["op"]
    if op == "plan":
        s.out, ids = [], []
        for i, (W, H, F) in enumerate(_shapes(case)):
            c = _Clip(case["scene"], W, H, F, seed * 31 + i)
            ss.ssvp_load_clip(s.ctx, i, W, H, F, c.rgb, c.depth, colour_fmt=fmt)
            ss.ssvp_set_cameras(s.ctx, i, c.K, 0, c.w2c)
            ss.ssvp_sync(s.ctx)
            s.out.append(torch.zeros(F, H, W, 3, device="cuda"))
            ids.append(i)
        s.plan = ss.ssvp_plan_create(s.ctx, s.p, ids)
        return s
    W, H, F = case["W"], case["H"], case["F"]
    c = _Clip(case["scene"], W, H, F, seed, clean=op == "grad")
    if op != "reload":
        ss.ssvp_load_clip(s.ctx, 0, W, H, F, c.rgb, c.depth, colour_fmt=fmt)
        ss.ssvp_set_cameras(s.ctx, 0, c.K, 0, c.w2c)
    if op == "reload":  # the context holds the previous clip of this size
        s.clip, s.fmt = c, fmt
        ss.ssvp_load_clip(s.ctx, 0, W, H, F, c.rgb.flip(2), c.depth.flip(2), colour_fmt=fmt)
        ss.ssvp_set_cameras(s.ctx, 0, c.K, 0, c.w2c)
    if op in ("learned", "grad"):
        ss.ssvp_set_mlp(s.ctx, *_mlp(seed))
    if op == "grad":
        s.batch, s.clean = _batch(case, seed), c.clean
    if case.get("mode") == "shutter":
        ss.ssvp_set_shutter(s.ctx, _shutter(case["T"]), case["T"])
    if case.get("mode") in ("inpaint", "semi"):
        ss.ssvp_mask_from_box(s.ctx, 0, c.box())
    ss.ssvp_sync(s.ctx)
    z = case.get("scale", 1)
    s.out = torch.zeros(case.get("n", 1), H * z, W * z, 3, device="cuda")
    return s


def run(s):
    c, p, op = s.case, s.p, s.case["op"]
    if op == "plan":
        ss.ssvp_plan_launch(s.plan)
        for i, o in enumerate(s.out):
            ss.ssvp_read_output(s.ctx, i, 0, o.shape[0], o)
        return s.out
    if op == "superres":
        ss.ssvp_superres(s.ctx, p, 0, c["scale"], s.out)
        return s.out
    if op == "grad":
        return ss.ssvp_mlp_grad(s.ctx, p, 0, s.batch, s.clean)
    if op == "reload":
        ss.ssvp_load_clip(s.ctx, 0, c["W"], c["H"], c["F"], s.clip.rgb, s.clip.depth, colour_fmt=s.fmt)
        ss.ssvp_set_cameras(s.ctx, 0, s.clip.K, 0, s.clip.w2c)
    ss.ssvp_gather_filter(s.ctx, p, [0])
    ss.ssvp_read_output(s.ctx, 0, p.frame_begin, p.frame_end, s.out)
    return s.out


def work(case):
    """Bytes: every colour and depth a pass reads, once, and its results.  Operations: 8 per examined candidate of
    a window, 30 per input pixel carried into the output view, the network's products."""
    px = 10 if case["f16"] else 16
    op = case["op"]
    if op == "plan":
        b = fl = 0
        for W, H, F in _shapes(case):
            b += W * H * F * (px + 12)
            fl += W * H * sum(min(F - 1, o + case["T"]) - max(0, o - case["T"]) + 1 for o in range(F)) * case["k"] ** 2 * 8
        return dict(bytes=b, flops=fl)
    W, H, T, n = case["W"], case["H"], case["T"], case.get("n", 1)
    frames = min(case["F"], 2 * T + n)
    slots = sum(min(case["F"] - 1, o + T) - max(0, o - T) + 1 for o in range(case["O"], case["O"] + n))
    out = n * W * H * 12 * case.get("scale", 1) ** 2
    b = frames * W * H * px + out
    fl = W * H * slots * 30
    if op in ("window", "reload", "learned"):
        fl = W * H * slots * case["k"] ** 2 * 8
    if op == "aperture":
        fl = W * H * slots * 100 * 20
    if op == "learned":
        fl += n * W * H * 64 * 2 * 64 * 18
    if op == "reload":
        b = case["F"] * W * H * 16 + out
    if op == "grad":
        m = case["batch"]
        b = min(frames * W * H * px, m * slots * 49 * px) + m * 12 + 1219 * 4
        fl = m * slots * 49 * 8 + m * 64 * 3 * 2 * 64 * 18
    return dict(bytes=b, flops=fl)


# ---------------------------------------------------------------- the same results in 64 bits

def _pair(K, wO, wJ):
    """M, e with K (R_JO K^-1 (u, v, 1) d + t_JO) = M (u, v, 1) d + e."""
    R = wJ[:, :3] @ wO[:, :3].T
    t = wJ[:, 3] - R @ wO[:, 3]
    return K @ R @ np.linalg.inv(K), K @ t


class _Exact:
    def __init__(self, c, f16):
        self.c = c
        rgb = c.rgb.half() if f16 else c.rgb
        self.rgb = [r.double() for r in rgb]
        self.depth = [torch.where(torch.isfinite(d) & (d > 0), d, torch.full_like(d, float("nan"))).double() for d in c.depth]
        v = c.depth[torch.isfinite(c.depth) & (c.depth > 0)]
        self.median = float(v.median())  # the lower one
        self.r = float(np.float32(RADIUS_REL)) * self.median
        self.srgb, self.sf = float(np.float32(SIGMA_RGB)), SIGMA_F
        y, x = torch.meshgrid(torch.arange(c.H, device="cuda", dtype=torch.float64), torch.arange(c.W, device="cuda", dtype=torch.float64), indexing="ij")
        self.y, self.x = y.reshape(-1), x.reshape(-1)

    def sharpness_log2(self):
        s = []
        for a in self.rgb:
            gx, gy = a[:-1, 1:] - a[:-1, :-1], a[1:, :-1] - a[:-1, :-1]
            s.append(float((gx.square().sum(-1) + gy.square().sum(-1)).sqrt().sum()))
        return [math.log2(v / max(s)) for v in s]

    def project(self, O, J, u, v, d):
        """(pixel position in J, depth in J) of points at depth d behind pixels (u, v) of O."""
        if J == O:
            return u, v, d
        M, e = _pair(self.c.K, self.c.w2c[O], self.c.w2c[J])
        w = [d * (M[i, 0] * u + M[i, 1] * v + M[i, 2]) + e[i] for i in range(3)]
        return w[0] / w[2], w[1] / w[2], w[2]

    def candidates(self, O, J, u, v, d, k):
        """For each of the k x k window pixels: (index, depth, squared distance to x_ref, dz), NaN outside."""
        c, h = self.c, (k - 1) // 2
        pu, pv, z = self.project(O, J, u, v, d)
        z = torch.where(z > 1e-6 * d, z, torch.full_like(z, float("nan")))
        cx, cy = torch.floor(pu + 0.5).nan_to_num(-1e6).clamp(-1e6, 1e6), torch.floor(pv + 0.5).nan_to_num(-1e6).clamp(-1e6, 1e6)
        fx, fy, ox, oy = c.K[0, 0], c.K[1, 1], c.K[0, 2], c.K[1, 2]
        yx, yy = z * (pu - ox) / fx, z * (pv - oy) / fy
        D = self.depth[J].reshape(-1)
        for dy in range(-h, h + 1):
            for dx in range(-h, h + 1):
                qx, qy = cx + dx, cy + dy
                inside = (qx >= 0) & (qx < c.W) & (qy >= 0) & (qy < c.H)
                i = (qy.clamp(0, c.H - 1) * c.W + qx.clamp(0, c.W - 1)).long()
                dq = torch.where(inside, D[i], torch.full_like(z, float("nan")))
                dz = dq - z
                X, Y = dq * (qx - ox) / fx - yx, dq * (qy - oy) / fy - yy
                yield i, dq, X * X + Y * Y + dz * dz, dz

    def window(self, O, T, k, mode, px=None):
        """Eq. 3-4 of output frame O (or of its pixels px): (n, 3)."""
        c = self.c
        u, v = (self.x, self.y) if px is None else (self.x[px], self.y[px])
        at = slice(None) if px is None else px
        d, ref = self.depth[O].reshape(-1)[at], self.rgb[O].reshape(-1, 3)[at]
        num, den, cnt = torch.zeros_like(ref), torch.zeros_like(d), torch.zeros_like(d)
        sharp = self.sharpness_log2() if mode == "deblur" else None
        for J in range(max(0, O - T), min(c.F - 1, O + T) + 1):
            col = self.rgb[J].reshape(-1, 3)
            lw = -((J - O) ** 2) / (2 * self.sf**2) + (math.log(2) * sharp[J] if sharp else 0.0)
            if mode == "shutter":
                lw = math.log(float(_shutter(T)[J - O + T]))
            for i, dq, d2, dz in self.candidates(O, J, u, v, d, k):
                e = col[i] - ref
                if mode == "mean":
                    w = torch.ones_like(d2)
                elif mode == "shutter":
                    w = torch.full_like(d2, math.exp(lw))
                else:
                    w = torch.exp(lw - e.square().sum(-1) / (2 * self.srgb**2) - d2 / (2 * self.r**2))
                ok = d2 < self.r * self.r
                w = torch.where(ok, w, torch.zeros_like(w))
                num += w[:, None] * e
                den += w
                cnt += ok
        return ref + torch.where(den[:, None] > 0, num / den[:, None], torch.zeros_like(num)), cnt

    def sets(self, O, T, k, px, plain, cnt, cap=64):
        """Features (n, cap, 16), colours (n, cap, 3) and counts of the first samples in canonical frame order."""
        c, n = self.c, len(px)
        u, v, d, ref = self.x[px], self.y[px], self.depth[O].reshape(-1)[px], self.rgb[O].reshape(-1, 3)[px]
        feat, at = torch.zeros(n, cap, 16, device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.int64)
        for t in range(2 * T + 1):
            J = O + (0 if t == 0 else -(t + 1) // 2 if t % 2 else t // 2)
            if not 0 <= J < c.F:
                continue
            col = self.rgb[J].reshape(-1, 3)
            for i, dq, d2, dz in self.candidates(O, J, u, v, d, k):
                r = torch.nonzero((d2 < self.r * self.r) & (at < cap)).squeeze(1)
                e = col[i[r]] - ref[r]
                lw = -e.square().sum(-1) / (2 * self.srgb**2) - d2[r] / (2 * self.r**2) - (J - O) ** 2 / (2 * self.sf**2)
                f = torch.cat([col[i[r]], e, torch.stack([d2[r].sqrt() / self.r, torch.full_like(lw, (J - O) / max(T, 1)), dz[r] / self.r, lw, torch.ones_like(lw),
                               cnt[r] / 64], 1), col[i[r]] - plain[r], torch.zeros_like(lw)[:, None]], 1)
                feat[r, at[r]] = f
                at[r] += 1
        return feat, feat[:, :, :3].clone(), at

    def network(self, feat, col, n, w):
        """Learned output (n, 3) and confidence (n,)."""
        W1, b1, W2, b2 = w
        z = torch.relu(feat @ W1.T + b1) @ W2.T + b2
        on = (torch.arange(feat.shape[1], device="cuda")[None] < n[:, None]).double()
        wt = torch.nn.functional.softplus(z[..., 0]) * on
        conf = (torch.sigmoid(z[..., 1]) * on).sum(1) / n.clamp(min=1)
        return (wt[..., None] * col).sum(1) / wt.sum(1).clamp(min=1e-300)[:, None], conf

    def aperture(self, O, T, k, cap=31, lens=16, A=float(np.float32(0.05))):
        c, h, hc = self.c, (k - 1) // 2, (cap - 1) // 2
        K, z0 = c.K, self.median
        fx, fy, ox, oy = K[0, 0], K[1, 1], K[0, 2], K[1, 2]
        a0 = 0.5 * z0 / fx
        d, ref = self.depth[O].reshape(-1), self.rgb[O].reshape(-1, 3)
        rx, ry = (self.x - ox) / fx, (self.y - oy) / fy
        rr = rx * rx + ry * ry + 1
        num, den = torch.zeros_like(ref), torch.zeros_like(d)
        for J in range(max(0, O - T), min(c.F - 1, O + T) + 1):
            R = c.w2c[J][:, :3] @ c.w2c[O][:, :3].T
            t = c.w2c[J][:, 3] - R @ c.w2c[O][:, 3]
            us, vs, bad = [], [], torch.isnan(d)
            for i in range(lens):
                rho, th = A * math.sqrt((i + 0.5) / lens), 2.399963229728653 * i
                s = 1 - d / z0
                X = [d * rx + rho * math.cos(th) * s, d * ry + rho * math.sin(th) * s, d]
                Y = [R[a, 0] * X[0] + R[a, 1] * X[1] + R[a, 2] * X[2] + t[a] for a in range(3)]
                bad |= ~(Y[2] > 1e-6 * d)
                us.append(fx * Y[0] / Y[2] + ox)
                vs.append(fy * Y[1] / Y[2] + oy)
            us, vs = torch.stack(us).nan_to_num(-1e6).clamp(-1e6, 1e6), torch.stack(vs).nan_to_num(-1e6).clamp(-1e6, 1e6)
            ccx, ccy = torch.floor(us.mean(0) + 0.5), torch.floor(vs.mean(0) + 0.5)
            x0, x1 = torch.maximum(torch.floor(us.amin(0) + 0.5) - h, ccx - hc), torch.minimum(torch.floor(us.amax(0) + 0.5) + h, ccx + hc)
            y0, y1 = torch.maximum(torch.floor(vs.amin(0) + 0.5) - h, ccy - hc), torch.minimum(torch.floor(vs.amax(0) + 0.5) + h, ccy + hc)
            D, col = self.depth[J].reshape(-1), self.rgb[J].reshape(-1, 3)
            y0 = torch.where(bad, torch.full_like(y0, 1e6), y0)
            for dy in range(int((y1 - y0).max()) + 1):
                qy = y0 + dy
                for dx in range(int((x1 - x0).max()) + 1):
                    qx = x0 + dx
                    inside = (qx >= 0) & (qx < c.W) & (qy >= 0) & (qy < c.H) & (qx <= x1) & (qy <= y1)
                    r = torch.nonzero(inside).squeeze(1)
                    i = (qy[r] * c.W + qx[r]).long()
                    dq = D[i]
                    Z = [dq * (qx[r] - ox) / fx - t[0], dq * (qy[r] - oy) / fy - t[1], dq - t[2]]
                    X = [R[0, a] * Z[0] + R[1, a] * Z[1] + R[2, a] * Z[2] for a in range(3)]
                    tt = (X[0] * rx[r] + X[1] * ry[r] + X[2]) / rr[r]
                    p2 = (X[0] - tt * rx[r]) ** 2 + (X[1] - tt * ry[r]) ** 2 + (X[2] - tt) ** 2
                    a = a0 + A * (z0 - tt).abs() / z0
                    w = torch.where(p2 < a * a, (dq / fx) ** 2 / (math.pi * a * a), torch.zeros_like(a))
                    num.index_add_(0, r, w[:, None] * (col[i] - ref[r]))
                    den.index_add_(0, r, w)
        return ref + torch.where(den[:, None] > 0, num / den[:, None], torch.zeros_like(num))

    def scatter(self, O, T, scale=1):
        """Every sample of every output pixel's frustum (l = 3 output pixels): yields per frame J (output pixel, sample index, X_q in O, J)."""
        c, K = self.c, self.c.K.copy()
        if scale > 1:
            K[0, 0], K[1, 1] = K[0, 0] * scale, K[1, 1] * scale
            K[0, 2], K[1, 2] = scale * (K[0, 2] + 0.5) - 0.5, scale * (K[1, 2] + 0.5) - 0.5
        Wo, Ho = c.W * scale, c.H * scale
        for J in range(max(0, O - T), min(c.F - 1, O + T) + 1):
            d = self.depth[J].reshape(-1)
            R = c.w2c[O][:, :3] @ c.w2c[J][:, :3].T
            t = c.w2c[O][:, 3] - R @ c.w2c[J][:, 3]
            if J == O:
                R, t = np.eye(3), np.zeros(3)
            Y = [d * (self.x - c.K[0, 2]) / c.K[0, 0], d * (self.y - c.K[1, 2]) / c.K[1, 1], d]
            X = [R[a, 0] * Y[0] + R[a, 1] * Y[1] + R[a, 2] * Y[2] + t[a] for a in range(3)]
            u, v = K[0, 0] * X[0] / X[2] + K[0, 2], K[1, 1] * X[1] / X[2] + K[1, 2]
            ok = (X[2] > 0.01) & (X[2] < 1000)
            bu, bv = torch.floor(u), torch.floor(v)
            for dv in range(-1, 3):
                for du in range(-1, 3):
                    pu, pv = bu + du, bv + dv
                    r = torch.nonzero(ok & ((pu - u).abs() + (pv - v).abs() < 1.5) & (pu >= 0) & (pu < Wo) & (pv >= 0) & (pv < Ho)).squeeze(1)
                    yield (pv[r] * Wo + pu[r]).long(), r, [a[r] for a in X], J

    def _weighted(self, terms, ref, base=None):
        """Weighted mean around ref of terms() -> (pixel, colour, log weight), with each pixel's largest log weight taken out."""
        top = torch.full((ref.shape[0],), -math.inf, device="cuda", dtype=torch.float64)
        for p, col, lw in terms():
            top.scatter_reduce_(0, p, lw, "amax")
        num, den = torch.zeros_like(ref), torch.zeros_like(top)
        for p, col, lw in terms():
            w = torch.exp(lw - top[p]).nan_to_num(0.0)
            num.index_add_(0, p, w[:, None] * (col - ref[p]))
            den.index_add_(0, p, w)
        return ref + torch.where(den[:, None] > 0, num / den[:, None], torch.zeros_like(num))

    def frustum(self, O, T, mode, scale=1):
        c = self.c
        K = c.K
        d, ref = self.depth[O].reshape(-1), self.rgb[O].reshape(-1, 3)
        rx, ry = (self.x - K[0, 2]) / K[0, 0], (self.y - K[1, 2]) / K[1, 1]
        if scale > 1:
            Wo, Ho = c.W * scale, c.H * scale
            y, x = torch.meshgrid(torch.arange(Ho, device="cuda", dtype=torch.float64), torch.arange(Wo, device="cuda", dtype=torch.float64), indexing="ij")
            xi, yi = ((x + 0.5) / scale - 0.5).clamp(0, c.W - 1).reshape(-1), ((y + 0.5) / scale - 0.5).clamp(0, c.H - 1).reshape(-1)
            x0, y0 = xi.floor(), yi.floor()
            fx, fy = xi - x0, yi - y0
            x0, y0 = x0.long(), y0.long()
            x1, y1 = (x0 + 1).clamp(max=c.W - 1), (y0 + 1).clamp(max=c.H - 1)
            D, C = self.depth[O], self.rgb[O]
            def lerp(a, fx, fy):
                return (1 - fy) * ((1 - fx) * a[y0, x0] + fx * a[y0, x1]) + fy * ((1 - fx) * a[y1, x0] + fx * a[y1, x1])
            d, ref = lerp(D, fx, fy), lerp(C, fx[:, None], fy[:, None])
            rx, ry = ((x.reshape(-1) + 0.5) / scale - 0.5 - K[0, 2]) / K[0, 0], ((y.reshape(-1) + 0.5) / scale - 0.5 - K[1, 2]) / K[1, 1]
        xr = [d * rx, d * ry, d]
        fcol = lambda J, i: self.rgb[J].reshape(-1, 3)[i]  # noqa: E731
        if mode not in ("inpaint", "semi"):
            sa = self.median / K[0, 0]

            def terms():
                for p, i, X, J in self.scatter(O, T, scale):
                    g = torch.isfinite(d[p])
                    p, i, X = p[g], i[g], [a[g] for a in X]
                    col = fcol(J, i)
                    d2 = sum((X[a] - xr[a][p]) ** 2 for a in range(3))
                    lw = -(col - ref[p]).square().sum(-1) / (2 * self.srgb**2) - d2 / (2 * self.r**2) - (J - O) ** 2 / (2 * self.sf**2)
                    if scale > 1:
                        lw = lw - (self.depth[J].reshape(-1)[i] / K[0, 0]) ** 2 / (2 * sa * sa)
                    yield p, col, torch.zeros_like(lw) if mode == "mean" else lw
            return self._weighted(terms, ref)
        box = c.box()
        mask = []
        for J in range(c.F):
            R, t, D = c.w2c[J][:, :3], c.w2c[J][:, 3], self.depth[J].reshape(-1)
            Y = [D * (self.x - K[0, 2]) / K[0, 0] - t[0], D * (self.y - K[1, 2]) / K[1, 1] - t[1], D - t[2]]
            Xw = [R[0, a] * Y[0] + R[1, a] * Y[1] + R[2, a] * Y[2] for a in range(3)]
            mask.append((Xw[0] >= box[0]) & (Xw[1] >= box[1]) & (Xw[2] >= box[2]) & (Xw[0] <= box[3]) & (Xw[1] <= box[4]) & (Xw[2] <= box[5]))
        cin, cur = ref, ref
        for step in range(3):
            last = step == 2 and mode == "semi"

            def terms(cur=cur):
                for p, i, X, J in self.scatter(O, T):
                    g = mask[O][p]
                    p, i, X = p[g], i[g], [a[g] for a in X]
                    col = fcol(J, i)
                    lw = -(col - cur[p]).square().sum(-1) / (2 * self.srgb**2)
                    if step == 0:
                        yield p, col, torch.zeros_like(lw)
                        continue
                    yield p, col, torch.where(mask[J][i], torch.full_like(lw, -math.inf), lw)
                    if last:
                        h = torch.isfinite(d[p])
                        d2 = sum((X[a] - xr[a][p]) ** 2 for a in range(3))
                        l4 = -(col - cin[p]).square().sum(-1) / (2 * self.srgb**2) - d2 / (2 * self.r**2) - (J - O) ** 2 / (2 * self.sf**2)
                        yield p[h], col[h], l4[h]
            cur = self._weighted(terms, cur)
        return cur


def exact(case, seed):
    op = case["op"]
    if op == "plan":
        out = []
        for i, (W, H, F) in enumerate(_shapes(case)):
            e = _Exact(_Clip(case["scene"], W, H, F, seed * 31 + i), case["f16"])
            out.append(torch.stack([e.window(O, case["T"], case["k"], "denoise")[0].reshape(H, W, 3) for O in range(F)]))
        return out
    W, H, O, T, n = case["W"], case["H"], case["O"], case["T"], case.get("n", 1)
    c = _Clip(case["scene"], W, H, case["F"], seed, clean=op == "grad")
    e = _Exact(c, case["f16"])
    if op in ("window", "reload"):
        return torch.stack([e.window(o, T, case["k"], case["mode"])[0].reshape(H, W, 3) for o in range(O, O + n)])
    if op == "aperture":
        return torch.stack([e.aperture(o, T, case["k"]).reshape(H, W, 3) for o in range(O, O + n)])
    if op == "frustum":
        return torch.stack([e.frustum(o, T, case["mode"]).reshape(H, W, 3) for o in range(O, O + n)])
    if op == "superres":
        z = case["scale"]
        return torch.stack([e.frustum(o, T, "denoise", z).reshape(H * z, W * z, 3) for o in range(O, O + n)])
    w = [torch.tensor(np.asarray(a, np.float32), device="cuda", dtype=torch.float64) for a in _mlp(seed)]
    if op == "learned":
        out = torch.empty(n, H * W, 3, device="cuda", dtype=torch.float64)
        for a in range(n):
            for px in torch.arange(H * W, device="cuda").split(1 << 18):
                plain, cnt = e.window(O + a, T, case["k"], "denoise", px)
                feat, col, m = e.sets(O + a, T, case["k"], px, plain, cnt)
                o, conf = e.network(feat, col, m, w)
                out[a, px] = torch.where(((m > 0) & (conf >= 0.5))[:, None], o, plain)
        return out.reshape(n, H, W, 3)
    px = torch.tensor(_batch(case, seed).astype(np.int64), device="cuda")
    plain, cnt = e.window(O, T, case["k"], "denoise", px)
    w = [a.requires_grad_() for a in w]
    loss = torch.zeros((), device="cuda", dtype=torch.float64)
    y = c.clean[O].reshape(-1, 3).double()[px]
    feat, col, m = e.sets(O, T, case["k"], px, plain, cnt)
    o, conf = e.network(feat, col, m, w)
    has = m > 0
    el, ep = (o - y).square().mean(1), (plain - y).square().mean(1)
    t = (el.detach() <= ep).double()
    cc = conf.clamp(1e-6, 1 - 1e-6)
    loss = ((el - float(np.float32(0.1)) * (t * cc.log() + (1 - t) * (1 - cc).log())) * has).sum() / len(px)
    loss.backward()
    return torch.cat([a.grad.reshape(-1) for a in w] + [loss.detach()[None]])
