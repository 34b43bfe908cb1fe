"""The calls whose speed counts: terrain tiles, suns, ray origins and views of the
sizes this framework is used at, each run through the public Python binding.

Terrain is seeded lunar-like fBm with craters (the recipe of the repository's
workloads, generated on the GPU), so every seed gives another tile.  Kinds:

  grid    maximum mipmap + exact shadow of every texel (a tile that changes)
  points  exact shadow at listed surface points of a tile whose mipmap is kept
  view    the terrain points a camera sees
  frame   one rendered frame: mipmap, light-only shadows of two lights, shading
  fit     one step of fitting heights and suns to lights (autograd)
  repro   forward and bit-reproducible backward of one sun
  batch   many tiles of uneven sizes, one captured launch
  mip     the maximum mipmap alone
"""
import math

import numpy as np
import torch

import paper_2005_06671_gb300 as ss

R_MOON = 1737.4e3
SUN_RADIUS = math.radians(0.2665)
EARTH = dict(elev=2.0, az=0.0, radius=math.radians(0.95), intensity=2e-4)


def listed():
    return [
        # the smallest tile in use (an insert or a preview): latency counts
        dict(name="tiny_grid", kind="grid", proj="gnomonic", nx=256, ny=256, g=20.0, amp=1500.0,
             elev=1.5, az=30.0, lmax=20e3),
        # a crop of a map: odd, not square, too few rays to fill the GPU many times over
        dict(name="crop_grid", kind="grid", proj="gnomonic", nx=1531, ny=1021, g=10.0, amp=1500.0,
             elev=0.7, az=251.0, lmax=60e3),
        # the benchmark's tile: 16.8 M rays of up to 60 km
        dict(name="mid_grid", kind="grid", proj="gnomonic", nx=4096, ny=4096, g=10.0, amp=1500.0,
             elev=1.0, az=120.0, lmax=60e3),
        # a whole polar tile of ordinary size, stereographic, low sun, 100 km rays
        dict(name="polar_grid", kind="grid", proj="polar_stereo", nx=1200, ny=1000, g=20.0,
             amp=4000.0, elev=0.5, az=210.0, lmax=100e3),
        # the surface points of a 1920 x 1080 view of a polar tile, in pixel order
        dict(name="polar_points", kind="points", proj="polar_stereo", n=8192, g=5.0, amp=4000.0,
             order="pixels", width=1920, height=1080, lift=False, elev=0.5, az=210.0, lmax=100e3),
        # scattered instrument masts: random origins above the ground, gnomonic
        dict(name="scatter_points", kind="points", proj="gnomonic", n=2048, g=10.0, amp=1500.0,
             order="random", rays=100003, lift=True, elev=1.2, az=75.0, lmax=50e3),
        # what a 3840 x 2160 camera sees of the 16384^2 polar tile
        dict(name="polar_view", kind="view", n=16384, g=5.0, amp=4000.0, width=3840, height=2160),
        # one frame of a renderer: Sun and Earth shadows of a tile, shaded
        dict(name="lit_frame", kind="frame", n=2048, g=10.0, amp=1500.0, elev=1.0, az=120.0,
             lmax=60e3),
        # one step of fitting a 1024^2 tile to four lights
        dict(name="fit_step", kind="fit", n=1024, g=10.0, amp=1500.0, suns=4, lmax=50e3),
        # the same for one sun where runs have to repeat bit for bit
        dict(name="fit_repro", kind="repro", n=2048, g=10.0, amp=1500.0, elev=1.2, az=93.0,
             lmax=50e3),
        # a map's visible tiles in one launch, each with its own sun
        dict(name="batch_mixed", kind="batch", g=10.0, amp=1500.0, lmax=50e3,
             sizes="512,4096,1024,2048,512,2048,4096,1024,1024,512,4096,2048,512,1024,2048,4096"),
        # a large tile streamed in: its mipmap alone, bound by memory
        dict(name="mip_large", kind="mip", nx=8192, ny=8192, g=10.0, amp=1500.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "points", "points", "view", "frame", "fit", "repro",
                       "batch", "mip"])
    g = rng.choice([5.0, 10.0, 20.0])
    sun = dict(elev=rng.uniform(0.2, 3.0), az=rng.uniform(0.0, 360.0))
    lmax = rng.choice([20e3, 50e3, 60e3, 100e3])
    if kind == "grid":
        stereo = rng.random() < 0.3
        return dict(kind=kind, proj="polar_stereo" if stereo else "gnomonic",
                    nx=_log_int(rng, 64, 4096), ny=_log_int(rng, 64, 4096), g=g,
                    amp=4000.0 if stereo else 1500.0, lmax=lmax, **sun)
    if kind == "points":
        stereo = rng.random() < 0.5
        c = dict(kind=kind, proj="polar_stereo" if stereo else "gnomonic", g=g,
                 n=_log_int(rng, 512, 6000), amp=4000.0 if stereo else 1500.0, lmax=lmax,
                 lift=rng.random() < 0.5, **sun)
        if stereo and rng.random() < 0.5:
            w = _log_int(rng, 240, 2560)
            return dict(c, order="pixels", width=w, height=max(1, w * 9 // 16))
        return dict(c, order="random", rays=_log_int(rng, 1, 2000000))
    if kind == "view":
        w = _log_int(rng, 240, 2560)
        g = rng.choice([5.0, 10.0])
        return dict(kind=kind, n=_log_int(rng, 2000, 8000), g=g, amp=4000.0, width=w,
                    height=max(1, w * 9 // 16))
    if kind == "frame":
        return dict(kind=kind, n=_log_int(rng, 128, 4096), g=g, amp=1500.0, lmax=lmax, **sun)
    if kind == "fit":
        return dict(kind=kind, n=_log_int(rng, 96, 2000), g=g, amp=1500.0,
                    suns=rng.randint(1, 4), lmax=50e3)
    if kind == "repro":
        return dict(kind=kind, n=_log_int(rng, 96, 3000), g=g, amp=1500.0, lmax=lmax, **sun)
    if kind == "batch":
        return dict(kind=kind, g=g, amp=1500.0, lmax=50e3, sizes=",".join(
            str(_log_int(rng, 96, 2500)) for _ in range(rng.randint(2, 20))))
    return dict(kind="mip", nx=_log_int(rng, 32, 12000), ny=_log_int(rng, 32, 12000), g=g,
                amp=1500.0)


# ------------------------------------------------------------------ terrain
def _noise(nx, ny, cells_x, cells_y, rng, dev):
    """One octave of gradient noise in separable matrix form (float32)."""
    ox, oy = rng.random_sample(2)

    def weights(n, cells, off):
        x = (torch.arange(n, device=dev, dtype=torch.float64) + 0.5) / n * cells + off
        s = x[:, None] - torch.arange(int(math.ceil(cells + 1.0)) + 1, device=dev,
                                      dtype=torch.float64)[None, :]
        f = (1.0 - s.abs()).clamp(0.0, 1.0)
        w = f * f * f * (f * (f * 6.0 - 15.0) + 10.0)
        return w.float(), (w * s).float()

    wxc, wxs = weights(nx, cells_x, ox)
    wyc, wys = weights(ny, cells_y, oy)
    theta = torch.from_numpy(rng.random_sample((wyc.shape[1], wxc.shape[1])) * 2.0 * math.pi).to(dev)
    return (wyc @ theta.cos().float()) @ wxs.T + (wys @ theta.sin().float()) @ wxc.T


def _terrain(nx, ny, g, amp, seed):
    """fBm (Hurst 0.8, 8 octaves, max |h| = amp) plus parabolic craters, float32 [ny, nx]."""
    dev = torch.device("cuda")
    rng = np.random.RandomState(seed % (1 << 32))
    h = torch.zeros((ny, nx), device=dev)
    for k in range(8):
        h += 2.0 ** (-0.8 * k) * _noise(nx, ny, 2.0 ** k, 2.0 ** k * ny / nx, rng, dev)
    h -= h.mean()
    h *= amp / h.abs().max()
    n = max(4, int(round(500 * nx * ny / 4096.0 ** 2)))
    n = min(n, 5000)
    cx, cy = rng.random_sample(n) * (nx - 1) * g, rng.random_sample(n) * (ny - 1) * g
    u = rng.random_sample(n)
    radii = (200.0 ** -2 - u * (200.0 ** -2 - 2000.0 ** -2)) ** -0.5
    ax = torch.arange(max(nx, ny), device=dev, dtype=torch.float32) * g
    for x, y, r in zip(cx.tolist(), cy.tolist(), radii.tolist()):
        i0, i1 = max(0, int((x - 3 * r) / g)), min(nx, int((x + 3 * r) / g) + 2)
        j0, j1 = max(0, int((y - 3 * r) / g)), min(ny, int((y + 3 * r) / g) + 2)
        q = ((ax[j0:j1, None] - y).square() + (ax[None, i0:i1] - x).square()) / (r * r)
        rim = torch.where(q <= 9.0, 0.08 * r * q.clamp(min=1.0).pow(-1.5), 0.0)
        h[j0:j1, i0:i1] += torch.where(q < 1.0, 0.08 * r + 0.4 * r * (q - 1.0), rim)
    return h


def _suns(k, seed):
    rng = np.random.RandomState((seed + 77) % (1 << 32))
    return [(math.radians(rng.uniform(0.2, 3.0)), math.radians(rng.uniform(0.0, 360.0)))
            for _ in range(k)]


def _camera(width, height, step):
    """10 km up, 30 km from the pole toward grid -y, aimed at the pole, 40 deg field of view."""
    th = 30e3 / R_MOON
    vert = np.array([0.0, -math.sin(th), math.cos(th)])
    pos = (R_MOON + 10e3) * vert
    fwd = np.array([0.0, 0.0, R_MOON]) - pos
    fwd /= np.linalg.norm(fwd)
    right = np.cross(fwd, vert)
    right /= np.linalg.norm(right)
    tan_y = math.tan(math.radians(20.0))
    return dict(pos=pos, forward=fwd, right=right, up=np.cross(right, fwd), tan_y=tan_y,
                tan_x=tan_y * width / height, width=width, height=height, step_m=step,
                max_dist_m=150e3)


def _pixel_dirs(cam, dev):
    W, H = cam["width"], cam["height"]
    i = torch.arange(W, device=dev, dtype=torch.float64)
    j = torch.arange(H, device=dev, dtype=torch.float64)
    a = ((2.0 * (i + 0.5) / W - 1.0) * cam["tan_x"])[None, :, None]
    b = ((1.0 - 2.0 * (j + 0.5) / H) * cam["tan_y"])[:, None, None]
    f, r, u = (torch.from_numpy(np.asarray(cam[k])).to(dev) for k in ("forward", "right", "up"))
    d = (f + a * r + b * u).reshape(-1, 3)
    return d / d.norm(dim=1, keepdim=True)


def _pixel_points(h, g, width, height):
    """Surface points along a view's pixel directions, pixel order (float32 [n, 2]): the
    directions met with the sphere of the terrain height found there, a few times over."""
    dev, n = h.device, h.shape[0]
    cam = _camera(width, height, g / 2)
    d, c = _pixel_dirs(cam, dev), 0.5 * (n - 1)
    p = torch.from_numpy(cam["pos"]).to(dev)
    hh = torch.zeros(d.shape[0], dtype=torch.float64, device=dev)
    b = d @ p
    for _ in range(8):
        disc = b * b - (p @ p - (R_MOON + hh).square())
        q = p + (-b - disc.clamp(min=0.0).sqrt())[:, None] * d
        k = 2.0 * R_MOON / (q.norm(dim=1) + q[:, 2]) / g
        u, v = q[:, 0] * k + c, q[:, 1] * k + c
        hh = _bilinear(h, u.clamp(0, n - 1), v.clamp(0, n - 1)).double()
    keep = (disc > 0) & (u >= 0) & (u <= n - 1) & (v >= 0) & (v <= n - 1)
    uv = torch.stack([u[keep], v[keep]], 1).float()
    # half as many points as pixels, whatever the terrain leaves in sight
    return uv[torch.arange((width * height + 1) // 2, device=dev) % uv.shape[0]].contiguous()


def _origins(case, h, seed):
    """a point set's texel coordinates, and metres above the ground or None"""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["order"] == "pixels":
        uv = _pixel_points(h, case["g"], case["width"], case["height"])
    else:
        uv = torch.rand((case["rays"], 2), generator=gen, device="cuda") * (case["n"] - 1)
    lift = torch.rand(uv.shape[0], generator=gen, device="cuda") * 20.0 if case["lift"] else None
    return uv, lift


def _targets(case, seed):
    """observed lights to fit a tile to: one smooth image a sun, values in [0, 1]"""
    x = torch.arange(case["n"], device="cuda", dtype=torch.float32) * case["g"]
    rng = np.random.RandomState((seed + 5) % (1 << 32))
    return [(0.5 + 0.5 * torch.sin(x / 160.0 + p)[None, :] * torch.sin(x / 190.0 + q)[:, None]).reshape(-1)
            for p, q in rng.random_sample((case["suns"], 2)) * 6.28]


def _loss_grad(n, seed):
    """dLoss/dlight of some loss"""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, generator=gen, device="cuda")


# ------------------------------------------------------- prepare, run, work
def prepare(case, seed):
    kind, g = case["kind"], case["g"]
    if kind == "batch":
        sizes = [int(x) for x in case["sizes"].split(",")]
        hfs = [ss.Heightfield(_terrain(n, n, g, case["amp"], seed * 1000 + i), g, R_MOON)
               for i, n in enumerate(sizes)]
        suns = [ss.Sun(e, a) for e, a in _suns(len(sizes), seed)]
        return dict(kind=kind, batch=ss.Batch(hfs, suns, case["lmax"]).plan())
    nx, ny = case.get("nx", case.get("n")), case.get("ny", case.get("n"))
    proj = case.get("proj", "polar_stereo" if kind == "view" else "gnomonic")
    hf = ss.Heightfield(_terrain(nx, ny, g, case["amp"], seed), g, R_MOON, proj)
    s = dict(kind=kind, hf=hf, lmax=case.get("lmax"))
    if "elev" in case:
        s["sun"] = ss.Sun(math.radians(case["elev"]), math.radians(case["az"]))
    if kind == "points":
        s["mip"] = ss.ss_build_maxmip(hf)
        s["uv"], s["lift"] = _origins(case, hf.h, seed)
    elif kind == "view":
        s["mip"] = ss.ss_build_maxmip(hf)
        s["cam"] = _camera(case["width"], case["height"], g / 2)
    elif kind == "fit":
        s["suns"] = [torch.tensor(x, dtype=torch.float64, requires_grad=True)
                     for x in _suns(case["suns"], seed)]
        s["h"] = hf.h.clone().requires_grad_(True)
        s["target"] = _targets(case, seed)
    elif kind == "repro":
        s["grad"] = _loss_grad(nx * ny, seed)
    elif kind == "mip":   # a program that streams tiles keeps the buffer and its views
        s["mip"] = ss.ss_build_maxmip(hf)
        s["levels"] = ss.maxmip_views(s["mip"], nx, ny) + [ss.maxmip_stats(s["mip"], nx, ny)]
        s["mip"].zero_()
    return s


def run(s):
    kind = s["kind"]
    if kind == "grid":
        mip = ss.ss_build_maxmip(s["hf"])
        r = ss.ss_shadow_forward(s["hf"], mip, s["sun"], s["lmax"])
        return [r["light"], r["argmin"], r["cost"]]
    if kind == "points":
        r = ss.ss_shadow_forward(s["hf"], s["mip"], s["sun"], s["lmax"], uv=s["uv"], lift=s["lift"])
        return [r["light"], r["argmin"], r["cost"]]
    if kind == "view":
        uv, pixel = ss.ss_view_rays(s["hf"], s["mip"], s["cam"])
        n = s["cam"]["width"] * s["cam"]["height"]   # as images: coordinates, ray of each pixel
        image, ray = uv.new_zeros((n, 2)), pixel.new_full((n,), -1)
        at = pixel.long()
        image[at], ray[at] = uv, torch.arange(len(pixel), dtype=torch.int32, device=uv.device)
        return [image, ray]
    if kind == "frame":
        hf, sun = s["hf"], s["sun"]
        earth = ss.Sun(math.radians(EARTH["elev"]), math.radians(EARTH["az"]), EARTH["radius"])
        mip = ss.ss_build_maxmip(hf)
        lit = [ss.ss_shadow_forward(hf, mip, x, s["lmax"], light_only=True, want_cost=False)["light"]
               for x in (sun, earth)]
        lights = [(sun.elevation, sun.azimuth, 1.0, lit[0]),
                  (earth.elevation, earth.azimuth, EARTH["intensity"], lit[1])]
        return [lit[0], lit[1], ss.ss_shade(hf, lights)]
    if kind == "fit":
        hf = s["hf"]
        loss = sum(torch.nn.functional.mse_loss(
            ss.shadow(s["h"], x, hf.texel_m, hf.radius_m, SUN_RADIUS, s["lmax"]), t)
            for x, t in zip(s["suns"], s["target"]))
        grads = torch.autograd.grad(loss, [s["h"]] + s["suns"])
        return [loss.detach()] + list(grads)
    if kind == "repro":
        hf = s["hf"]
        mip = ss.ss_build_maxmip(hf)
        r = ss.ss_shadow_forward(hf, mip, s["sun"], s["lmax"])
        gh, gs = ss.ss_shadow_backward(hf, s["sun"], s["lmax"], r["argmin"], s["grad"],
                                       cost=r["cost"], deterministic=True)
        return [r["light"], r["argmin"], gh, gs]
    if kind == "batch":
        return [x for o in s["batch"].launch() for x in (o["light"], o["argmin"])]
    ss.ss_build_maxmip(s["hf"], mip=s["mip"])
    return s["levels"]


#: float operations of one ray: about 100 bounds and samples of 30 operations for the exact
#: minimum, a quarter of that where the light alone is wanted, 300 in a backward pass
EXACT, LIGHT, BACK = 3000.0, 750.0, 300.0


def work(case):
    kind = case["kind"]
    if kind == "batch":
        t = sum(int(x) ** 2 for x in case["sizes"].split(","))
        return dict(bytes=4.0 * t + 8.0 * t, flops=EXACT * t)
    t = float(case.get("nx", case.get("n")) * case.get("ny", case.get("n")))
    if kind == "grid":
        return dict(bytes=4 * t + 12 * t, flops=EXACT * t)
    if kind == "points":
        n = (case["width"] * case["height"] + 1) // 2 if case["order"] == "pixels" else case["rays"]
        lift = 4 if case["lift"] else 0
        # a point set reads the part of the tile its rays pass over: at most all of it
        return dict(bytes=min(4 * t, n * 100 * 16) + (20 + lift) * n, flops=EXACT * n)
    if kind == "view":
        n = float(case["width"] * case["height"])
        return dict(bytes=min(4 * t, n * 100 * 16) + 12 * n, flops=EXACT * n)
    if kind == "frame":
        return dict(bytes=4 * t + 4 * 3 * t, flops=2 * LIGHT * t)
    if kind == "fit":
        k = case["suns"]
        return dict(bytes=4 * t * (2 + k), flops=k * (EXACT + BACK) * t)
    if kind == "repro":
        return dict(bytes=4 * t * 5, flops=(EXACT + BACK) * t)
    return dict(bytes=4 * t * (1 + 1 / 3), flops=t)


# ------------------------------------------------ the same in 64 bits, plainly
def _bilinear(h, u, v):
    ny, nx = h.shape
    i, j = u.floor().long().clamp(0, nx - 2), v.floor().long().clamp(0, ny - 2)
    fu, fv = u - i, v - j
    k = j * nx + i
    f = h.reshape(-1)
    top = f[k] * (1 - fu) + f[k + 1] * fu
    return top * (1 - fv) + (f[k + nx] * (1 - fu) + f[k + nx + 1] * fu) * fv


def _sun_vec(e, a):
    return torch.stack([e.cos() * a.sin(), e.cos() * a.cos(), e.sin()])


class _Plain:
    """A tile and a sun in 64 bits: every sample of every ray, no skipping but the exact
    stop once a ray is above all terrain by more than its minimum."""

    def __init__(self, h, g, proj, elev, az, alpha, lmax):
        self.h, self.g, self.proj, self.alpha = h, g, proj, alpha
        self.ny, self.nx = h.shape
        self.cx, self.cy = 0.5 * (self.nx - 1), 0.5 * (self.ny - 1)
        self.s = _sun_vec(elev, az)
        self.delta = 0.5 * g
        self.J = int(math.floor(lmax / self.delta))

    def direction(self, u, v):
        X, Y = (u - self.cx) * self.g, (v - self.cy) * self.g
        if self.proj == "gnomonic":
            m = (X * X + Y * Y + R_MOON ** 2).sqrt()
            return torch.stack([X / m, Y / m, R_MOON / m])
        fr, r2 = 4.0 * R_MOON ** 2, X * X + Y * Y
        return torch.stack([4 * R_MOON * X, 4 * R_MOON * Y, fr - r2]) / (fr + r2)

    def origins(self, u, v, lift):
        n = self.direction(u, v)
        hp = _bilinear(self.h, u, v)
        return n, (hp if lift is None else hp + lift)

    def sample(self, n, hp, sin_e, t):
        """height over the sphere, texel image of the points at distance t"""
        rho = R_MOON + hp
        w = t * (2.0 * rho * sin_e + t)
        rise = w / (rho + (rho * rho + w).sqrt())
        q = [rho * n[k] + t * self.s[k] for k in range(3)]
        k = R_MOON / q[2] if self.proj == "gnomonic" else 2.0 * R_MOON / (rho + rise + q[2])
        return hp + rise, q[0] * k / self.g + self.cx, q[1] * k / self.g + self.cy

    def minimum(self, u, v, lift=None, part=1 << 20):
        cost = torch.full_like(u, math.inf)
        at = torch.full(u.shape, -1, dtype=torch.int64, device=u.device)
        top = self.h.max()
        for lo in range(0, u.shape[0], part):
            sl = slice(lo, lo + part)
            n, hp = self.origins(u[sl], v[sl], None if lift is None else lift[sl])
            sin_e = (n * self.s[:, None]).sum(0)
            idx = torch.arange(lo, lo + hp.shape[0], device=u.device)
            best, arg, j = cost[sl].clone(), at[sl].clone(), 1
            while j <= self.J and idx.numel():
                m = int(min(self.J - j + 1, max(4, min(256, (8 << 20) // idx.numel()))))
                js = torch.arange(j, j + m, device=u.device, dtype=torch.float64)[:, None]
                t = js * self.delta
                H, U, V = self.sample([x[None] for x in n], hp[None], sin_e[None], t)
                ok = (U >= 0) & (U <= self.nx - 1) & (V >= 0) & (V <= self.ny - 1)
                ok = ok.to(torch.uint8).cumprod(0).bool()
                hb = _bilinear(self.h, U.clamp(0, self.nx - 1), V.clamp(0, self.ny - 1))
                c, k = torch.where(ok, (H - hb) / t, math.inf).min(0)
                less = c < best
                best, arg = torch.where(less, c, best), torch.where(less, k + j, arg)
                on = ok[-1] & ((H[-1] - torch.maximum(top, hp)) / t[-1] < best)
                off = ~on
                cost[idx[off]], at[idx[off]] = best[off], arg[off]
                idx, best, arg, hp, sin_e, n = idx[on], best[on], arg[on], hp[on], sin_e[on], n[:, on]
                j += m
            cost[idx], at[idx] = best, arg
        return cost, at

    def d_of(self, u, v, at, lift=None):
        """cost cos(elevation) / alpha at the given samples (differentiable)"""
        n, hp = self.origins(u, v, lift)
        sin_e = (n * self.s[:, None]).sum(0)
        t = at.double() * self.delta
        H, U, V = self.sample(n, hp, sin_e, t)
        return (H - _bilinear(self.h, U, V)) / t * (1 - sin_e * sin_e).sqrt() / self.alpha

    def light(self, u, v, cost):
        n = self.direction(u, v)
        sin_e = (n * self.s[:, None]).sum(0)
        d = (cost * (1 - sin_e * sin_e).sqrt() / self.alpha).clamp(-1.0, 1.0)
        return (math.pi - d.acos() + d * (1 - d * d).sqrt()) / math.pi


def _grid_uv(h):
    ny, nx = h.shape
    r = torch.arange(nx * ny, device=h.device)
    return (r % nx).double(), (r // nx).double()


def _backward(P, u, v, at, gl, wrt):
    """gradients of sum(gl * light) at the samples `at`"""
    r = (at > 0).nonzero()[:, 0]
    d = P.d_of(u[r], v[r], at[r])
    slope = torch.where(d.abs() < 1, 2.0 / math.pi * (1 - d * d).clamp(min=0).sqrt(), 0.0).detach()
    return torch.autograd.grad(d, wrt, grad_outputs=gl[r] * slope, retain_graph=False)


def _shade64(h, g, lights):
    ny, nx = h.shape
    u, v = _grid_uv(h)
    X, Y = (u - 0.5 * (nx - 1)) * g, (v - 0.5 * (ny - 1)) * g
    m = (X * X + Y * Y + R_MOON ** 2).sqrt()
    n = torch.stack([X / m, Y / m, R_MOON / m])
    dv, du = torch.gradient(h)
    rho = R_MOON + h.reshape(-1)

    def tangent(axis, dh):
        e = torch.zeros(3, 1, dtype=torch.float64, device=h.device)
        e[axis] = 1.0
        return dh.reshape(-1) * n + rho * g / m * (e - n * n[axis])

    N = torch.linalg.cross(tangent(0, du), tangent(1, dv), dim=0)
    N = N / N.norm(dim=0)
    E = torch.zeros_like(u)
    for e, a, inten, lit in lights:
        s = _sun_vec(torch.tensor(e, dtype=torch.float64), torch.tensor(a, dtype=torch.float64))
        E += inten * lit * (N * s.to(h.device)[:, None]).sum(0).clamp(min=0.0)
    return E


def _view64(h, g, cam):
    """texel coordinates of each pixel's first sample on or below the terrain, the step before
    it halved down to the crossing"""
    ny, nx = h.shape
    dev, step = h.device, cam["step_m"]
    K = int(math.floor(cam["max_dist_m"] / step))
    p = torch.from_numpy(cam["pos"]).to(dev)
    d = _pixel_dirs(cam, dev)
    b, pp = d @ p, p @ p

    def gap(tau, b, d):
        """height over the terrain, its texel, and whether that is in the tile"""
        w = tau * (2.0 * b + tau)
        r0 = pp.sqrt()
        q2 = p[2] + tau * d[:, 2]
        alt = (r0 - R_MOON) + w / (r0 + (pp + w).sqrt())
        k = 2.0 * R_MOON / (R_MOON + alt + q2) / g
        U = (p[0] + tau * d[:, 0]) * k + 0.5 * (nx - 1)
        V = (p[1] + tau * d[:, 1]) * k + 0.5 * (ny - 1)
        ok = (U >= 0) & (U <= nx - 1) & (V >= 0) & (V <= ny - 1)
        return alt - _bilinear(h, U.clamp(0, nx - 1), V.clamp(0, ny - 1)), U, V, ok

    top, low = R_MOON + h.max(), R_MOON + h.min() - 1.0
    disc = b * b - (pp - top * top)
    start = ((-b - disc.clamp(min=0).sqrt()) / step).floor().clamp(min=1) - 1
    disc_low = b * b - (pp - low * low)
    end = torch.where(disc_low > 0, (-b - disc_low.clamp(min=0).sqrt()) / step + 1,
                      (-b + disc.clamp(min=0).sqrt()) / step + 1).clamp(max=K)
    hit = torch.full_like(b, -1.0)
    idx = ((disc > 0) & (b < 0)).nonzero()[:, 0]
    k = start[idx] + 1
    while idx.numel():
        f, _, _, ok = gap(k * step, b[idx], d[idx])
        now = ok & (f <= 0)
        hit[idx[now]] = k[now]
        on = ~now & (k < end[idx])
        idx, k = idx[on], k[on] + 1
    pix = (hit > 0).nonzero()[:, 0]
    b, d, hi = b[pix], d[pix], hit[pix] * step
    lo = hi - step
    f, _, _, ok = gap(lo, b, d)
    lo = torch.where(ok & (lo > 0), lo, hi)
    for _ in range(48):
        mid = 0.5 * (lo + hi)
        f, _, _, _ = gap(mid, b, d)
        lo, hi = torch.where(f > 0, mid, lo), torch.where(f > 0, hi, mid)
    _, U, V, _ = gap(hi, b, d)
    image = torch.zeros((hit.shape[0], 2), dtype=torch.float64, device=dev)
    image[pix] = torch.stack([U.clamp(0, nx - 1), V.clamp(0, ny - 1)], 1)
    return image


#: rays beyond which every sample of every ray in 64 bits takes too long
MOST_RAYS = 5e6


def exact(case, seed):
    kind, g = case["kind"], case["g"]
    if kind == "batch":
        sizes = [int(x) for x in case["sizes"].split(",")]
        if sum(n * n for n in sizes) > MOST_RAYS:
            return None
        out = []
        for i, (n, (e, a)) in enumerate(zip(sizes, _suns(len(sizes), seed))):
            h = _terrain(n, n, g, case["amp"], seed * 1000 + i).double()
            out += [_grid64(h, g, "gnomonic", e, a, SUN_RADIUS, case["lmax"])[0], None]
        return out
    nx, ny = case.get("nx", case.get("n")), case.get("ny", case.get("n"))
    if kind in ("grid", "frame", "fit", "repro") and nx * ny > MOST_RAYS:
        return None
    if kind == "view" and case["width"] * case["height"] > 1e6:
        return None
    h = _terrain(nx, ny, g, case["amp"], seed).double()
    rad = math.radians
    if kind == "grid":
        light, _, cost = _grid64(h, g, case["proj"], rad(case["elev"]), rad(case["az"]),
                                 SUN_RADIUS, case["lmax"])
        return [light, None, cost]
    if kind == "points":
        uv, lift = _origins(case, h.float(), seed)
        P = _plain(h, g, case["proj"], rad(case["elev"]), rad(case["az"]), SUN_RADIUS, case["lmax"])
        u, v = uv.double().unbind(1)
        cost, _ = P.minimum(u, v, None if lift is None else lift.double())
        return [P.light(u, v, cost), None, cost]
    if kind == "view":
        return [_view64(h, g, _camera(case["width"], case["height"], g / 2)), None]
    if kind == "frame":
        sun = (rad(case["elev"]), rad(case["az"]))
        earth = (rad(EARTH["elev"]), rad(EARTH["az"]))
        lit = [_grid64(h, g, "gnomonic", *x, r, case["lmax"])[0]
               for x, r in ((sun, SUN_RADIUS), (earth, EARTH["radius"]))]
        return lit + [_shade64(h, g, [(*sun, 1.0, lit[0]), (*earth, EARTH["intensity"], lit[1])])]
    if kind == "fit":
        target = _targets(case, seed)
        h.requires_grad_(True)
        u, v = _grid_uv(h)
        loss, gh, gs = 0.0, torch.zeros_like(h), []
        for (e, a), t in zip(_suns(case["suns"], seed), target):
            ang = torch.tensor([e, a], dtype=torch.float64, device=h.device, requires_grad=True)
            P = _Plain(h, g, "gnomonic", ang[0], ang[1], SUN_RADIUS, case["lmax"])
            with torch.no_grad():
                cost, at = P.minimum(u, v)
                diff = P.light(u, v, cost) - t.double()
            loss += float(diff.square().mean())
            dh, da = _backward(P, u, v, at, 2.0 * diff / diff.numel(), [h, ang])
            gh += dh
            gs.append(da)
        return [loss, gh] + gs
    if kind == "repro":
        gl = _loss_grad(nx * ny, seed).double()
        h.requires_grad_(True)
        ang = torch.tensor([rad(case["elev"]), rad(case["az"])], dtype=torch.float64,
                           device=h.device, requires_grad=True)
        P = _Plain(h, g, "gnomonic", ang[0], ang[1], SUN_RADIUS, case["lmax"])
        P.s.retain_grad()
        u, v = _grid_uv(h)
        with torch.no_grad():
            cost, at = P.minimum(u, v)
            light = P.light(u, v, cost)
        dh, da, dsun = _backward(P, u, v, at, gl, [h, ang, P.s])
        return [light, None, dh, torch.cat([da, dsun])]
    out, m = [], h
    while max(m.shape) > 1:
        m = torch.nn.functional.max_pool2d(m[None], 2, ceil_mode=True)[0]
        out.append(m)
    return out + [torch.stack([h.max(), h.min()])]


def _plain(h, g, proj, e, a, alpha, lmax):
    e, a = (torch.tensor(x, dtype=torch.float64, device=h.device) for x in (e, a))
    return _Plain(h, g, proj, e, a, alpha, lmax)


def _grid64(h, g, proj, e, a, alpha, lmax):
    P = _plain(h, g, proj, e, a, alpha, lmax)
    u, v = _grid_uv(h)
    cost, at = P.minimum(u, v)
    return P.light(u, v, cost), at, cost
