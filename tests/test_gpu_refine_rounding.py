"""The cost of a penumbra ray is the float32 nearest to its argmin sample's cost in 64
bits, also where it is small against the terms that it is made of."""
import math

import pytest
import torch

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu
R = 1737.4e3


def _cost64(h, g, proj, sun, delta, u, v, j, hp=None):
    """(H_p + rise - h) / t of sample j of the rays at (u, v), in float64."""
    ny, nx = h.shape
    s = [math.cos(sun[0]) * math.sin(sun[1]), math.cos(sun[0]) * math.cos(sun[1]), math.sin(sun[0])]
    cx, cy = 0.5 * (nx - 1), 0.5 * (ny - 1)
    hp = h[v.long(), u.long()].double() if hp is None else hp
    X, Y = (u - cx) * g, (v - cy) * g
    rho, jd = R + hp, j.double()
    t = jd * delta
    if proj == "gnomonic":
        m = (X * X + Y * Y + R * R).sqrt()
        se = (X * s[0] + Y * s[1] + R * s[2]) / m
        f = delta * m / rho
        tau = jd / (1.0 + f * s[2] / R * jd)
        U = u + f / (g * R) * (R * s[0] - s[2] * X) * tau
        V = v + f / (g * R) * (R * s[1] - s[2] * Y) * tau
    else:
        fr, r2 = 4.0 * R * R, X * X + Y * Y
        n = [4.0 * R * X / (fr + r2), 4.0 * R * Y / (fr + r2), (fr - r2) / (fr + r2)]
        se = n[0] * s[0] + n[1] * s[1] + n[2] * s[2]
    w = t * (2.0 * rho * se + t)
    rise = w / (rho + (rho * rho + w).sqrt())
    if proj != "gnomonic":
        ia0, ws, k = (fr + r2) / (2.0 * fr * rho), rise + t * s[2], 2.0 * R / g
        id_ = 1.0 / (1.0 + ws * ia0)
        U = u + (delta * k * s[0] * ia0 * jd - k * rho * n[0] * ia0 * ia0 * ws) * id_
        V = v + (delta * k * s[1] * ia0 * jd - k * rho * n[1] * ia0 * ia0 * ws) * id_
    i0 = U.floor().long().clamp(0, nx - 2)
    j0 = V.floor().long().clamp(0, ny - 2)
    fu, fv = U - i0, V - j0
    h00, h10 = h[j0, i0].double(), h[j0, i0 + 1].double()
    h01, h11 = h[j0 + 1, i0].double(), h[j0 + 1, i0 + 1].double()
    hb = h00 + fu * (h10 - h00) + fv * ((h01 - h00) + fu * ((h11 - h01) - (h10 - h00)))
    return ((hp - hb) + rise) / t


def _wrong(got, c, tol):
    """Costs that are not the float32 nearest to c, nor within tol of the middle."""
    near = c.float()
    lo = torch.nextafter(near, torch.full_like(near, -math.inf)).double()
    hi = torch.nextafter(near, torch.full_like(near, math.inf)).double()
    tie = torch.minimum((c - 0.5 * (near.double() + lo)).abs(),
                        (c - 0.5 * (near.double() + hi)).abs())
    return ((got != near) & (tie > tol)).sum().item()


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
def test_cost_is_the_nearest_float32(proj):
    """Texel coordinates up to 60,000: their last bits, on cells as steep as the costs."""
    nx, ny, g, lmax = 60000, 256, 20.0, 300.0
    gen = torch.Generator(device="cuda").manual_seed(4)
    h = 2.0 * torch.randn((ny, nx), device="cuda", generator=gen)
    hf = ss.Heightfield(h, g, R, projection=proj)
    mip = ss.ss_build_maxmip(hf)
    seen = bad = 0
    for elev, az in ((2.0, 40.0), (-1.0, 155.0)):
        sun = (math.radians(elev), math.radians(az))
        r = ss.ss_shadow_forward(hf, mip, ss.Sun(*sun, 0.5), lmax)
        ids = ((r["light"] > 0) & (r["light"] < 1)).nonzero()[:, 0]
        for k in ids.split(2_000_000):
            c = _cost64(h, g, proj, sun, 0.5 * g, (k % nx).double(), (k // nx).double(),
                        r["argmin"][k].long())
            # 64 bits: half a unit in the last place of a coordinate (2^-38 texel), twice on
            # either side, times the slope of a cell (20 m) over the distance (10 m)
            bad += _wrong(r["cost"][k], c, 2.0 ** -36 * 20.0 / 10.0)
        seen += ids.numel()
    assert seen > 5_000_000
    assert bad == 0


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
def test_cost_of_listed_rays_is_the_nearest_float32(proj):
    """Origins between texels of terrain 8 km up: the origin's height is a sum of terms far
    larger than the clearances that the cost is made of."""
    n, g, lmax = 1024, 20.0, 300.0
    gen = torch.Generator(device="cuda").manual_seed(6)
    h = 8000.0 + torch.randn((n, n), device="cuda", generator=gen)
    hf = ss.Heightfield(h, g, R, projection=proj)
    mip = ss.ss_build_maxmip(hf)
    sun = (math.radians(0.4), math.radians(70.0))
    uv = 8.0 + torch.rand((4_000_000, 2), device="cuda", generator=gen) * (n - 17.0)
    r = ss.ss_shadow_forward(hf, mip, ss.Sun(*sun, 0.5), lmax, uv=uv)
    ids = ((r["light"] > 0) & (r["light"] < 1)).nonzero()[:, 0]
    u, v = uv[ids, 0].double(), uv[ids, 1].double()
    i0, j0 = u.floor().long(), v.floor().long()
    a, b = u - i0, v - j0
    hp = (h[j0, i0].double() * ((1 - a) * (1 - b)) + h[j0, i0 + 1].double() * (a * (1 - b))
          + h[j0 + 1, i0].double() * ((1 - a) * b) + h[j0 + 1, i0 + 1].double() * (a * b))
    c = _cost64(h, g, proj, sun, 0.5 * g, u, v, r["argmin"][ids].long(), hp)
    bad = _wrong(r["cost"][ids], c, 1e-12)   # 64 bits: eight roundings of 8 km over 10 m
    assert ids.numel() > 1_000_000
    assert bad == 0
