"""Stereographic tiles whose rays' images bend: default launches and the walks against
uniform stepping (the same bits; light-only: the light, and the argmin in the penumbra)."""
import math

import pytest
import torch

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu


def _spikes(n, R, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    h = torch.zeros(n * n, device="cuda")
    k = torch.randint(0, n * n, (n * n // 40,), device="cuda", generator=gen)
    h[k] = 0.3 * R * torch.rand(k.numel(), device="cuda", generator=gen)
    uv = torch.rand((5000, 2), device="cuda", generator=gen) * (n - 1)
    return h.view(n, n), uv


def _same(R, g, n, elev, az, shapes=(dict(), dict(block_threads=256))):
    h, uv = _spikes(n, R, n)
    hf = ss.Heightfield(h, g, R, "polar_stereo")
    mip = ss.ss_build_maxmip(hf)
    sun = ss.Sun(math.radians(elev), math.radians(az))
    for kw in (dict(), dict(uv=uv)):
        b = ss.ss_shadow_uniform(hf, mip, sun, 3.0 * R, early_exit=False, **kw)
        pen = (b["light"] > 0) & (b["light"] < 1)
        for shape in shapes:
            a = ss.ss_shadow_forward(hf, mip, sun, 3.0 * R, **shape, **kw)
            for k in ("argmin", "cost", "light"):
                assert torch.equal(a[k], b[k]), (k, shape, (a[k] != b[k]).sum().item())
            a = ss.ss_shadow_forward(hf, mip, sun, 3.0 * R, light_only=True, **shape, **kw)
            assert torch.equal(a["light"], b["light"])
            assert torch.equal(a["argmin"][pen], b["argmin"][pen])


# Rays from the border's texels along the border: the arc leaves the tile and comes in
# again, so the first usable sample is not the first.
@pytest.mark.parametrize("R,g,n,elev,az", [
    (2e3, 5.0, 700, 25.0, 30.0), (2e3, 20.0, 280, 2.0, 200.0), (2e3, 20.0, 280, 10.0, 135.0),
    (2e3, 5.0, 300, 25.0, 351.4), (2e3, 66.6, 84, 2.0, 200.0), (2e3, 20.0, 90, 25.0, 351.4)])
def test_rays_that_start_off_the_tile(R, g, n, elev, az):
    _same(R, g, n, elev, az)


# Tiles of up to the whole hemisphere of a small body: blocks of samples whose images are arcs
# of up to a radian and more.
@pytest.mark.parametrize("R,g,n", [(2e3, 66.6, 84), (2e3, 40.0, 140), (2e3, 20.0, 280),
                                   (2e3, 5.0, 500), (1e5, 250.0, 1000)])
@pytest.mark.parametrize("elev,az", [(2.0, 351.4), (25.0, 49.0), (-20.0, 300.0)])
def test_tiles_of_a_hemisphere(R, g, n, elev, az):
    assert 0.5 * math.hypot(n - 1, n - 1) * g <= 2.0 * R
    _same(R, g, n, elev, az)


# Tiles that reach beyond the hemisphere: a ray's image between two samples on the tile can
# be the arc of its circle that passes the antipode, far off the tile.
@pytest.mark.parametrize("R,g,n", [(2e3, 20.0, 700), (2e3, 66.7, 90), (5e3, 60.0, 301)])
@pytest.mark.parametrize("elev,az", [(2.0, 171.9), (25.0, 49.0), (-20.0, 300.0)])
def test_tiles_beyond_the_hemisphere(R, g, n, elev, az):
    assert 0.5 * math.hypot(n - 1, n - 1) * g > 2.0 * R
    _same(R, g, n, elev, az, shapes=(dict(), dict(block_threads=256), dict(lane_leaves=True)))
