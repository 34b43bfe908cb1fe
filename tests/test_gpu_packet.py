"""The packet descent (the default ss_shadow_forward and batch) against uniform
stepping, which evaluates every sample with the same arithmetic: argmin, cost and
light have to be the same bits whatever the shape, mapping, sun or ray set.  In
light-only mode the light is, and the argmin of rays in the penumbra."""
import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

R_MOON = 1737.4e3


def _ss():
    import paper_2005_06671_gb300 as ss
    return ss


def _tile(nx, ny, g, proj="gnomonic", radius=R_MOON, amp=300.0, pad=0, seed=5, nan=0):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:ny, 0:nx]
    h = amp * (np.sin(x / 7.3 + 1.0) * np.cos(y / 5.1) + 0.4 * np.sin(x / 2.9 - y / 3.7))
    h += 0.05 * amp * rng.standard_normal((ny, nx))
    if nan:
        h[rng.integers(0, ny, nan), rng.integers(0, nx, nan)] = np.nan
    buf = torch.zeros((ny, nx + pad), dtype=torch.float32, device="cuda")
    buf[:, :nx] = torch.from_numpy(h.astype(np.float32)).cuda()
    return _ss().Heightfield(buf[:, :nx], g, radius, proj)


def _same(hf, sun, lmax, **kw):
    ss = _ss()
    mip = ss.ss_build_maxmip(hf)
    a = ss.ss_shadow_forward(hf, mip, sun, lmax, **kw)
    b = ss.ss_shadow_uniform(hf, mip, sun, lmax, early_exit=False, **kw)
    for k in ("argmin", "cost", "light"):
        assert torch.equal(a[k], b[k]), k
    c = ss.ss_shadow_forward(hf, mip, sun, lmax, count_samples=True, **kw)
    for k in ("argmin", "cost", "light"):
        assert torch.equal(c[k], b[k]), k
    pen = (b["light"] > 0) & (b["light"] < 1)
    for count in (False, True):
        lit = ss.ss_shadow_forward(hf, mip, sun, lmax, light_only=True, count_samples=count, **kw)
        assert torch.equal(lit["light"], b["light"])
        assert torch.equal(lit["argmin"][pen], b["argmin"][pen])
    return b


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("nx,ny,pad", [(2, 2, 0), (3, 41, 0), (8, 4, 5), (9, 5, 0), (64, 33, 3),
                                       (130, 127, 1)])
def test_grid_shapes(proj, nx, ny, pad):
    for elev, az in ((1.0, 120.0), (-1.5, 301.0), (35.0, 10.0)):
        _same(_tile(nx, ny, 20.0, proj, pad=pad), _ss().Sun(math.radians(elev), math.radians(az)),
              20e3)


# packets of 8, 16 and 32 rays, and strips of several (chosen by the number of rays)
@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("nx,ny", [(301, 263), (601, 527), (2053, 2501)])
def test_grid_packet_sizes(proj, nx, ny):
    for elev, az in ((1.0, 120.0), (38.0, 10.0)):
        _same(_tile(nx, ny, 20.0, proj), _ss().Sun(math.radians(elev), math.radians(az)), 6e3)


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("n", [100003, 700001])
def test_many_listed_rays(proj, n):
    hf = _tile(700, 600, 20.0, proj)
    rng = np.random.default_rng(n)
    near = np.stack([np.arange(n) % 5990 * 0.1, np.arange(n) // 5990 * 4.0], 1)
    for uv in (near, rng.uniform(0.0, 590.0, (n, 2))):
        _same(hf, _ss().Sun(math.radians(1.3), 0.7), 6e3, uv=torch.from_numpy(uv.astype(np.float32)).cuda())


# closed form of the rise (|x| > 1/32), a small sphere, long and short steps, rays of no and of
# one sample, more than 32 blocks of 256 samples
@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("g,radius,elev,lmax,step", [
    (500.0, 300e3, 4.0, 100e3, 0.5), (500.0, 300e3, -6.0, 100e3, 0.5), (20.0, R_MOON, 60.0, 60e3, 0.5),
    (20.0, R_MOON, 0.3, 9.0, 0.5), (20.0, R_MOON, 0.3, 10.0, 0.5), (20.0, R_MOON, 2.0, 4e3, 2.5),
    (2000.0, R_MOON, 1.0, 300e3, 0.02)])
def test_grid_geometry(proj, g, radius, elev, lmax, step):
    _same(_tile(90, 70, g, proj, radius, amp=0.02 * g * 90), _ss().Sun(math.radians(elev), 2.3),
          lmax, step_texels=step)


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("n", [1, 31, 33, 1000])
def test_listed_rays(proj, n):
    hf = _tile(211, 180, 20.0, proj)
    rng = np.random.default_rng(n)
    near = np.cumsum(rng.uniform(0, 0.6, (n, 2)), 0) % 170            # neighbours in id order
    far = rng.uniform(-9.0, 215.0, (n, 2))                            # scattered, some off the tile
    for uv in (near, far):
        t = torch.from_numpy(uv.astype(np.float32)).cuda()
        lift = torch.from_numpy(rng.uniform(0, 30, n).astype(np.float32)).cuda()
        for lf in (None, lift):
            _same(hf, _ss().Sun(math.radians(1.3), 0.7), 20e3, uv=t, lift=lf)


@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
def test_nan_heights(proj):
    hf = _tile(96, 80, 20.0, proj, nan=6)
    ss = _ss()
    mip = ss.ss_build_maxmip(hf)
    sun = ss.Sun(math.radians(1.0), 4.0)
    a = ss.ss_shadow_forward(hf, mip, sun, 20e3)
    b = ss.ss_shadow_uniform(hf, mip, sun, 20e3, early_exit=False)
    ok = torch.isfinite(hf.h).reshape(-1)     # (rays on a NaN texel are unspecified)
    assert torch.equal(a["argmin"][ok], b["argmin"][ok])
    assert torch.equal(a["light"][ok], b["light"][ok])


@pytest.mark.parametrize("elev", [1.0, 35.0])
@pytest.mark.parametrize("light_only", [False, True])
def test_batch(elev, light_only):
    ss = _ss()
    hfs = [_tile(nx, ny, 20.0, pad=p, seed=k)
           for k, (nx, ny, p) in enumerate([(2, 2, 0), (65, 33, 1), (128, 96, 0), (7, 300, 2)])]
    suns = [ss.Sun(math.radians(elev + 0.1 * k), 0.9 * k) for k in range(4)]
    b = ss.Batch(hfs, suns, 20e3, want_cost=True, light_only=light_only)
    for go in (b.submit, b.launch):
        for hf, sun, o in zip(hfs, suns, go()):
            r = ss.ss_shadow_uniform(hf, ss.ss_build_maxmip(hf), sun, 20e3, early_exit=False)
            assert torch.equal(o["light"], r["light"])
            pen = (r["light"] > 0) & (r["light"] < 1) if light_only else slice(None)
            assert torch.equal(o["argmin"][pen], r["argmin"][pen])
            assert torch.equal(o["cost"][pen], r["cost"][pen])
            o["light"].fill_(7.0)
    b.close()
