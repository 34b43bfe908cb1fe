"""Kernels that a launch shape, long rays or the closed form of the rise select, against
uniform stepping (the same bits; in light-only mode the light, and the argmin of rays in the
penumbra): the walks, which default launches no longer reach, the packets' closed-form
instances, batches of either form and of both, and rays at the length that packets take."""
import math

import numpy as np
import pytest
import torch

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu
R = 1737.4e3


def _tile(nx, ny, g, proj="gnomonic", seed=5, pad=0, amp=300.0):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(nx, device="cuda")[None, :]
    y = torch.arange(ny, device="cuda")[:, None]
    h = torch.zeros((ny, nx + pad), device="cuda")
    h[:, :nx] = amp * (torch.sin(x / 7.3 + 1.0) * torch.cos(y / 5.1) + 0.4 * torch.sin(x / 2.9 - y / 3.7))
    h[:, :nx] += 0.05 * amp * torch.randn((ny, nx), device="cuda", generator=gen)
    return ss.Heightfield(h[:, :nx], g, R, proj)


def _points(nx, ny, n, seed):
    rng = np.random.default_rng(seed)
    uv = np.concatenate([np.cumsum(rng.uniform(0, 0.6, (n // 2, 2)), 0) % (min(nx, ny) - 9),
                         rng.uniform(-9.0, max(nx, ny) + 9.0, (n - n // 2, 2))])
    return torch.from_numpy(uv.astype(np.float32)).cuda()


def _series(hf, sun, lmax, listed):
    """Whether the host takes the series of the rise (|x| <= 1/32 for every ray)."""
    ny, nx = hf.shape
    st = min(1.0, (3.0 if listed else 1.0) * 0.5 * math.hypot((nx - 1) * hf.texel_m, (ny - 1) * hf.texel_m) / R)
    se = min(1.0, abs(math.sin(sun.elevation)) + st * abs(math.cos(sun.elevation)))
    return lmax * (4.0 * se / R + 4.0 * lmax / (R * R)) <= 0.03125


def _check(hf, sun, lmax, modes=(False, True), counts=(False, True), step=0.5, shape=None, **rays):
    mip = ss.ss_build_maxmip(hf)
    b = ss.ss_shadow_uniform(hf, mip, sun, lmax, early_exit=False, step_texels=step, **rays)
    pen = (b["light"] > 0) & (b["light"] < 1)
    for light_only in modes:
        for count in counts:
            a = ss.ss_shadow_forward(hf, mip, sun, lmax, light_only=light_only, count_samples=count,
                                     step_texels=step, **(shape or {}), **rays)
            assert torch.equal(a["light"], b["light"])
            keep = pen if light_only else slice(None)
            assert torch.equal(a["argmin"][keep], b["argmin"][keep])
            assert torch.equal(a["cost"][keep], b["cost"][keep])
            if count:
                assert (a["counters"].sum(0) > 0).all()


# the walks: leaf-task, single-lane and light-only kernels, both forms of the rise
@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("shape", [dict(block_threads=256), dict(refill_min=9, leaf_level=0),
                                   dict(lane_leaves=True), dict(strip_len=6)])
@pytest.mark.parametrize("elev", [1.0, 35.0])
def test_walks(proj, shape, elev):
    hf = _tile(260, 190, 20.0, proj, pad=3)
    sun = ss.Sun(math.radians(elev), 2.1)
    lmax = 60e3 if elev > 10 else 20e3
    assert _series(hf, sun, lmax, True) == (elev < 10)
    _check(hf, sun, lmax, shape=shape)
    _check(hf, sun, lmax, shape=shape, uv=_points(260, 190, 4000, 3))


# the packets' closed form of the rise: grid and listed rays
@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("nx,ny", [(130, 127), (601, 527)])
def test_packets_closed_form(proj, nx, ny):
    hf = _tile(nx, ny, 20.0, proj, pad=1)
    for elev, az in ((35.0, 2.1), (-20.0, 0.4)):
        sun = ss.Sun(math.radians(elev), az)
        assert not _series(hf, sun, 60e3, False)
        _check(hf, sun, 60e3)
        _check(hf, sun, 60e3, uv=_points(nx, ny, nx * ny // 2, 4))


# 2.5e5 texels: the longest rays that take packets, and the shortest that take the walks
@pytest.mark.parametrize("proj", ["gnomonic", "polar_stereo"])
@pytest.mark.parametrize("samples", [62500, 62501])
def test_longest_rays_of_packets(proj, samples):
    hf = _tile(400, 300, 20.0, proj)
    lmax = (samples + 0.5) * 4.0 * 20.0
    for elev, az in ((1.0, 2.1), (38.0, 5.0)):
        sun = ss.Sun(math.radians(elev), az)
        _check(hf, sun, lmax, step=4.0)
        _check(hf, sun, lmax, step=4.0, uv=_points(400, 300, 3000, 7))


@pytest.mark.parametrize("light_only", [False, True])
@pytest.mark.parametrize("elevs", [(35.0, 40.0, 50.0, 30.0), (1.0, 1.2, 50.0, 2.0)])
@pytest.mark.parametrize("shape", [dict(), dict(refill_min=9), dict(lane_leaves=True)])
@pytest.mark.parametrize("count", [False, True])
def test_batch_rise_forms(light_only, elevs, shape, count):
    lmax = 50e3
    hfs = [_tile(nx, ny, 20.0, pad=p, seed=k)
           for k, (nx, ny, p) in enumerate([(3, 2, 0), (65, 33, 1), (128, 96, 0), (301, 300, 2)])]
    suns = [ss.Sun(math.radians(e), 0.9 * k) for k, e in enumerate(elevs)]
    assert [_series(h, s, lmax, False) for h, s in zip(hfs, suns)] == [e < 10 for e in elevs]
    b = ss.Batch(hfs, suns, lmax, want_cost=True, light_only=light_only, count_samples=count, **shape)
    for go in (b.submit, b.launch):
        for hf, sun, o in zip(hfs, suns, go()):
            r = ss.ss_shadow_uniform(hf, ss.ss_build_maxmip(hf), sun, lmax, early_exit=False)
            assert torch.equal(o["light"], r["light"])
            keep = (r["light"] > 0) & (r["light"] < 1) if light_only else slice(None)
            assert torch.equal(o["argmin"][keep], r["argmin"][keep])
            assert torch.equal(o["cost"][keep], r["cost"][keep])
            o["light"].fill_(7.0)
    b.close()
