"""Edges of the packet descent that test_gpu_packet.py's cases do not reach.  Bars as
there: the bits of uniform stepping."""
import math

import pytest
import torch

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu


# A small sphere, rays diving under a wide tile, a wall far out: past the last usable
# sample the gnomonic denominator 1 + b j is zero or negative, so a block's far end must
# not be taken there (the last block then misses the wall, which holds the minimum).
@pytest.mark.parametrize("n,R,elev,wall,width,height,u0", [
    (402, 636.0, -41.33, 274, 22, 1043.0, 187), (402, 2894.0, -33.61, 357, 28, 9562.0, 78),
    (402, 1505.0, -39.85, 298, 24, 1331.0, 153), (402, 2350.0, -37.99, 349, 12, 6881.0, 66),
    (402, 1811.0, -49.07, 257, 18, 9658.0, 179)])
def test_block_past_the_last_sample(n, R, elev, wall, width, height, u0):
    h = torch.zeros((n, n), device="cuda")
    h[:, wall:wall + width] = height
    hf = ss.Heightfield(h, 20.0, R)
    mip = ss.ss_build_maxmip(hf)
    sun = ss.Sun(math.radians(elev), math.radians(90.0))
    v = torch.arange(n // 2 - 20, n // 2 + 20, device="cuda")
    uv = torch.stack([torch.full_like(v, u0), v], 1).float()
    a = ss.ss_shadow_forward(hf, mip, sun, 20.0 * R, uv=uv)
    b = ss.ss_shadow_uniform(hf, mip, sun, 20.0 * R, uv=uv, early_exit=False)
    for k in ("argmin", "cost", "light"):
        assert torch.equal(a[k], b[k]), k


def _scene(nx, ny, seed=5):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.arange(nx, device="cuda")[None, :]
    y = torch.arange(ny, device="cuda")[:, None]
    h = 300.0 * (torch.sin(x / 7.3 + 1.0) * torch.cos(y / 5.1))
    return (h + 15.0 * torch.randn((ny, nx), device="cuda", generator=gen)).float()


# Every bound shared by a packet counts for one of its rays, also where the packet has
# fewer than 32 (small launches: 8 or 16; the tile's edges).  On flat ground under a high
# sun the light-only count is known: the packet's blocks of 256 samples, the blocks of 8
# of the first one, and the two halves of each ray's own first block, none else survives.
@pytest.mark.parametrize("nx,ny,rows", [(64, 64, 1), (301, 263, 2), (603, 530, 4)])
def test_counters_hold_every_shared_bound(nx, ny, rows):
    hf = ss.Heightfield(torch.zeros((ny, nx), device="cuda"), 20.0, 1737.4e3)
    mip = ss.ss_build_maxmip(hf)
    kw = dict(step_texels=0.1, count_samples=True)
    for az in (120.0, 301.0):
        sun = ss.Sun(math.radians(30.0), math.radians(az))
        a = ss.ss_shadow_forward(hf, mip, sun, 20e3, light_only=True, **kw)
        b = ss.ss_shadow_uniform(hf, mip, sun, 20e3, early_exit=False, **kw)
        jh = b["counters"][:, 1].long()                     # usable samples of the ray
        py, px = (ny + rows - 1) // rows, (nx + 7) // 8
        r = torch.arange(nx * ny, device="cuda")
        packet = (r // nx // rows) * px + r % nx // 8
        zero = torch.zeros(py * px, dtype=torch.long, device="cuda")
        jmax = zero.scatter_reduce(0, packet, jh, "amax")
        want = (jmax + 255) // 256 + ((jmax + 7) // 8).clamp(max=32)
        want = want.scatter_add(0, packet, 2 * (jh > 0).long())
        got = zero.scatter_add(0, packet, a["counters"][:, 0].long())
        assert torch.equal(got, want)


# A leaf task clipped to the ray's last sample counts the samples it has: tasks of rays of
# one or two samples hold one or two (a seed and a leaf task per ray; listed neighbours
# take up to three seeds more from each other).
@pytest.mark.parametrize("samples", [1, 2])
def test_counters_of_clipped_leaf_tasks(samples):
    hf = ss.Heightfield(_scene(130, 61), 20.0, 1737.4e3)
    mip = ss.ss_build_maxmip(hf)
    gen = torch.Generator(device="cuda").manual_seed(2)
    uv = torch.rand((501, 2), device="cuda", generator=gen) * 59.0
    for tasks, kw in ((2, dict()), (5, dict(uv=uv))):
        r = ss.ss_shadow_forward(hf, mip, ss.Sun(math.radians(1.0), 0.3), 10.0 * samples + 1.0,
                                 count_samples=True, **kw)
        c = r["counters"][:, 1]
        assert c.max() <= tasks * samples
        assert (c[r["argmin"] > 0] >= 1).all()
