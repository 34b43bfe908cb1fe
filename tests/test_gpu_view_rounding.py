"""Coordinates of view hits are rounded as FP64 rounds them."""
import numpy as np
import pytest
import torch

import oracle
from workloads import camera, lunar_tile, MOON_RADIUS_M

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("proj,n,g", [("polar_stereo", 2048, 20.0), ("gnomonic", 1500, 30.0)])
def test_coordinates_are_the_nearest_float32(proj, n, g):
    """FP64 places a crossing within eight roundings of |x| - R - h (1.6e-8 m) over the slope
    along the ray (0.3 and more here), so at most 2 x 1.6e-8 / 0.3 / g / 6e-5 of the coordinates
    (float32 steps of 6e-5 texel from 512 on) round to the other side: 8.9e-5 and 5.9e-5."""
    h = lunar_tile(n, g, seed=5, amplitude=3000.0, n_craters=30)
    cam = camera(1280, 720)
    cam["step_m"] = 0.5 * g
    hf = ss.Heightfield(torch.from_numpy(h).cuda(), g, MOON_RADIUS_M, projection=proj)
    uv, pix = ss.ss_view_rays(hf, ss.ss_build_maxmip(hf), cam)
    u, v = oracle.view_hits(h, g, MOON_RADIUS_M, cam, np.arange(1280 * 720), proj=proj)
    hit = ~np.isnan(u)
    assert np.array_equal(pix.cpu().numpy(), np.nonzero(hit)[0])
    ref = np.stack([u[hit], v[hit]], 1)
    keep = ref.min(1) >= 4.0
    got = uv.cpu().numpy()[keep]
    assert len(got) > 200_000
    off = np.abs(got - ref[keep].astype(np.float32)) / np.spacing(np.abs(got))
    assert off.max() <= 1.0
    assert (off > 0.5).mean() <= 2 * 1.6e-8 / 0.3 / g / 6e-5
