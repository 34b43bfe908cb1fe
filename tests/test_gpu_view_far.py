"""View rays of distant cameras against the FP64 view oracle: the float32 march's error
grows with the camera's distance over the texel size (positions) and with its height over
the radius (heights), and where it could decide a sample, the sample is decided exactly.
Bars as in test_gpu_view.py: the same pixels hit, coordinates within one float32 step."""
import numpy as np
import pytest

import oracle
from test_gpu_view import _check_hits, _dev

import paper_2005_06671_gb300 as ss

pytestmark = pytest.mark.gpu


def _look_at_centre(R, alt, dist, az, width, height, half_m):
    """A camera `alt` over the sphere, `dist` along it from the tile's centre, aimed at the
    centre, that sees half_m to each side of it."""
    th = dist / R
    up = np.array([np.sin(th) * np.sin(az), np.sin(th) * np.cos(az), np.cos(th)])
    pos = (R + alt) * up
    fwd = np.array([0.0, 0.0, R]) - pos
    far = np.linalg.norm(fwd)
    fwd = fwd / far
    right = np.cross(fwd, up)
    right = right / np.linalg.norm(right)
    return dict(pos=pos, forward=fwd, right=right, up=np.cross(right, fwd), tan_x=half_m / far,
                tan_y=half_m / far * height / width, width=width, height=height,
                max_dist_m=far + 4.0 * half_m + 2e4)


def _compare(h, g, R, proj, cam):
    W, H = cam["width"], cam["height"]
    hf = ss.Heightfield(_dev(h), g, R, projection=proj)
    uv, pix = ss.ss_view_rays(hf, ss.ss_build_maxmip(hf), cam)
    u, v = oracle.view_hits(h, g, R, cam, np.arange(W * H), proj=proj)
    idx, _ = _check_hits(uv.cpu().numpy(), pix.cpu().numpy(), u, v, np.arange(W * H))
    return len(idx)


# The tile is a plateau: rays below its top meet it at the border, where the first sample
# inside is the hit, so a position 0.01 texel off decides it wrongly for every fiftieth.
@pytest.mark.parametrize("proj", ["polar_stereo", "gnomonic"])
@pytest.mark.parametrize("g,alt,dist", [(1.0, 200e3, 300e3), (2.0, 100e3, 300e3), (0.5, 60e3, 400e3)])
def test_plateau_border_from_afar(proj, g, alt, dist):
    rng = np.random.default_rng(int(alt))
    n = 300
    h = (150.0 * g + 3.0 * g * rng.standard_normal((n, n))).astype(np.float32)
    cam = _look_at_centre(1737.4e3, alt, dist, 0.6, 320, 240, 0.8 * n * g)
    cam["step_m"] = 0.5 * g
    assert _compare(h, g, 1737.4e3, proj, cam) > 10000


# Cameras several radii away from a small body: rise() cancels, to 10 m, on flat ground.
@pytest.mark.parametrize("proj", ["polar_stereo", "gnomonic"])
@pytest.mark.parametrize("alt,dist", [(3.9e6, 40e3), (2.5e6, 150e3)])
def test_small_body_from_many_radii(proj, alt, dist):
    rng = np.random.default_rng(int(dist))
    n, g, R = 200, 3.0, 200e3
    h = 0.1 * rng.standard_normal((n, n))
    cam = _look_at_centre(R, alt, dist, 2.0, 160, 120, 0.4 * n * g)
    cam["step_m"] = 0.5 * g
    assert _compare(h.astype(np.float32), g, R, proj, cam) > 10000


@pytest.mark.parametrize("max_dist", [3e5, 2e9])
def test_hits_do_not_depend_on_max_dist(max_dist):
    rng = np.random.default_rng(1)
    n, g, R = 512, 20.0, 1737.4e3
    h = (500.0 * np.sin(np.arange(n) / 30.0)[None, :] + rng.standard_normal((n, n))).astype(np.float32)
    cam = _look_at_centre(R, 8e3, 20e3, 1.0, 160, 90, 4e3)
    cam.update(step_m=10.0, max_dist_m=max_dist)
    assert _compare(h, g, R, "polar_stereo", cam) > 5000
