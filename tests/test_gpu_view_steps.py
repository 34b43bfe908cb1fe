"""View rays at the edges of their fast paths against the FP64 view oracle: steps much
shorter and much longer than a texel (the crossing lies in one, two or many cells),
tiny images, cameras below the highest terrain, tiles whose low edges are in view, a
frame that is not normalised.  Bars as in test_gpu_view.py: the same pixels hit,
coordinates within one float32 step."""
import numpy as np
import pytest

import oracle
from test_gpu_view import R, _check_hits, _gpu_view
from workloads import camera, lunar_tile

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("proj", ["polar_stereo", "gnomonic"])
@pytest.mark.parametrize("step_texels", [0.05, 0.5, 1.7, 9.0])
def test_step_lengths(proj, step_texels):
    g = 60.0
    h = lunar_tile(700, g, seed=17, amplitude=2500.0, n_craters=12)
    cam = camera(97, 55)
    cam["step_m"] = step_texels * g
    _, _, uv, pix = _gpu_view(h, g, proj, cam)
    u, v = oracle.view_hits(h, g, R, cam, np.arange(97 * 55), proj=proj)
    idx, _ = _check_hits(uv.cpu().numpy(), pix.cpu().numpy(), u, v, np.arange(97 * 55))
    assert len(idx) > 500


@pytest.mark.parametrize("w,hgt", [(1, 1), (31, 1), (33, 3), (257, 5)])
def test_small_images(w, hgt):
    h = lunar_tile(400, 90.0, seed=3, amplitude=2000.0, n_craters=8)
    cam = camera(w, hgt)
    cam["right"] = np.asarray(cam["right"]) * 1e20     # the frame's scale is free with the
    cam["tan_x"] /= 1e20                               # tangent: d is normalised
    _, _, uv, pix = _gpu_view(h, 90.0, "polar_stereo", cam)
    u, v = oracle.view_hits(h, 90.0, R, cam, np.arange(w * hgt))
    _check_hits(uv.cpu().numpy(), pix.cpu().numpy(), u, v, np.arange(w * hgt))


@pytest.mark.parametrize("alt", [1500.0, 4.0e5])
def test_low_and_high_camera(alt):
    """Below the highest terrain (rays start among it), and far above it."""
    g = 80.0
    h = lunar_tile(600, g, seed=23, amplitude=3000.0, n_craters=12)
    cam = camera(120, 68)
    up = np.asarray(cam["pos"]) / np.linalg.norm(cam["pos"])
    cam["pos"] = (R + alt) * up
    if alt > 1e5:
        cam["max_dist_m"] = 3.0 * alt
        fwd = np.array([0.0, 0.0, R]) - cam["pos"]
        cam["forward"] = fwd / np.linalg.norm(fwd)
        cam["right"] = np.array([1.0, 0.0, 0.0])
        cam["up"] = np.cross(cam["right"], cam["forward"])
        cam["tan_x"], cam["tan_y"] = 0.09, 0.05
    cam["step_m"] = 0.5 * g
    _, _, uv, pix = _gpu_view(h, g, "polar_stereo", cam)
    u, v = oracle.view_hits(h, g, R, cam, np.arange(120 * 68))
    idx, _ = _check_hits(uv.cpu().numpy(), pix.cpu().numpy(), u, v, np.arange(120 * 68))
    assert len(idx) > 1000
