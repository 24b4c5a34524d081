"""The forward against the oracle where its rounds and slices end: tile lists
around its rounds of four Gaussians and its batches (32, 64 and 128 entries),
with one and with two slices of the list per tile, for every tile shape.
"""
import numpy as np
import pytest

import oracle
import wsr_scenes as ws

from tests.gpu_util import TIE, assert_image_parity, gpu_render

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8)])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 33, 64, 65, 127, 128, 129, 257, 515])
@pytest.mark.parametrize("size", [(37, 21), (513, 313)])        # up to 608 tiles: two slices; more: one
def test_forward_list_lengths(n, tile, size):
    sc = ws.random_scene(n, 100 + n, sh_degree=1, vd_opacity=True, clusters=0, box=0.02, log_scale_mu=-4.0,
                         log_scale_sd=0.6)
    # the cluster sits at the meeting point of four tiles near the image's middle
    cam = ws.look_at((0.0, 0.0, -3.0), width=size[0], height=size[1])
    cam.cx, cam.cy = 32.0 * (size[0] // 64), 16.0 * (size[1] // 32)
    cam = cam.rounded()
    w = ws.default_weight(ws.EXP, c_bg=(0.2, 0.1, 0.3))
    (rgb, den), = gpu_render(sc, [cam], w, tile=tile)
    ref = oracle.render(sc, cam, w, amb_tau=TIE)
    assert_image_parity(rgb, ref)
    assert np.isfinite(den).all()
