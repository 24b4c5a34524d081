"""The forward's two kernels for more than 608 tiles against the oracle and each other.  Which one renders depends on the
record count passed alone: n itself takes the one for sparse views here, one record per pixel the other."""
import numpy as np
import pytest

import oracle
import wsr_scenes as ws
from tests.gpu_util import TIE, assert_image_parity

pytestmark = pytest.mark.gpu

TILES = [(16, 16), (8, 8), (32, 8), (16, 8)]


def _both(sc, cam, w, tile, persistent=False):
    """(image, denominator) by the kernel for sparse views, then by the other."""
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    wpar = torch.tensor(w.as_array(), device="cuda")
    r = Renderer([cam], tile=tile, persistent=persistent)
    assert r.num_tiles > 608
    g = Gaussians.from_scene(sc)
    st = r.forward(g, w.kind, wpar)
    out = []
    for n in (1, r.num_pix):
        st.rgb.fill_(-7.0)
        st.den.fill_(-7.0)
        r.wsr_render_fwd(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den)
        out.append((st.rgb.cpu().numpy().reshape(cam.height, cam.width, 3), st.den.cpu().numpy()))
    return out


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("n", [1, 3, 4, 5, 31, 33, 64, 65, 127, 128, 129, 257, 515])
def test_list_lengths_with_one_slice(n, tile):
    """Lists around the rounds of four and the batches of 32, 64 and 128 entries, at the meeting point of four tiles."""
    sc = ws.random_scene(n, 100 + n, sh_degree=1, vd_opacity=True, clusters=0, box=0.02, log_scale_mu=-4.0,
                         log_scale_sd=0.6)
    cam = ws.look_at((0.0, 0.0, -3.0), width=513, height=313)
    cam.cx, cam.cy = 32.0 * (513 // 64), 16.0 * (313 // 32)
    cam = cam.rounded()
    w = ws.default_weight(ws.EXP, c_bg=(0.2, 0.1, 0.3))
    ref = oracle.render(sc, cam, w, amb_tau=TIE)
    for rgb, den in _both(sc, cam, w, tile):
        assert_image_parity(rgb, ref)
        assert np.isfinite(den).all()


@pytest.mark.parametrize("tile", TILES)
@pytest.mark.parametrize("persistent", [False, True])
def test_close_up(tile, persistent):
    """A few wide Gaussians over the whole view: every tile's list holds several batches, and the kernels' images
    agree up to the order of 32-bit sums (they decide a pair at the cutoff by the same operations): 900 terms, each
    sum within 900 2^-24 of its terms' absolute values."""
    sc = ws.random_scene(900, 4, sh_degree=0, vd_opacity=False, clusters=0, box=1.2, log_scale_mu=-0.8, log_scale_sd=0.4)
    cam = ws.look_at((0.1, -0.2, -3.0), width=601, height=403).rounded()
    w = ws.default_weight(ws.EXP)
    (a, da), (b, db) = _both(sc, cam, w, tile, persistent)
    assert np.abs(da / db - 1.0).max() <= 2 * 900 * 2.0 ** -24
    assert np.abs(a - b).max() <= 2 * 900 * 2.0 ** -24 * 4.0        # colours of at most about 2, numerator and denominator
