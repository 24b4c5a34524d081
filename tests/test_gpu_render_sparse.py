"""The forward's kernel for sparse views against the other one, which its own tests hold against the oracle: odd and
even widths, a second view that starts at an odd pixel, every tile shape, both schedules, unaligned outputs, lists
longer than a batch, empty tiles.  Both decide a pair at the cutoff by the same operations, so only the order of the
sums differs."""
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu

VIEWS = [[(640, 480)], [(641, 483), (640, 480)], [(337, 241), (800, 301)]]


def _setup(n, sizes, tile, persistent, mu=-3.5):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(n, n, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=mu, log_scale_sd=0.8)
    cams = [ws.look_at((0.2, -0.1 + 0.3 * k, -4.0), width=w, height=h).rounded() for k, (w, h) in enumerate(sizes)]
    weight = ws.default_weight(ws.EXP)
    r = Renderer(cams, tile=tile, persistent=persistent)
    return sc, cams, weight, r, Gaussians.from_scene(sc), torch.tensor(weight.as_array(), device="cuda")


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8)])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("sizes", VIEWS, ids=lambda s: "+".join("%dx%d" % v for v in s))
def test_both_kernels_agree_and_stay_inside(sizes, persistent, tile, shift):
    """The same records rendered as a sparse view and, by passing a larger record count (only the route depends on it),
    by the other kernel: equal up to the order of 32-bit sums, whatever the outputs' alignment, and nothing beside
    them is written."""
    import torch
    sc, cams, weight, r, g, w = _setup(900, sizes, tile, persistent, mu=-2.5)
    st = r.forward(g, weight.kind, w)
    P = r.num_pix
    images = []
    many = 9 * r.num_tiles * tile[0] * tile[1] // 1024 // r.n_cams + 1
    assert r.num_tiles > 608 and many > 900
    for n in (900, many):
        buf = torch.full((3 * P + 16,), -7.0, device="cuda")
        bd = torch.full((P + 16,), -7.0, device="cuda")
        rgb, den = buf[shift:shift + 3 * P], bd[shift:shift + P]
        r.wsr_render_fwd(st.records, n, st.tile_offsets, st.tile_list, weight.kind, w, rgb, den)
        torch.cuda.synchronize()
        assert (buf[:shift] == -7.0).all() and (buf[shift + 3 * P:] == -7.0).all()
        assert (bd[:shift] == -7.0).all() and (bd[shift + P:] == -7.0).all()
        images.append((rgb.clone(), den.clone()))
    assert torch.allclose(images[0][0], images[1][0], rtol=0, atol=1e-5)
    assert torch.allclose(images[0][1], images[1][1], rtol=1e-5, atol=0)
