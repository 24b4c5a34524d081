"""The slots that wsr_count_pairs gives for a sparse view's forward: a warp per 16x8 region (8x8 in tiles of that
width), so one region's pixels for every listed Gaussian where a tile is one region, and for every region that it
reaches where a tile has two; the same call with a record count past the sparse limit counts the other kernel's
rounds of four."""
import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8)])
def test_sparse_slots(tile):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(700, 9, sh_degree=0, vd_opacity=False, clusters=0, box=1.0, log_scale_mu=-3.0, log_scale_sd=0.8)
    cam = ws.look_at((0.1, -0.2, -3.0), width=601, height=403).rounded()
    w = ws.default_weight(ws.EXP)
    r = Renderer([cam], tile=tile)
    st = r.forward(Gaussians.from_scene(sc), w.kind, torch.tensor(w.as_array(), device="cuda"))
    pairs, slots, _ = r.wsr_count_pairs(st)
    assert r.num_tiles > 608
    off = st.tile_offsets.cpu().numpy().astype(np.int64)
    lst = st.tile_list.cpu().numpy()[:off[-1]]
    if tile in ((8, 8), (16, 8)):
        assert slots == off[-1] * tile[0] * tile[1]
    else:
        # the regions with a pixel inside the footprint, and those whose widened box a footprint meets
        rec = st.records.cpu().numpy().reshape(-1, 12).astype(np.float64)[lst]
        t = np.repeat(np.arange(r.num_tiles), np.diff(off))
        tx, ty = t % -(-601 // tile[0]), t // -(-601 // tile[0])
        lo = hi = 0
        for k in range(2):
            x0 = tx * tile[0] + (16 * k if tile[0] == 32 else 0) + 0.5 - rec[:, 0]
            y0 = ty * tile[1] + (8 * k if tile[1] == 16 else 0) + 0.5 - rec[:, 1]
            dx, dy = x0[:, None, None] + np.arange(16), y0[:, None, None] + np.arange(8)[:, None]
            qs, qw, qd = (rec[:, c][:, None, None] for c in (2, 3, 4))
            q = (qs * dy + qw * dx) ** 2 + qd * dx ** 2
            lo += int((q <= 9 * 0.7213475).any(axis=(1, 2)).sum())
            # a margin of half a pixel and more of footprint than the kernel's test allows
            fx, fy = (np.linspace(-0.6, n - 0.4, 4 * n + 1) for n in (16, 8))
            dx, dy = x0[:, None, None] + fx, y0[:, None, None] + fy[:, None]
            hi += int(((qs * dy + qw * dx) ** 2 + qd * dx ** 2 <= 9.3 * 0.7213475).any(axis=(1, 2)).sum())
        assert slots % 128 == 0 and lo * 128 <= slots <= hi * 128
    st.n = r.num_pix
    pairs2, slots2, _ = r.wsr_count_pairs(st)
    assert pairs2 == pairs and slots2 != slots if tile != (8, 8) else slots2 <= slots


def test_a_dense_view_keeps_its_batch_from_the_sparse_kernel():
    """Few records for all pixels, but many for a small view's: the whole batch takes the other kernel, and the count
    of its slots is that of one record per pixel (tiles wider than 8; 8x8 ones go by all pixels alone)."""
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(700, 9, sh_degree=0, vd_opacity=False, clusters=0, box=1.0, log_scale_mu=-3.0, log_scale_sd=0.8)
    w = ws.default_weight(ws.EXP)
    for tile in ((16, 16), (32, 8), (16, 8)):
        slots = {}
        for small in (False, True):
            cams = [ws.look_at((0.1, -0.2, -3.0), width=601, height=403).rounded()]
            if small:
                cams.append(ws.look_at((0.1, -0.2, -3.0), width=57, height=43).rounded())
            r = Renderer(cams, tile=tile)
            st = r.forward(Gaussians.from_scene(sc), w.kind, torch.tensor(w.as_array(), device="cuda"))
            own = r.wsr_count_pairs(st)[1]
            st.n = r.num_pix
            slots[small] = own, r.wsr_count_pairs(st)[1]
        assert slots[True][0] == slots[True][1], tile
        assert slots[False][0] != slots[False][1], tile
