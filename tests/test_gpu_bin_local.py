"""Binning with per-block counters in shared memory against the pass with global
counters (``wsr_bin_static``): tile offsets equal and every tile's list equal as
a set, at the edges of the two block sizes, of the scan's row counts and of the
list size up to which the scatter takes that path; and the persistent tile
order is a permutation of the tiles (an image rendered by it is the image
rendered tile by tile).
"""
import ctypes

import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu

# (Gaussians, view sizes, tile shape): tile counts 1; 1023 and 1025; 4096 and 4160; 8160; 12288 and 12352 (two
# blocks per SM or one); 16384 and 16512; 40960 and 41040 (shared or global counters); three uneven views
CASES = [
    (1, [(7, 5)], (16, 16)), (255, [(16 * 33, 16 * 31)], (16, 16)), (257, [(16 * 41, 16 * 25 - 3)], (16, 16)),
    (3000, [(64 * 8, 64 * 8)], (8, 8)), (3000, [(65 * 8 - 7, 64 * 8)], (8, 8)), (40_000, [(1920, 1080)], (16, 16)),
    (5000, [(128 * 8, 96 * 8)], (8, 8)), (5000, [(128 * 8 + 1, 95 * 8)], (8, 8)),
    (5000, [(128 * 8, 128 * 8)], (8, 8)), (5000, [(129 * 8, 128 * 8)], (8, 8)),
    (5000, [(256 * 8, 160 * 8)], (8, 8)), (5000, [(270 * 8, 152 * 8)], (8, 8)),
    (20_000, [(640, 360), (57, 43), (1280, 720)], (16, 8)),
]


@pytest.mark.parametrize("n,sizes,tile", CASES, ids=lambda v: str(v).replace(" ", ""))
@pytest.mark.parametrize("long_list", [False, True])
def test_local_counters_give_the_same_lists(n, sizes, tile, long_list):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    from paper_2410_18931_gb300 import _abi as A
    sc = ws.random_scene(n, n, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=-4.0, log_scale_sd=1.0)
    cams = [ws.look_at((0.2, -0.1, -4.0), width=w, height=h).rounded() for w, h in sizes]
    weight = ws.default_weight(ws.EXP)
    g = Gaussians.from_scene(sc)
    wpar = torch.tensor(weight.as_array(), device="cuda")
    r = Renderer(cams, tile=tile)
    st = r.alloc_state(n)
    r.wsr_project(g, weight.kind, wpar, st.records)
    r.wsr_bin_count(st.records, n, st.tile_offsets)
    total = r.wsr_bin_total()
    capacity = (1 << 25) + 1 if long_list else total + 5        # beyond 2^25 entries the scatter's counters are global
    st.tile_list = torch.full((capacity,), -1, dtype=torch.int32, device="cuda")
    r.wsr_bin(st.records, n, st.tile_offsets, st.tile_list)
    assert r.wsr_check() == 0
    off = torch.empty_like(st.tile_offsets)
    lst = torch.full((total + 5,), -1, dtype=torch.int32, device="cuda")
    A.check("wsr_bin_static", r.lib.wsr_bin_static(
        ctypes.c_void_p(st.records.data_ptr()), n, r.cams_c, r.n_cams, ctypes.byref(r.tiles_c),
        ctypes.c_void_p(off.data_ptr()), ctypes.c_void_p(lst.data_ptr()), lst.numel(), None, None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    assert torch.equal(off, st.tile_offsets) and int(off[-1]) == total
    tile_of = np.repeat(np.arange(r.num_tiles), np.diff(off.cpu().numpy()))

    def as_sets(t):
        a = t[:total].cpu().numpy()
        return a[np.lexsort((a, tile_of))]

    assert np.array_equal(as_sets(st.tile_list), as_sets(lst))
    assert (st.tile_list[total:] == -1).all()
    if not long_list:
        # the same image with the persistent schedule's tile order: equal up to the order of FP32 sums
        r.wsr_render_fwd(st.records, n, st.tile_offsets, st.tile_list, weight.kind, wpar, st.rgb, st.den)
        p = Renderer(cams, tile=tile, persistent=True).forward(g, weight.kind, wpar)
        torch.cuda.synchronize()
        assert float((p.rgb - st.rgb).abs().max()) <= 1e-5
