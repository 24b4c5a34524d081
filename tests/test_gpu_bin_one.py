"""The binning of small scenes in one launch against the pass with global counters (``wsr_bin_static``): offsets
equal and every tile's list equal as a set, at both limits of its range and one beyond them; the persistent tile order
a permutation, longest first by bucket; a list that is too short; no Gaussians at all."""
import ctypes

import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu

# (Gaussians, view sizes, tile shape): 1, 1024, 1025, 4096 and 4160 tiles; 8192 and 8193, 4096 and 4097 Gaussians;
# batches of 32 that end early; several uneven views, whose batches follow one another
CASES = [
    (0, [(40, 30)], (16, 16)), (1, [(7, 5)], (16, 16)), (33, [(250, 140)], (32, 8)), (8192, [(512, 512)], (16, 16)),
    (8193, [(512, 512)], (16, 16)), (4096, [(41 * 16, 25 * 16 - 3)], (16, 16)), (4097, [(41 * 16, 25 * 16)], (16, 16)),
    (4000, [(64 * 8, 64 * 8)], (8, 8)), (4000, [(65 * 8, 64 * 8)], (8, 8)),
    (1365, [(320, 180), (57, 43), (200, 120)], (16, 8)), (1366, [(640, 360), (57, 43), (200, 120)], (16, 16)),
]


def _scene(n, sizes, tile, **kw):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(max(n, 1), n + 1, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=-4.0,
                         log_scale_sd=1.0)
    cams = [ws.look_at((0.2, -0.1, -4.0), width=w, height=h).rounded() for w, h in sizes]
    weight = ws.default_weight(ws.EXP)
    r = Renderer(cams, tile=tile, **kw)
    st = r.alloc_state(max(n, 1))
    r.wsr_project(Gaussians.from_scene(sc), weight.kind, torch.tensor(weight.as_array(), device="cuda"), st.records)
    return r, st


def _static(r, st, n, capacity):
    import torch

    from paper_2410_18931_gb300 import _abi as A
    off = torch.empty_like(st.tile_offsets)
    lst = torch.full((max(capacity, 1),), -1, dtype=torch.int32, device="cuda")
    cams = A.make_cameras(r.cams)[0]
    tiles = A.tiles(*r.tile, A.WSR_SCHEDULE_TILE_BLOCKS, 0, 0)
    A.check("wsr_bin_static", r.lib.wsr_bin_static(
        ctypes.c_void_p(st.records.data_ptr()), n, cams, r.n_cams, ctypes.byref(tiles),
        ctypes.c_void_p(off.data_ptr()), ctypes.c_void_p(lst.data_ptr()), capacity, None, None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return off, lst


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("n,sizes,tile", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_one_launch_gives_the_same_lists(n, sizes, tile, persistent):
    import torch
    r, st = _scene(n, sizes, tile, persistent=persistent)
    r.wsr_bin_count(st.records, n, st.tile_offsets)
    total = r.wsr_bin_total()
    off, lst = _static(r, st, n, total)
    st.tile_list = torch.full((total + 5,), -1, dtype=torch.int32, device="cuda")
    r.capacity = total + 5
    r.workspace.fill_(0xAB)                     # nothing is expected of an earlier call
    st.tile_offsets.fill_(-1)
    for _ in range(2):
        r.wsr_bin(st.records, n, st.tile_offsets, st.tile_list)
        assert r.wsr_check() == 0 and r.wsr_bin_total() == total
        assert torch.equal(off, st.tile_offsets) and int(off[-1]) == total
        tile_of = np.repeat(np.arange(r.num_tiles), np.diff(off.cpu().numpy()))
        key = [np.sort(tile_of.astype(np.int64) << 32 | t[:total].cpu().numpy()) for t in (lst, st.tile_list)]
        assert np.array_equal(*key) and (st.tile_list[total:] == -1).all()


def test_one_launch_order_renders_every_tile():
    """The persistent schedule's image is the image rendered tile by tile: the order names every tile once."""
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(3000, 7, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=-4.0, log_scale_sd=1.0)
    weight = ws.default_weight(ws.EXP)
    g, w = Gaussians.from_scene(sc), torch.tensor(weight.as_array(), device="cuda")
    for size in ((500, 500), (1000, 700)):
        cam = ws.look_at((0.2, -0.1, -4.0), width=size[0], height=size[1]).rounded()
        img = []
        for p in (False, True):
            r = Renderer([cam], persistent=p)
            st = r.forward(g, weight.kind, w)
            st.rgb.fill_(-7.0)
            r.forward(g, weight.kind, w, st)
            img.append(st.rgb.clone())
        assert torch.allclose(img[0], img[1], rtol=0, atol=1e-5)       # lists in any order: sums of 32-bit terms


@pytest.mark.parametrize("short", [0, 1, 100])
def test_one_launch_short_list(short):
    """Capacity below the total: the status and the total say so, the offsets stay within the capacity, nothing is
    written behind it."""
    import torch

    from paper_2410_18931_gb300 import _abi as A
    n = 2000
    r, st = _scene(n, [(200, 120)], (16, 16))
    r.wsr_bin_count(st.records, n, st.tile_offsets)
    total = r.wsr_bin_total()
    capacity = short if short != 1 else total - 1
    buf = torch.full((capacity + 64,), -1, dtype=torch.int32, device="cuda")
    r.capacity = capacity
    st.tile_list = buf[:capacity]
    r.wsr_bin(st.records, n, st.tile_offsets, st.tile_list)
    assert r.wsr_bin_total() == total and r.wsr_check() == A.WSR_ERR_CAPACITY
    assert int(st.tile_offsets.max()) == capacity and (buf[capacity:] == -1).all()
