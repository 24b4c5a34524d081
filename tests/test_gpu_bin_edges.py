"""Binning with per-block counters where it begins and ends: few Gaussians over more tiles than the binning in one
launch takes (one block, partial batches), and that many tiles and one more at its own edges; and the persistent tile
order itself, for every kernel that makes it."""
import ctypes

import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu


def _binned(n, sizes, tile, capacity=None, persistent=False, seed=None):
    """(renderer, state, total): n Gaussians binned by wsr_bin from a workspace that held anything."""
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(n, seed or n, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=-4.0,
                         log_scale_sd=1.0)
    weight = ws.default_weight(ws.EXP)
    r = Renderer([ws.look_at((0.2, -0.1, -4.0), width=w, height=h).rounded() for w, h in sizes], tile=tile,
                 persistent=persistent)
    st = r.alloc_state(n)
    r.wsr_project(Gaussians.from_scene(sc), weight.kind, torch.tensor(weight.as_array(), device="cuda"), st.records)
    r.wsr_bin_count(st.records, n, st.tile_offsets)
    total = r.wsr_bin_total()
    st.tile_list = torch.full((capacity or total + 5,), -1, dtype=torch.int32, device="cuda")
    r.workspace.fill_(0xAB)
    st.tile_offsets.fill_(-1)
    r.wsr_bin(st.records, n, st.tile_offsets, st.tile_list)
    assert r.wsr_check() == 0 and r.wsr_bin_total() == total
    return r, st, total


# one block and partial batches beyond 4096 tiles; 1, 1023, 1025 and 4096 tiles beyond the one launch's Gaussians
# (8192, and 4096 past 1024 tiles); the same beside a small view
CASES = [(n, [(65 * 8, 64 * 8)], (8, 8)) for n in (1, 31, 32, 33, 255, 257)] + [
    (8193, [(7, 5)], (16, 16)), (8193, [(16 * 33, 16 * 31)], (16, 16)), (4097, [(16 * 41, 16 * 25 - 3)], (16, 16)),
    (4097, [(64 * 8, 64 * 8)], (8, 8)), (33, [(65 * 8, 64 * 8), (57, 43)], (8, 8)),
    (100, [(270 * 8, 152 * 8)], (8, 8)),
]


@pytest.mark.parametrize("long_list", [False, True])
@pytest.mark.parametrize("n,sizes,tile", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_same_lists_as_global_counters(n, sizes, tile, long_list):
    import torch

    from paper_2410_18931_gb300 import _abi as A
    r, st, total = _binned(n, sizes, tile, capacity=(1 << 25) + 1 if long_list else None)
    assert r.bin_launches(n) > 1                # not the binning in one launch
    off = torch.empty_like(st.tile_offsets)
    lst = torch.full((total + 5,), -1, dtype=torch.int32, device="cuda")
    A.check("wsr_bin_static", r.lib.wsr_bin_static(
        ctypes.c_void_p(st.records.data_ptr()), n, r.cams_c, r.n_cams, ctypes.byref(r.tiles_c),
        ctypes.c_void_p(off.data_ptr()), ctypes.c_void_p(lst.data_ptr()), lst.numel(), None, None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    assert torch.equal(off, st.tile_offsets) and int(off[-1]) == total
    tile_of = np.repeat(np.arange(r.num_tiles, dtype=np.int64), np.diff(off.cpu().numpy()))
    a, b = (np.sort(tile_of << 32 | t[:total].cpu().numpy()) for t in (st.tile_list, lst))
    assert np.array_equal(a, b) and bool((st.tile_list[total:] == -1).all())


def _order(r):
    """The tile order in the workspace: behind the 8 KB header, the buckets (66 words), two arrays of tiles + 1 words
    and the scan's sums (8 bytes per 4096 tiles and one more), each rounded up to 256 bytes."""
    t, up = r.num_tiles, lambda x: (x + 255) // 256 * 256
    at = 8192 + up(4 * 66) + 2 * up(4 * (t + 1)) + up(8 * ((t + 4095) // 4096 + 1))
    return r.workspace[at:at + 4 * t].cpu().numpy().view(np.uint32)


def _is_longest_first(order, offsets):
    counts = np.diff(offsets.cpu().numpy().astype(np.int64))
    assert np.array_equal(np.sort(order), np.arange(len(counts)))
    bucket = np.where(counts > 0, np.frexp(np.maximum(counts, 1))[1], 0)        # floor(log2(count)) + 1, 0 if empty
    assert len(set(bucket)) > 3
    assert (np.diff(bucket[order]) <= 0).all()


# the binning in one launch (up to 1024 tiles and up to 4096); the scan by one, four, eight and sixteen rows of 32
# tiles per warp; the scan of up to 32768 tiles from shared memory; beyond that the two ordering kernels
ORDERS = [(900, (16 * 20, 16 * 15), (16, 16)), (900, (64 * 8, 64 * 8), (8, 8)), (9000, (32 * 8, 32 * 8), (8, 8)),
          (9000, (64 * 8, 64 * 8), (8, 8)), (9000, (128 * 8, 64 * 8), (8, 8)), (9000, (128 * 8, 128 * 8), (8, 8)),
          (9000, (200 * 8, 160 * 8), (8, 8)), (9000, (270 * 8, 152 * 8), (8, 8))]


@pytest.mark.parametrize("n,size,tile", ORDERS, ids=lambda v: str(v).replace(" ", ""))
def test_persistent_order(n, size, tile):
    r, st, _ = _binned(n, [size], tile, persistent=True, seed=3)
    _is_longest_first(_order(r), st.tile_offsets)


# the backward's own order with the per-tile schedule: one kernel of four, eight and sixteen rows, and the two kernels
@pytest.mark.parametrize("size", [(41 * 8, 25 * 8), (64 * 8, 65 * 8), (128 * 8, 65 * 8), (129 * 8, 128 * 8), (270 * 8, 152 * 8)],
                         ids=lambda v: str(v).replace(" ", ""))
def test_order_of_the_per_tile_schedule(size):
    import torch
    n = 9000
    r, st, _ = _binned(n, [size], (8, 8), seed=3)
    w = ws.default_weight(ws.EXP)
    wpar = torch.tensor(w.as_array(), device="cuda")
    r.wsr_render_fwd(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den)
    rec = torch.empty(n * r.record_floats, device="cuda")
    r.wsr_render_bwd_tiles(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den,
                           torch.ones(r.num_pix, 3, device="cuda"), rec)
    _is_longest_first(_order(r), st.tile_offsets)
