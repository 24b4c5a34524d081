"""The scatter with per-block counters and the one with global counters on either side of the capacity at which one
gives way to the other (views of one and of two blocks per SM): the same offsets, and every tile's list equal as a set
to that of ``wsr_bin_static``; in the fixed workspace of both, so that neither depends on what the other left there."""
import ctypes

import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu


def _limit(tiles):
    """The largest capacity that takes the scatter with per-block counters."""
    if tiles <= 12288:
        return 1 << 25
    return min((134_000_000 - 32 * 152 * tiles // 3) // 16 * 5 + 4, 1 << 25)


@pytest.mark.parametrize("size,tile", [((128 * 8, 96 * 8), (8, 8)), ((2560, 1440), (16, 16)), ((256 * 8, 160 * 8), (8, 8))],
                         ids=["12288", "14400", "40960"])
def test_both_scatters_at_the_limit(size, tile):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    from paper_2410_18931_gb300 import _abi as A
    n = 9000
    sc = ws.random_scene(n, 3, sh_degree=0, vd_opacity=False, clusters=4, box=1.0, log_scale_mu=-4.0, log_scale_sd=1.0)
    weight = ws.default_weight(ws.EXP)
    r = Renderer([ws.look_at((0.2, -0.1, -4.0), width=size[0], height=size[1]).rounded()], tile=tile)
    st = r.alloc_state(n)
    r.wsr_project(Gaussians.from_scene(sc), weight.kind, torch.tensor(weight.as_array(), device="cuda"), st.records)
    r.wsr_bin_count(st.records, n, st.tile_offsets)
    total = r.wsr_bin_total()
    off = torch.empty_like(st.tile_offsets)
    lst = torch.empty(total, dtype=torch.int32, device="cuda")
    A.check("wsr_bin_static", r.lib.wsr_bin_static(
        ctypes.c_void_p(st.records.data_ptr()), n, r.cams_c, r.n_cams, ctypes.byref(r.tiles_c),
        ctypes.c_void_p(off.data_ptr()), ctypes.c_void_p(lst.data_ptr()), total, None, None,
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    tile_of = np.repeat(np.arange(r.num_tiles, dtype=np.int64), np.diff(off.cpu().numpy()))
    want = np.sort(tile_of << 32 | lst.cpu().numpy())
    r.workspace.fill_(0xAB)
    for capacity in (_limit(r.num_tiles), _limit(r.num_tiles) + 1, _limit(r.num_tiles)):
        st.tile_list = torch.full((capacity,), -1, dtype=torch.int32, device="cuda")
        r.wsr_bin(st.records, n, st.tile_offsets, st.tile_list)
        assert r.wsr_check() == 0 and r.wsr_bin_total() == total
        assert torch.equal(off, st.tile_offsets)
        got = np.sort(tile_of << 32 | st.tile_list[:total].cpu().numpy())
        assert np.array_equal(got, want) and bool((st.tile_list[total:] == -1).all())
