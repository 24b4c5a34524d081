"""The backward's schedules in the deterministic mode, whose sums do not depend on which block takes a tile or a part
of its list: the per-tile schedule (tiles as numbered up to 1024, ordered by one kernel up to 16384, else by two) and
the persistent one give the same gradient records and weight gradients, bit for bit, at the edges of those ranges;
with most tiles empty or short (several claimed at once), with lists of several parts (shared by idle blocks), with
fewer tiles than blocks; from a workspace that held anything."""
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu

# (tiles across, down, shape): 1; 35; 608 and 609 (the blocks that fit); 1024 and 1025; 16384 and 16385
CASES = [(1, 1, (16, 16)), (7, 5, (8, 8)), (32, 19, (16, 16)), (29, 21, (8, 8)), (32, 32, (16, 8)), (41, 25, (16, 16)),
         (128, 128, (8, 8)), (145, 113, (8, 8))]


@pytest.mark.parametrize("chunk", [0, 64])
@pytest.mark.parametrize("n", [40, 9000])
@pytest.mark.parametrize("tx,ty,tile", CASES, ids=lambda v: str(v).replace(" ", ""))
def test_schedules_agree(tx, ty, tile, n, chunk):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    from paper_2410_18931_gb300 import _abi as A
    # 9000: most of them in a tight stack, whose tile's list is cut into parts
    sc = ws.random_scene(n, n + 1, sh_degree=0, vd_opacity=False, clusters=0, box=0.8, log_scale_mu=-4.5, log_scale_sd=0.5)
    if n > 40:
        sc.means[:5000] *= 0.004
    cam = ws.look_at((0.0, 0.0, -3.0), width=tx * tile[0] - 3, height=ty * tile[1] - 1)
    cam.cx += 0.4 * tile[0]
    cam = cam.rounded()
    w = ws.default_weight(ws.EXP, c_bg=(0.2, 0.1, 0.3))
    g, wpar = Gaussians.from_scene(sc), torch.tensor(w.as_array(), device="cuda")
    gen = torch.Generator("cuda").manual_seed(3)
    res = []
    for persistent in (False, True):
        r = Renderer([cam], tile=tile, persistent=persistent, chunk=chunk, deterministic=True)
        assert r.num_tiles == tx * ty
        r.workspace.fill_(0xAB)
        st = r.forward(g, w.kind, wpar)
        if not res:
            G = torch.randn(r.num_pix, 3, device="cuda", generator=gen)
        rec = torch.full((n * r.record_floats,), 7.0, device="cuda")
        for _ in range(2):
            r.wsr_render_bwd_tiles(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den, G, rec)
        out = torch.empty(6, device="cuda")
        r.wsr_project_bwd(g, w.kind, wpar, rec, A.wsr_grads(None, None, None, None, None, None, out.data_ptr()))
        torch.cuda.synchronize()
        res.append((st.rgb.clone(), rec.clone().view(torch.int32), out.clone()))
    assert bool((res[0][1] != 0).any())
    for a, b in zip(*res):
        assert torch.equal(a, b)


@pytest.mark.parametrize("tx,ty,tile", [CASES[1], CASES[5], CASES[7]], ids=lambda v: str(v).replace(" ", ""))
def test_default_mode_matches_deterministic(tx, ty, tile):
    """The default mode's record sums against the deterministic mode's exact ones: a record is a sum of one float per
    tile it reaches, at most 50 here, so it lies within 50 2^-24 of their absolute values' sum (the bound kept beside
    the deterministic sums is above that)."""
    import numpy as np
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    n = 9000
    sc = ws.random_scene(n, 5, sh_degree=0, vd_opacity=False, clusters=0, box=0.8, log_scale_mu=-4.5, log_scale_sd=0.5)
    sc.means[:5000] *= 0.004
    cam = ws.look_at((0.0, 0.0, -3.0), width=tx * tile[0] - 3, height=ty * tile[1] - 1).rounded()
    w = ws.default_weight(ws.EXP, c_bg=(0.2, 0.1, 0.3))
    g, wpar = Gaussians.from_scene(sc), torch.tensor(w.as_array(), device="cuda")
    rec = {}
    for det in (False, True):
        r = Renderer([cam], tile=tile, deterministic=det)
        r.workspace.fill_(0xAB)
        st = r.forward(g, w.kind, wpar)
        if det:
            st.rgb.copy_(image[0])
            st.den.copy_(image[1])
        else:
            G = torch.randn(r.num_pix, 3, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
            image = st.rgb.clone(), st.den.clone()
        out = torch.empty(n * r.record_floats, device="cuda")
        r.wsr_render_bwd_tiles(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den, G, out)
        rec[det] = out.cpu().numpy().reshape(n, r.record_floats)
    bounds = rec[True][:, 18:27].astype(np.float64)
    exact = np.where(bounds > 0, np.ldexp(rec[True][:, :18].copy().view(np.int64).astype(np.float64), np.frexp(bounds)[1] - 60), 0.0)
    assert (exact != 0).any()
    assert (np.abs(rec[False][:, :9] - exact) <= 50 * 2.0 ** -24 * bounds + 1e-30).all()
