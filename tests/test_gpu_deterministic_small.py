"""The deterministic mode's gradient records where the terms' bounds are subnormal floats: their exponents reach -148.
The records of an image gradient of about 2^scale are those of the same gradient at 1, scaled: a pixel's term is
rounded to a multiple of 2^-149 twice (in the pixel table and in its product with the Gaussian's value there, at most
1), sums of such multiples are exact, so a record's sum over its npx pixels lies within npx 2^-149 of the scaled one,
beside the 32-bit rounding of the other (a few 2^-24 per term)."""
import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu


def _records(r, st, n, w, wpar, G):
    import torch
    out = torch.empty(n * r.record_floats, device="cuda")
    r.wsr_render_bwd_tiles(st.records, n, st.tile_offsets, st.tile_list, w.kind, wpar, st.rgb, st.den, G, out)
    rec = out.cpu().numpy().reshape(n, r.record_floats)
    bounds = rec[:, 18:27].astype(np.float64)
    sums = rec[:, :18].copy().view(np.int64).astype(np.float64)
    return np.where(bounds > 0, np.ldexp(sums, np.frexp(bounds)[1] - 60), 0.0), bounds


@pytest.mark.parametrize("scale", [-141, -139, -137])
def test_subnormal_bounds(scale):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    n = 300
    sc = ws.random_scene(n, 5, sh_degree=0, vd_opacity=False, clusters=0, box=0.6, log_scale_mu=-5.0, log_scale_sd=0.4)
    cam = ws.look_at((0.0, 0.0, -3.0), width=120, height=90).rounded()
    w = ws.default_weight(ws.EXP)
    g, wpar = Gaussians.from_scene(sc), torch.tensor(w.as_array(), device="cuda")
    r = Renderer([cam], deterministic=True)
    st = r.forward(g, w.kind, wpar)
    gen = torch.Generator().manual_seed(7)
    G = (1.0 + torch.rand(r.num_pix, 3, generator=gen)).cuda()          # one sign: nothing cancels
    pmax = float((G / st.den[:, None]).max())
    want, bounds = _records(r, st, n, w, wpar, G)
    got, tiny = _records(r, st, n, w, wpar, (G.double() * 2.0 ** scale).float())
    npx = bounds[:, 6:7] / pmax
    seen = bounds[:, 6] > 0
    assert seen.sum() > 100 and tiny[seen, 6].max() < 2.0 ** -129
    ref = want[:, 6:9] * 2.0 ** scale                                   # d/d(c u w): sums of G / D times the value
    tol = npx * 2.0 ** -149 + 64 * 2.0 ** -24 * np.abs(ref)
    assert (np.abs(ref) > 4 * tol).sum() > 100                          # the tolerance leaves most of them standing
    assert (np.abs(got[:, 6:9] - ref) <= tol).all()
