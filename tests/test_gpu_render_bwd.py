"""The backward's rows and classes against the oracle: thin footprints at many
angles, round ones from a pixel to a tile wide, in every tile shape, with
every chunk size.
"""
import numpy as np
import pytest

import wsr_scenes as ws
from tests.gpu_util import GRAD_TOL, grad_envelope, grad_excess

pytestmark = pytest.mark.gpu
KEYS = ("means", "log_scales", "quats", "sh", "opacity")


def _scene(kind, n=400):
    rng = np.random.default_rng(31)
    sc = ws.random_scene(n, 32, sh_degree=1, vd_opacity=False, box=0.9)
    if kind == "needles":                        # seen face on, turned about the view axis through every angle
        half = 0.5 * rng.uniform(0.0, np.pi, n)
        sc.quats[:] = np.stack([np.cos(half), 0 * half, 0 * half, np.sin(half)], 1)
        sc.log_scales[:] = np.log(1e-3)
        sc.log_scales[:, 0] = rng.uniform(np.log(0.05), np.log(0.6), n)
        sc.means[:, 2] *= 0.2
    else:                                        # 3-sigma radii from the dilation alone to about a tile
        sc.log_scales[:] = rng.uniform(np.log(1e-3), np.log(0.12), n)[:, None]
    return sc


@pytest.mark.parametrize("kind", ["needles", "round"])
@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8)])
@pytest.mark.parametrize("chunk", [64, 512])
def test_backward_rows_and_classes(kind, tile, chunk):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = _scene(kind)
    cam = ws.look_at((0.0, 0.0, -3.0), width=131, height=93).rounded()
    w = ws.WeightParams(ws.EXP, 0.1, 0.8, 0.9, (0.1, 0.2, 0.1))
    g = Gaussians.from_scene(sc)
    wpar = torch.tensor(w.as_array(), device="cuda")
    r = Renderer([cam], tile=tile, chunk=chunk)
    st = r.forward(g, w.kind, wpar)
    G = np.random.default_rng(5).normal(size=(cam.height, cam.width, 3)).astype(np.float32)
    out = r.backward(g, w.kind, wpar, st, torch.tensor(G, device="cuda").reshape(-1, 3))
    env = grad_envelope(sc, cam, w, G.astype(np.float64))
    for k in KEYS:
        if kind == "round" and k == "quats":
            continue                             # a sphere has no orientation: the gradient is zero
        ex = grad_excess(out[k].cpu().numpy(), env, k)
        assert ex <= GRAD_TOL, (k, ex)


@pytest.mark.parametrize("n,size", [(5000, (64, 48)), (4097, (64, 48)), (9000, (480, 352)), (9000, (16 * 41, 240))])
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("chunk", [0, 128, 512])
def test_split_lists_give_the_gradients_of_one_block_per_list(n, size, persistent, chunk):
    """Most of the Gaussians on one tile, so that its list has many parts (few tiles: a chunk each; more: four), taken
    by several blocks: the gradients are the deterministic mode's (exact integer sums) up to FP32 rounding."""
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    sc = ws.random_scene(n, 7, sh_degree=0, vd_opacity=False, box=0.02, log_scale_mu=-5.0, log_scale_sd=0.4)
    sc.means[::50] *= 60.0                       # a few elsewhere
    cam = ws.look_at((0.0, 0.0, -3.0), width=size[0], height=size[1])
    cam.cx, cam.cy = 24.0, 24.0                  # the cluster in the middle of the second tile
    cam = cam.rounded()
    w = ws.default_weight(ws.EXP)
    g = Gaussians.from_scene(sc)
    wpar = torch.tensor(w.as_array(), device="cuda")
    G = torch.tensor(np.random.default_rng(3).normal(size=(size[0] * size[1], 3)).astype(np.float32), device="cuda")
    outs = []
    for det in (False, True):
        r = Renderer([cam], tile=(16, 16), chunk=chunk, persistent=persistent, deterministic=det)
        st = r.forward(g, w.kind, wpar, check=not det)           # the list may be too long for the mode's sort
        r.wsr_check()
        outs.append(r.backward(g, w.kind, wpar, st, G))
        longest = int(torch.diff(st.tile_offsets).max())
    assert longest > 2048
    for k in (*KEYS, "weight_params"):
        a, b = outs[0][k].double(), outs[1][k].double()
        assert float((a - b).abs().max()) <= 1e-4 * max(float(b.abs().max()), 1e-12), k
