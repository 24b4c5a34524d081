"""The projection backward's rows in shared memory: a Gaussian's gradients do not
depend on where it lies in a block (every value is formed by one thread), at the
ends of blocks, for every SH degree, opacity mode and storage, one view and
several, and for outputs aligned only to their elements.
"""
import numpy as np
import pytest

import wsr_scenes as ws

pytestmark = pytest.mark.gpu
NAMES = ("means", "log_scales", "quats", "sh", "opacity", "lc_v")


@pytest.mark.parametrize("reduced", [False, True])
@pytest.mark.parametrize("vd", [False, True])
@pytest.mark.parametrize("degree", [0, 1, 2, 3])
@pytest.mark.parametrize("n_views", [1, 3])
def test_rows_of_every_shape(degree, vd, reduced, n_views):
    import torch

    from paper_2410_18931_gb300 import Gaussians, Renderer
    from paper_2410_18931_gb300 import _abi as A
    n = 389
    sc = ws.random_scene(n, 40 + degree, sh_degree=degree, vd_opacity=vd, box=1.0, log_scale_mu=-3.0)
    cams = [ws.look_at(p, width=64, height=48).rounded() for p in ((0, 0, -4.0), (3.0, 1.0, -3.0), (-2.0, 2.0, 3.0))]
    w = ws.default_weight(ws.LC)
    wpar = torch.tensor(w.as_array(), device="cuda")
    r = Renderer(cams[:n_views], tile=(16, 16))
    rec = np.random.default_rng(1).normal(size=(n_views, n, 12)).astype(np.float32)
    rec[:, ::7] = 0.0                                # Gaussians that no pixel saw

    def run(first, count, off):
        """Gradients of Gaussians [first, first + count); outputs start ``off`` floats past a 16-byte boundary."""
        g = Gaussians.from_scene(sc.subset(np.arange(first, first + count)), reduced=reduced)
        gr = torch.tensor(rec[:, first:first + count].copy(), device="cuda").reshape(-1)
        bufs = [torch.full((getattr(g, k).numel() + 8,), 7.0, device="cuda") for k in NAMES]
        outs = [b[off:off + getattr(g, k).numel()] for b, k in zip(bufs, NAMES)]
        # quaternion gradients, and rows of 16 bytes that stay in registers (degree 1), are stored as float4
        for i, k in enumerate(NAMES):
            if k == "quats" or (degree == 1 and k in ("sh", "opacity")):
                outs[i] = bufs[i][:getattr(g, k).numel()]
        r.wsr_project_bwd(g, w.kind, wpar, gr, A.wsr_grads(*[o.data_ptr() for o in outs], None))
        for b, o in zip(bufs, outs):                 # nothing is written beside the outputs
            at = o.storage_offset()
            assert bool((b[:at] == 7.0).all()) and bool((b[at + o.numel():] == 7.0).all())
        return [o.cpu().numpy().reshape(count, -1).copy() for o in outs]

    whole = run(0, n, 0)
    assert all(np.isfinite(a).all() for a in whole) and np.abs(whole[3]).max() > 0
    for first, count, off in ((0, n, 1), (0, 1, 0), (5, 127, 0), (5, 127, 3), (130, 128, 0), (3, 129, 2)):
        for a, b, k in zip(run(first, count, off), whole, NAMES):
            assert np.array_equal(a, b[first:first + count]), (k, first, count, off)
