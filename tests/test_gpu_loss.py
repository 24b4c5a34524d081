"""The 3DGS loss's strips and row batches against the FP64 oracle: widths around one and two strips of 65 pixels,
heights around a segment's rows (11 k - 20), segments whose last batch holds one row, several views in one launch,
images that start between 16-byte boundaries, and the reach of a pixel that is not a number."""
import numpy as np
import pytest

from oracle import train as OT
from tests.gpu_util import rel_err
from tests.test_gpu_train import _cams, _gpu_loss, _images

pytestmark = pytest.mark.gpu

# One view per entry; a tuple of several is one launch.  13 rows are the shortest segment, 24 the next; with many
# pixels the plan takes longer ones, so the last two cases go through other segment lengths.
VIEWS = [((65, 13),), ((64, 12),), ((66, 14),), ((130, 24),), ((131, 25),), ((5, 1),), ((1, 27),), ((10, 35),),
         ((75, 9), (65, 40), (3, 3), (129, 26)), ((1300, 331),), ((2000, 1111),)]


@pytest.mark.parametrize("sizes", VIEWS, ids=lambda s: ",".join("%dx%d" % v for v in s))
def test_loss_strips_match_oracle(sizes):
    xs, ys = _images(sizes, 11), _images(sizes, 12)
    ref = OT.loss_3dgs(xs, ys, lam=0.2)
    loss, grad = _gpu_loss(sizes, xs, ys, 0.2)
    assert abs(loss[0] - ref["loss"]) <= 1e-5 * ref["loss"]
    assert abs(loss[1] - ref["l1"]) <= 1e-5 * ref["l1"]
    assert abs(loss[2] - ref["ssim"]) <= 1e-5
    for g, gr in zip(grad, ref["grad"]):
        assert rel_err(g, gr) <= 1e-4


def test_loss_any_alignment_and_no_stray_write():
    """rgb, target and gradient three different multiples of 4 bytes past a 16-byte boundary: the same numbers as
    aligned buffers give, and nothing written beside the gradient."""
    import torch
    from paper_2410_18931_gb300 import Renderer
    sizes = [(131, 30)]
    xs, ys = _images(sizes, 21), _images(sizes, 22)
    loss0, grad0 = _gpu_loss(sizes, xs, ys, 0.2)
    n = xs[0].size
    bufs = [torch.full((n + 16,), 7.0, device="cuda") for _ in range(3)]
    rgb, tgt, grad = (b[o:o + n] for b, o in zip(bufs, (1, 2, 3)))
    rgb.copy_(torch.from_numpy(xs[0].reshape(-1)))
    tgt.copy_(torch.from_numpy(ys[0].reshape(-1)))
    loss = torch.zeros(3, device="cuda")
    Renderer(_cams(sizes)).wsr_loss_3dgs(rgb, tgt, 0.2, loss, grad)
    torch.cuda.synchronize()
    assert np.array_equal(grad.cpu().numpy(), grad0[0].reshape(-1))
    assert np.allclose(loss.cpu().numpy(), loss0, rtol=1e-6)
    assert (bufs[2][:3] == 7.0).all() and (bufs[2][3 + n:] == 7.0).all()


def test_loss_nan_reaches_its_window_only():
    """A pixel enters the statistics 5 pixels around it and the gradient 10 around it, in its own channel."""
    sizes = [(140, 50)]
    xs, ys = _images(sizes, 31), _images(sizes, 32)
    xs[0][20, 66, 1] = np.nan
    _, grad = _gpu_loss(sizes, xs, ys, 0.2)
    want = np.zeros((50, 140, 3), bool)
    want[10:31, 56:77, 1] = True
    assert np.array_equal(np.isnan(grad[0]), want)
