"""Adam's bias corrections at any step number: powers by squaring against 64-bit ones."""
import numpy as np
import pytest

from tests.test_gpu_train import _adam_call, _adam_setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("done", [0, 1, 2, 6, 7, 8, 62, 998, 12344, 999999, 2**31 - 2])
def test_bias_corrections(done):
    """c1 and c2 to a float's rounding (2^-24, one more bit for the two roundings that may fall on either side)."""
    import torch
    groups, _, _, grads, dev = _adam_setup(5)
    dev["state"][0] = done
    _adam_call(groups, dev, grads[0])
    torch.cuda.synchronize()
    st = dev["state"].cpu().numpy()
    t = done + 1
    c = st[1:3].view(np.float32).astype(np.float64)
    want = np.array([1.0 / (1.0 - 0.9 ** t), 1.0 / np.sqrt(1.0 - 0.999 ** t)])
    assert st[0] == t and st[3] == 0
    assert np.all(np.abs(c - want) <= 2.0 ** -23 * want), (c, want)
