"""Launch counts and their limits: what the Python side counts by is what the header states, and what the launchers
use; a step's count follows the binning that its own number of Gaussians takes."""
import os
import re
from types import SimpleNamespace

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _header():
    text = open(os.path.join(ROOT, "include", "wsr.h")).read()
    return {k: int(v) for k, v in re.findall(r"^#define (WSR_[A-Z_]+)\s+(\d+)\b", text, flags=re.M)}


def test_limits_are_the_headers():
    import __graft_entry__
    __graft_entry__._build_module().build()
    from paper_2410_18931_gb300 import _abi as A
    h = _header()
    for name in ("WSR_SCAN_ONE_BLOCK_TILES", "WSR_BIN_ONE_TILES", "WSR_BIN_ONE_GAUSSIANS", "WSR_ORDER_MIN_TILES",
                 "WSR_ORDER_ONE_BLOCK_TILES"):
        assert getattr(A, name) == h[name], name
    code = "".join(open(os.path.join(ROOT, "paper_2410_18931_gb300", "csrc", f)).read() for f in ("api.cu", "bin.cu"))
    assert "WSR_ORDER_MIN_TILES" in code and "WSR_ORDER_ONE_BLOCK_TILES" in code


def test_a_steps_count_follows_its_binning():
    import __graft_entry__
    __graft_entry__._build_module().build()
    from paper_2410_18931_gb300 import GraphStep, Renderer
    for n, tiles, bins in ((8192, 1024, 1), (8193, 1024, 3), (4096, 4096, 1), (4097, 4096, 3), (10, 4097, 3)):
        r = Renderer.__new__(Renderer)
        r.num_tiles, r.n_cams, r.deterministic, r.bin_kernels, r.order_kernels = tiles, 1, False, 3, 1
        step = GraphStep.__new__(GraphStep)
        step.r, step.g = r, SimpleNamespace(n=n)
        assert r.bin_launches(n) == bins and step.kernels_per_step == 5 + bins + 1
        assert r.bin_kernels == 3
