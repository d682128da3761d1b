"""FP32 engines on both sides of the rules that choose the fused or the tiled
contractions (n1 = 32 for r > 8, n1 = 80 and 192 for r <= 8), with an FFT length and
without: W against the FP64 oracle within the FP32 parity tolerance 1e-5."""
import numpy as np
import pytest

import workloads as wl
from oracle import method as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_09838_gb300 import build
    build.build()


@pytest.mark.parametrize("n3", [9, 112])
@pytest.mark.parametrize("n1,r", [(31, 12), (32, 12), (31, 20), (32, 20), (79, 8), (80, 8), (191, 6), (192, 6)])
def test_both_sides(n1, r, n3):
    from paper_2005_09838_gb300 import api
    w = wl.custom(n1, 34, n3, r, 0.5, seed=8800 + n1 + n3, iters=2)
    inst = wl.as_precision(wl.generate(w), np.float32)
    ref = O.tctf2r(inst["G"], inst["mask"], r, 1e-3, 1e-3, 1e-1, inst["Y0"], iters=2)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], r, 2, 1e-3, 1e-3, 1e-1, "fp32")
    rel = np.linalg.norm(got["W"] - ref["W"]) / np.linalg.norm(ref["W"])
    assert rel <= 1e-5, rel
