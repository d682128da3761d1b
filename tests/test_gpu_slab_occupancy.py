"""The plain slab kernel (tube lengths past the folded transform) with registers for
one, two and three CTAs per SM, by the number of slabs: W against the FP64 oracle
within the FP32 parity tolerance 1e-5."""
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


@pytest.mark.parametrize("n1", [8, 160, 310])
def test_slabs_per_sm(n1):
    from paper_2005_09838_gb300 import api
    w = wl.custom(n1, 20, 520, 2, 0.4, seed=8400 + n1, iters=2)
    inst = wl.as_precision(wl.generate(w), np.float32)
    ref = O.tctf2r(inst["G"], inst["mask"], 2, 1e-3, 1e-3, 1e-1, inst["Y0"], iters=2)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], 2, 2, 1e-3, 1e-3, 1e-1, "fp32")
    rel = np.linalg.norm(got["W"] - ref["W"]) / np.linalg.norm(ref["W"])
    assert rel <= 1e-5, rel
