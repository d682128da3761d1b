"""FP64 X-step Grams on both sides of rho1 = 1, where their form changes (stencil on one
factor below, sums of products of differences above): W against the FP64 oracle
within the parity tolerance 1e-10."""
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


@pytest.mark.parametrize("rho1", [0.5, 1.0, 1.5, 1e4])
@pytest.mark.parametrize("shape,r", [((1, 24, 5), 1), ((2, 24, 5), 2), ((60, 40, 1), 3), ((33, 30, 6), 5)])
def test_gram_forms(shape, r, rho1):
    from paper_2005_09838_gb300 import api
    inst = wl.generate(wl.custom(*shape, r, 0.6, seed=8600 + sum(shape), iters=3))
    ref = O.tctf2r(inst["G"], inst["mask"], r, 1e-3, rho1, 1e-1, inst["Y0"], iters=3)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], r, 3, 1e-3, rho1, 1e-1, "fp64")
    rel = np.linalg.norm(got["W"] - ref["W"]) / np.linalg.norm(ref["W"])
    assert rel <= 1e-10, rel
