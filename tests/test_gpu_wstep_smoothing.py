"""W-step where long runs of missing entries and strong smoothing meet.

A row without an observed entry, and rows with 2% observed, at weights up to
rho2 = 1e8, where the coefficients of the sweeps are within 1e-4 of 1.  W
against the FP64 oracle within the FP32 parity tolerance 1e-5.  The sums are
positive and every coefficient carries a few roundings, so the W-step itself
stays within some 100 units of 2^-24 = 6e-6 (n2 = 100).
"""
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


@pytest.mark.parametrize("rho2", [1e3, 1e5, 1e6, 1e8])
@pytest.mark.parametrize("n3", [13, 14])  # odd and even folding
def test_missing_rows(n3, rho2):
    from paper_2005_09838_gb300 import api
    w = wl.custom(6, 100, n3, 2, 0.5, seed=8300 + n3, iters=2)
    inst = wl.generate(w)
    rng = np.random.default_rng(8301)
    inst["mask"][0] = False
    inst["mask"][1] = rng.random(inst["mask"][1].shape) < 0.02
    inst["G"] = np.where(inst["mask"], inst["M"], 0.0)
    inst = wl.as_precision(inst, np.float32)
    ref = O.tctf2r(inst["G"], inst["mask"], 2, 1e-3, 1e-3, rho2, inst["Y0"], iters=2)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], 2, 2, 1e-3, 1e-3, rho2, "fp32")
    for i in (0, 1, slice(None)):
        rel = np.linalg.norm(got["W"][i] - ref["W"][i]) / np.linalg.norm(ref["W"][i])
        assert rel <= 1e-5, (i, rel)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 1e-5)])
@pytest.mark.parametrize("rho2", [0.1, 3.0])
@pytest.mark.parametrize("n2", [128, 129, 175, 200])
def test_runs_around_segment_edges(n2, rho2, precision, tol):
    # runs of missing entries from every offset within two segments, of lengths
    # around those from which the segments of a run are taken whole, and in a third
    # of the slabs a row without data
    from paper_2005_09838_gb300 import api
    w = wl.custom(48, n2, 9, 2, 0.5, seed=8320 + n2, iters=2)
    inst = wl.generate(w)
    lengths = (15, 16, 17, 31, 32, 33, 47, 63, 64, 65, 80, 96, n2)
    for i in range(48):
        for l in range(9):
            n = n2 if l == 4 and i % 3 == 0 else lengths[(9 * i + l) % len(lengths)]
            a = i if i < 40 and n < n2 else max(0, n2 - n)  # (the last slabs: runs that end with the row)
            inst["mask"][i, a:a + n, l] = False
    inst["G"] = np.where(inst["mask"], inst["M"], 0.0)
    if precision == "fp32":
        inst = wl.as_precision(inst, np.float32)
    ref = O.tctf2r(inst["G"], inst["mask"], 2, 1e-3, 1e-3, rho2, inst["Y0"], iters=2)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], 2, 2, 1e-3, 1e-3, rho2, precision)
    rel = np.linalg.norm(got["W"] - ref["W"]) / np.linalg.norm(ref["W"])
    assert rel <= tol, rel
