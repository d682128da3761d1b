"""Slab kernel of the folded mode-3 transform, at the sizes where it can go wrong.

W, f0 and the factors against the FP64 oracle after a few iterations: tube
lengths around the folding's special rows (n3 = 1, 2, 3, 4, 2M with M even and
odd), tile and 64-tube remainders, mask words that a run of missing entries
enters, leaves or fills (sparse masks, whole rows missing or observed), slabs
with one and with several stages, without stages, and past shared memory.
Tolerances are those of the parity tests: 1e-10 (FP64) and 1e-5 (FP32) on W.
"""
import numpy as np
import pytest

import workloads as wl
from oracle import method as O

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_09838_gb300 import build
    build.build()


def _check(shape, r, obs, precision, iters=3, rows=None, weights=(1e-3, 1e-3, 1e-1)):
    from paper_2005_09838_gb300 import api
    w = wl.custom(*shape, r, obs, seed=8100 + sum(shape), iters=iters)
    inst = wl.generate(w)
    if rows is not None:  # whole rows (i1, :, i3) observed or missing
        inst["mask"][0, :, :] = rows
        inst["G"] = np.where(inst["mask"], inst["M"], 0.0)
    if precision == "fp32":
        inst = wl.as_precision(inst, np.float32)
    ref = O.tctf2r(inst["G"], inst["mask"], r, *weights, inst["Y0"], iters=iters)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], r, iters, *weights, precision)
    rel = np.linalg.norm(got["W"] - ref["W"]) / np.linalg.norm(ref["W"])
    assert rel <= TOL[precision], (shape, precision, rel)
    assert abs(got["f0"] - ref["f0"]) <= TOL[precision] * abs(ref["f0"])
    assert abs(got["resid_obs"] - ref["resid_obs"]) <= 10 * TOL[precision] * max(ref["resid_obs"], 1.0)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("n3", [1, 2, 3, 4, 5, 6, 10, 15, 16, 17, 30, 33])
def test_tube_lengths(n3, precision):
    _check((7, 33 + 32 * (n3 % 3), n3), 3, 0.4, precision)


@pytest.mark.parametrize("n2", [1, 2, 31, 32, 63, 64, 65, 96, 128, 161])
def test_tubes_and_mask_words(n2):
    _check((5, n2, 9), min(2, n2), 0.3, "fp32")
    _check((5, n2, 12), min(2, n2), 0.02 if n2 > 40 else 0.3, "fp64")


@pytest.mark.parametrize("rows", [True, False])
@pytest.mark.parametrize("weights", [(1e-3, 1e-3, 1e-1), (0.0, 0.0, 0.0), (0.5, 0.1, 30.0)])
def test_whole_rows_and_weights(rows, weights):
    _check((6, 100, 14), 2, 0.5, "fp64", rows=rows, weights=weights)
    _check((6, 100, 13), 2, 0.5, "fp32", rows=rows, weights=weights)


@pytest.mark.parametrize("shape,precision", [
    ((2, 200, 120), "fp32"),   # a spectrum of several stages
    ((2, 288, 165), "fp32"),   # no room for a stage
    ((2, 300, 190), "fp32"),   # slab past shared memory
    ((2, 150, 60), "fp64"),    # FP64 in stages
    ((2, 160, 100), "fp64"),   # FP64 past shared memory
])
def test_large_slabs(shape, precision):
    _check(shape, 2, 0.3, precision, iters=2)


@pytest.mark.parametrize("shape,r", [
    ((70, 65, 112), 12),    # eight strided partials of D, two per CTA; odd n2
    ((200, 34, 112), 8),    # four per CTA; rows past a multiple of 8
    ((66, 97, 112), 20),    # one per CTA, r padded
    ((65, 64, 10), 16),     # contiguous ranges, compensated real slices
    ((200, 129, 9), 7),     # tiled Q, four groups sharing a sum
])
def test_tiled_contractions(shape, r):
    _check(shape, r, 0.4, "fp32")
