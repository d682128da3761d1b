"""Sums of squares (f0, the observed residual, the loss of the differentiation form)
of FP32 data far from 1.

At the initial point (X0, Y0 given, no iteration) everything but these sums scales
exactly when G is multiplied by 4^e and the factors by 2^e, so f0 and the loss
must scale by 16^e and the residual by 4^e.  At 4^+-32 a square leaves FP32's range
and at 4^-36 its rounding error does too.  Tolerance 1e-5, the FP32 parity
tolerance of f0.  The lengths take the three slab kernels.  The loss is taken
at rho1 = 0: its rho1 term is summed in FP32 pairs.
"""
import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(7, 40, 112), (7, 40, 9), (7, 70, 12), (3, 20, 520)]
SCALES = [-36, -32, 0, 32]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_09838_gb300 import build
    build.build()


def _instance(shape, seed):
    inst = wl.as_precision(wl.generate(wl.custom(*shape, 2, 0.5, seed=seed + sum(shape), iters=1)), np.float32)
    X0 = np.random.default_rng(seed).standard_normal((shape[0], 2, shape[2])).astype(np.float32)
    return inst, X0


@pytest.mark.parametrize("shape", SHAPES)
def test_objective_scales(shape):
    from paper_2005_09838_gb300 import tc
    inst, X0 = _instance(shape, 8500)
    p = tc.make_params(*shape, 2, 1e-3, 1e-3, 1e-1, precision=tc.TC_FP32)
    got = {}
    for e in SCALES:
        g = wl.to_colmajor(inst["G"] * 4.0 ** e, np.float32)
        y = wl.to_colmajor(inst["Y0"] * 2.0 ** e, np.float32)
        x = wl.to_colmajor(X0 * 2.0 ** e, np.float32)
        with tc.Completion(p, g, wl.to_colmajor(inst["mask"], np.uint8), y, x) as c:
            f0, resid = c.objective()
        got[e] = np.array([f0 / 16.0 ** e, resid / 4.0 ** e])
    for e in SCALES:
        np.testing.assert_allclose(got[e], got[0], rtol=1e-5, err_msg=str(e))


@pytest.mark.parametrize("shape", SHAPES)
def test_static_objective_scales(shape):
    import torch
    from paper_2005_09838_gb300 import tc
    inst, X0 = _instance(shape, 8520)
    p = tc.make_params(*shape, 2, 1e-3, 1e-3, 1e-1, precision=tc.TC_FP32)
    got = {}
    for e in SCALES:
        g, m, y, x = (torch.from_numpy(a).cuda() for a in (
            wl.to_colmajor(inst["G"] * 4.0 ** e, np.float32), wl.to_colmajor(inst["mask"], np.uint8),
            wl.to_colmajor(inst["Y0"] * 2.0 ** e, np.float32), wl.to_colmajor(X0 * 2.0 ** e, np.float32)))
        f0 = tc.complete_static(p, g, m, y, 0, torch.empty_like(g), X0=x,
                                stream=torch.cuda.current_stream().cuda_stream)
        got[e] = f0 / 16.0 ** e
    for e in SCALES:
        assert abs(got[e] - got[0]) <= 1e-5 * got[0], (e, got)


@pytest.mark.parametrize("shape", SHAPES)
def test_gradient_loss_scales(shape):
    import torch
    from paper_2005_09838_gb300 import autograd as ag
    rng = np.random.default_rng(8540 + sum(shape))
    n1, n2, n3 = shape
    G, X, Y = (torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda()
               for s in (shape, (n1, 2, n3), (2, n2, n3)))
    mask = torch.from_numpy(rng.random(shape) < 0.5).cuda()
    G = torch.where(mask, G, torch.zeros_like(G))
    got = {}
    for e in SCALES:
        g = ag.grad_context(G * 4.0 ** e, mask, 2, 0.0)
        xc, yc = ((t * 2.0 ** e).permute(2, 1, 0).contiguous() for t in (X, Y))
        got[e] = g.eval(xc, yc, torch.empty_like(xc), torch.empty_like(yc), on_device=True) / 16.0 ** e
        g.close()
    for e in SCALES:
        assert abs(got[e] - got[0]) <= 1e-5 * got[0], (e, got)


def test_sum_of_squares_of_the_iterate():
    # f0 at a weight mu that leaves nothing else of it: mu / 2 times the sum over the
    # W that tc_result returns.  Its additions in FP64: some 60 per value (threads,
    # warps, blocks, rows), each within 2^-53 of the sum.
    from paper_2005_09838_gb300 import tc
    shape = (5, 288, 100)
    w = wl.custom(*shape, 2, 0.7, seed=8560, iters=1)
    inst = wl.as_precision(wl.generate(w), np.float32)
    mu = 2.0 ** 70
    p = tc.make_params(*shape, 2, mu, 0.0, 0.0, precision=tc.TC_FP32)
    with tc.Completion(p, *(wl.to_colmajor(inst[k], t) for k, t in (
            ("G", np.float32), ("mask", np.uint8), ("Y0", np.float32)))) as c:
        c.iterate(1)
        f0, _ = c.objective()
        W, _, _ = c.result_numpy()
    W = np.asarray(W, dtype=np.float64)
    import math
    exact = 0.5 * mu * math.fsum(float(v) * float(v) for v in W)
    assert abs(f0 - exact) <= 60 * 2.0 ** -53 * exact, (f0, exact)
