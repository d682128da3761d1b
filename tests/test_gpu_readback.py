"""tc_result into device buffers: no device memory allocated by the call (tc_init
allocates what it needs), and W the same for every way of writing it (whole
tensor through the row buffer, in parts, straight)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_09838_gb300 import build
    build.build()


# small; rows through the buffer (folded transform, FFT length); the plain kernel; a
# tensor of more than the buffer's 128 MiB, in parts with a remainder
@pytest.mark.parametrize("shape", [(16, 48, 7), (200, 100, 30), (150, 60, 112), (40, 60, 520), (1400, 200, 126)])
def test_read_back_allocates_nothing(shape):
    import torch
    from paper_2005_09838_gb300 import tc
    n1, n2, n3 = shape
    gen = torch.Generator(device="cuda").manual_seed(sum(shape))
    G = torch.randn(n1 * n2 * n3, generator=gen, device="cuda")
    ones = torch.ones(G.numel(), dtype=torch.uint8, device="cuda")
    y = torch.randn(2 * n2 * n3, generator=gen, device="cuda")
    W = torch.zeros_like(G)
    p = tc.make_params(*shape, 2, 0.0, 0.0, 0.0, precision=tc.TC_FP32)
    with tc.Completion(p, G, ones, y, on_device=True, stream=torch.cuda.current_stream().cuda_stream) as c:
        free = torch.cuda.mem_get_info()[0]
        c.result(W, on_device=True)
        assert torch.cuda.mem_get_info()[0] == free
    # fully observed: W is G, up to the transform there and back (FP32 parity tolerance)
    assert float((W - G).norm()) <= 1e-5 * float(G.norm())


def test_many_small_fp64_slabs():
    # more than two slabs per SM: the read-back kernels run with half the threads
    import workloads as wl
    from oracle import method as O
    from paper_2005_09838_gb300 import api
    inst = wl.generate(wl.custom(310, 20, 7, 2, 0.5, seed=8700, iters=2))
    ref = O.tctf2r(inst["G"], inst["mask"], 2, 1e-3, 1e-3, 1e-1, inst["Y0"], iters=2)
    got = api.complete(inst["G"], inst["mask"], inst["Y0"], 2, 2, 1e-3, 1e-3, 1e-1, "fp64")
    assert np.linalg.norm(got["W"] - ref["W"]) <= 1e-10 * np.linalg.norm(ref["W"])
    assert abs(got["f0"] - ref["f0"]) <= 1e-10 * abs(ref["f0"])
