"""The work that a user of this library has it do, as timed cases.

Every case goes through the public entry points of ``paper_2005_09838_gb300``
(``tc.Completion``, ``tc.Batch``, ``tc.complete_static``, ``autograd``):

* ``iterate``   a context that a program keeps (``tc_init`` done): a number of
                iterations, then the iterate W, X, Y read back on the device,
                as a loop does that looks at its progress;
* ``complete``  a whole completion of a new tensor: ``tc_init`` from device
                buffers, the iterations, the objective, W, ``tc_free``;
* ``static``    the same for a small tensor through the allocation-free call;
* ``batch``     many tensors of different sizes advanced together, then every W;
* ``grad``      one training step's loss and both gradients, through autograd.

Sizes are those of the repository's own workloads (16x48x7, 144x288x168,
529x96x112, 529x288x168 and the batched form's n1 64-1024, n2 96-288, n3
28-168, r 4-32, 10-60% observed) and of the one-week traffic traces of Sec. 5
(121 OD pairs x 144 ten-minute slots x 7 days).  The data are seeded traffic
tensors drawn like ``workloads.generate`` (low tubal rank, lognormal scale per
OD pair, daily profile, 1% noise), made on the GPU.
"""
import math

import numpy as np
import torch

from paper_2005_09838_gb300 import autograd as ag
from paper_2005_09838_gb300 import tc

MU, RHO1, RHO2 = 1e-3, 1e-3, 1e-1
PRECISION = {"fp64": tc.TC_FP64, "fp32": tc.TC_FP32, "tf32": tc.TC_TF32, "bf16": tc.TC_BF16}
MOST_ENTRIES = 529 * 288 * 168  # the largest listed tensor
MOST_FP64 = 1 << 20             # entries of a drawn FP64 tensor


def case(name, kind, n1, n2, n3, r, precision, observed, iters, eps=0.0, members=1):
    return {"name": name, "kind": kind, "n1": n1, "n2": n2, "n3": n3, "r": r, "precision": precision,
            "observed": observed, "iters": iters, "eps": eps, "members": members}


def listed():
    return [
        # a small tensor completed inside a latency-critical program that may not
        # allocate: 16 OD pairs x 48 half-hours x 7 days in FP64
        case("static_16x48x7_fp64", "static", 16, 48, 7, 2, "fp64", 0.5, 50),
        # the same tensor in a context that a program keeps and looks at often: the
        # smallest call, launches and latency
        case("iterate_16x48x7_fp64", "iterate", 16, 48, 7, 2, "fp64", 0.5, 10),
        # one week of a traffic trace (121 OD pairs, ten-minute slots) in FP64 with the
        # stopping test of the algorithm at 1e-6, as the method is run in Sec. 5
        case("complete_121x144x7_fp64_eps", "complete", 121, 144, 7, 4, "fp64", 0.4, 50, eps=1e-6),
        # the plain FP32 method on 168 days of five-minute slots: a whole completion
        case("complete_144x288x168_fp32", "complete", 144, 288, 168, 8, "fp32", 0.2, 100),
        # the same tensor in a kept context
        case("iterate_144x288x168_fp32", "iterate", 144, 288, 168, 8, "fp32", 0.4, 10),
        # large rank, 112 days of fifteen-minute slots: plain FP32, and the precision
        # form with its contractions on the tensor cores
        case("iterate_529x96x112_fp32", "iterate", 529, 96, 112, 32, "fp32", 0.3, 5),
        case("iterate_529x96x112_tf32", "iterate", 529, 96, 112, 32, "tf32", 0.3, 5),
        # tensors of no special length, as other networks and periods give them: a tube
        # length with small factors at a small rank, a prime one at a middle rank, and
        # the BF16 form at a ragged one
        case("iterate_925x153x92_fp32", "iterate", 925, 153, 92, 8, "fp32", 0.35, 5),
        case("iterate_224x233x109_fp32", "iterate", 224, 233, 109, 13, "fp32", 0.25, 5),
        case("iterate_435x205x34_bf16", "iterate", 435, 205, 34, 28, "bf16", 0.45, 5),
        # many tensors of uneven sizes completed together (sizes drawn from the case's
        # own numbers over the ranges of the batched form)
        case("batch_8", "batch", 1024, 288, 168, 32, "tf32", 0.3, 5, members=8),
        # block gradient descent on the factors: loss and both gradients
        case("grad_529x288x168_fp32", "grad", 529, 288, 168, 16, "fp32", 0.2, 1),
    ]


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["iterate", "iterate", "iterate", "complete", "static", "batch", "grad"])
    observed = round(rng.uniform(0.1, 0.6), 3)
    if kind == "static":
        n1, n2, n3 = log_int(rng, 8, 64), log_int(rng, 24, 96), rng.choice([7, 8, 9, 12, 14])
        c = case("", kind, n1, n2, n3, rng.randint(1, 4), rng.choice(["fp64", "fp32"]), max(observed, 0.3),
                 rng.randint(10, 50))
    elif kind == "batch":
        c = case("", kind, log_int(rng, 256, 1024), 288, 168, 32, "tf32", observed, rng.randint(2, 5),
                 members=rng.randint(2, 8))
    elif kind in ("iterate", "complete") and rng.random() < 0.25:
        n1, n2, n3 = log_int(rng, 16, 256), rng.randint(48, 150), log_int(rng, 7, 31)
        n1 = max(16, min(n1, MOST_FP64 // (n2 * n3)))
        c = case("", kind, n1, n2, n3, rng.randint(2, 8), "fp64", max(observed, 0.3), rng.randint(1, 10),
                 eps=1e-6 if kind == "complete" else 0.0)
    else:
        n3 = rng.choice([112, 168]) if rng.random() < 0.25 else rng.randint(28, 168)
        n1, n2, r = log_int(rng, 64, 1024), rng.randint(96, 288), log_int(rng, 4, 32)
        n1 = max(64, min(n1, MOST_ENTRIES // (n2 * n3)))
        precision = rng.choice(["fp32", "tf32", "bf16"]) if kind != "grad" and r > 16 else "fp32"
        iters = {"iterate": rng.randint(1, 5), "complete": rng.randint(10, 30), "grad": 1}[kind]
        iters = min(iters, 100 * 144 * 288 * 168 // (n1 * n2 * n3))  # no more than the listed completion
        c = case("", kind, n1, n2, n3, r, precision, observed, iters)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def real_type(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def shapes(case):
    """(n1, n2, n3, r, precision) of every tensor of a case.  The members of a
    batch are spread over the ranges of the batched form below the case's sizes;
    as in use, those with r > 16 take the case's tensor-core precision."""
    if case["kind"] != "batch":
        return [(case["n1"], case["n2"], case["n3"], case["r"], case["precision"])]
    rng = np.random.default_rng(1000 * case["n1"] + 10 * case["iters"] + case["members"])
    out = []
    for _ in range(case["members"]):
        n1, n2 = int(rng.integers(64, case["n1"] + 1)), int(rng.integers(96, case["n2"] + 1))
        n3, r = int(rng.integers(28, case["n3"] + 1)), int(rng.integers(4, case["r"] + 1))
        out.append((n1, n2, n3, r, case["precision"] if r > 16 else "fp32"))
    return out


def tensor(n1, n2, n3, r, dtype, observed, seed):
    """One seeded traffic tensor (indices [i1, i2, i3]): G (0 off the mask), mask, Y0, X0."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float32)

    A, B = normal(n1, r, n3).abs(), normal(r, n2, n3).abs()
    At = torch.fft.rfft(A, dim=2).permute(2, 0, 1)
    Bt = torch.fft.rfft(B, dim=2).permute(2, 0, 1)
    T = torch.fft.irfft((At @ Bt).permute(1, 2, 0), n=n3, dim=2)
    scale = torch.exp(0.5 * normal(n1))
    profile = 1.0 + 0.5 * torch.sin(2.0 * math.pi * torch.arange(n2, device="cuda", dtype=torch.float32) / n2)
    T = T * scale[:, None, None] * profile[None, :, None]
    M = T + 0.01 * T.square().mean().sqrt() * normal(n1, n2, n3)
    mask = torch.rand(n1, n2, n3, generator=gen, device="cuda", dtype=torch.float32) < observed
    G = torch.where(mask, M, torch.zeros_like(M)).to(dtype)
    return G, mask, normal(r, n2, n3).to(dtype), normal(n1, r, n3).to(dtype)


def flat(t):
    """The C ABI's element order (first index fastest)."""
    return t.permute(2, 1, 0).contiguous().reshape(-1)


def params(case, n1, n2, n3, r, precision):
    return tc.make_params(n1, n2, n3, r, MU, RHO1, RHO2, PRECISION[precision], eps=case["eps"])


def prepare(case, seed):
    dtype, kind = real_type(case), case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "grad":
        G, mask, Y, X = tensor(case["n1"], case["n2"], case["n3"], case["r"], dtype, case["observed"], seed)
        return {"case": case, "g": ag.grad_context(G, mask, case["r"], RHO1, dtype=dtype),
                "X": X.requires_grad_(True), "Y": Y.requires_grad_(True)}
    state = {"case": case, "stream": stream, "contexts": [], "inputs": [], "out": []}
    for q, (n1, n2, n3, r, precision) in enumerate(shapes(case)):
        G, mask, Y0, _ = tensor(n1, n2, n3, r, dtype, case["observed"], seed + 7919 * q)
        g, m, y = flat(G), flat(mask.to(torch.uint8)), flat(Y0)
        p = params(case, n1, n2, n3, r, precision)
        torch.cuda.current_stream().synchronize()
        if kind in ("iterate", "batch"):
            state["contexts"].append(tc.Completion(p, g, m, y, on_device=True, stream=stream))
        else:
            state["inputs"].append((p, g, m, y))
        W = torch.empty(n1 * n2 * n3, dtype=dtype, device="cuda")
        X = torch.empty(n1 * r * n3, dtype=dtype, device="cuda") if kind == "iterate" else None
        Y = torch.empty(r * n2 * n3, dtype=dtype, device="cuda") if kind == "iterate" else None
        state["out"].append((W, X, Y))
    if kind == "batch":
        state["batch"] = tc.Batch(state["contexts"], stream=stream)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "grad":
        X, Y = state["X"], state["Y"]
        X.grad = Y.grad = None
        loss = ag.factor_loss(X, Y, state["g"])
        loss.backward()
        return {"loss": loss.detach(), "dX": X.grad, "dY": Y.grad}
    if kind == "iterate":
        c, (W, X, Y) = state["contexts"][0], state["out"][0]
        c.iterate(case["iters"], count=False)
        c.result(W, X, Y, on_device=True)
        return {"W": W, "X": X, "Y": Y}
    if kind == "batch":
        state["batch"].iterate(case["iters"])
        for c, (W, _, _) in zip(state["contexts"], state["out"]):
            c.result(W, on_device=True)
        return [W for W, _, _ in state["out"]]
    (p, g, m, y), (W, _, _) = state["inputs"][0], state["out"][0]
    if kind == "static":
        f0 = tc.complete_static(p, g, m, y, case["iters"], W, stream=state["stream"])
        return {"W": W, "f0": f0}
    with tc.Completion(p, g, m, y, on_device=True, stream=state["stream"]) as c:
        c.iterate(case["iters"], count=case["eps"] > 0)
        f0, resid = c.objective()
        c.result(W, on_device=True)
        out = {"W": W, "f0": f0, "resid_obs": resid}
        if case["eps"] > 0:
            out["changes"] = list(c.convergence()[0])
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    s = 8 if case["precision"] == "fp64" else 4
    total_bytes = total_flops = 0.0
    for n1, n2, n3, r, _ in shapes(case):
        N, S = n1 * n2 * n3, n3 // 2 + 1
        transform = 2.5 * N * math.log2(max(n3, 2))
        contraction = 8.0 * r * n1 * n2 * S
        factors = s * r * (n1 + n2) * n3
        if case["kind"] == "grad":
            total_bytes += s * N + N / 8 + 2 * factors
            total_flops += 3 * contraction + 2 * transform
            continue
        # one iteration: the observed values and the mask once, the residual's half
        # spectrum written once and read by both factor updates
        total_bytes += case["iters"] * (s * N + N / 8 + 6.0 * s * n1 * n2 * S)
        total_flops += case["iters"] * (3 * contraction + 2 * transform + 4.0 * N)
        total_bytes += s * N + (factors if case["kind"] == "iterate" else 0)       # what is read back
        if case["kind"] in ("complete", "static"):
            total_bytes += (s + 1.0) * N + s * r * n2 * n3                          # the inputs
    return {"bytes": total_bytes, "flops": total_flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def stencil(X):
    """H^T H along dim 1 of [S, n1, r]."""
    d = X[:, 1:] - X[:, :-1]
    out = torch.zeros_like(X)
    out[:, 1:] += d
    out[:, :-1] -= d
    return out


def pinv(A, rtol):
    lam, V = torch.linalg.eigh(0.5 * (A + A.mH))
    keep = lam > rtol * lam[:, -1:].clamp_min(0)
    inv = torch.where(keep, 1.0 / torch.where(keep, lam, torch.ones_like(lam)), torch.zeros_like(lam))
    return (V * inv[:, None, :].to(V.dtype)) @ V.mH


def w_step(Z, G, mask):
    """The masked tridiagonal rows of (1 + mu) I + rho2 K^T K, identity on the mask."""
    n2 = Z.shape[1]
    miss = (~mask).to(torch.float64)
    cs, ds = [], []
    c = d = None
    for j in range(n2):
        deg = (j > 0) + (j + 1 < n2)
        m = miss[:, j]
        diag = 1.0 + m * (MU + RHO2 * deg)
        rhs = torch.where(mask[:, j], G[:, j], Z[:, j])
        if c is None:
            den, num = diag, rhs
        else:
            den, num = diag - (RHO2 * m) * c, rhs + (RHO2 * m) * d
        c, d = RHO2 * m / den, num / den
        cs.append(c)
        ds.append(d)
    W = torch.empty_like(Z)
    W[:, n2 - 1] = w = ds[-1]
    for j in range(n2 - 2, -1, -1):
        w = ds[j] + cs[j] * w
        W[:, j] = w
    return W


def spectrum(A):
    At = torch.fft.rfft(A, dim=2).permute(2, 0, 1).contiguous()
    return real_slices(At, A.shape[2])


def real_slices(At, n3):
    At[0].imag.zero_()
    if n3 % 2 == 0:
        At[-1].imag.zero_()
    return At


def spatial(At, n3):
    return torch.fft.irfft(At.permute(1, 2, 0), n=n3, dim=2)


def completion(G, mask, Y0, iters):
    n1, n2, n3 = G.shape
    r = Y0.shape[0]
    rtol = r * 2.0 ** -52
    W = G.clone()
    Wt, Yt = spectrum(W), spectrum(Y0)
    Xt = torch.zeros(Yt.shape[0], n1, r, dtype=Yt.dtype, device=G.device)
    H = torch.eye(n1, dtype=torch.float64, device=G.device)
    H = H + RHO1 * stencil(H[None])[0]
    Hinv = torch.linalg.inv(H).to(Yt.dtype)
    changes = None
    for _ in range(iters):
        Xold, Yold, Wold = Xt, Yt, W
        A = Yt @ Yt.mH
        grad = Xt @ A - Wt @ Yt.mH + RHO1 * (stencil(Xt) @ A)
        Xt = real_slices(Xt - Hinv @ (grad @ pinv(A, rtol)), n3)
        E = Xt.mH @ Xt
        gram = E + RHO1 * (Xt.mH @ stencil(Xt))
        grad = gram @ Yt - Xt.mH @ Wt
        Yt = real_slices(Yt - pinv(gram, rtol) @ grad, n3)
        W = w_step(spatial(Xt @ Yt, n3), G, mask)
        Wt = spectrum(W)
        changes = (Xt - Xold, Yt - Yold, W - Wold)
    return W, Xt, Yt, [changes[0].abs().max(), changes[1].abs().max(), changes[2].norm()]


def objective(W, Xt, Yt, G, mask):
    Z = spatial(Xt @ Yt, W.shape[2])
    f0 = 0.5 * (Z - W).square().sum() + 0.5 * MU * W.square().sum()
    f0 = f0 + 0.5 * RHO2 * (W[:, 1:] - W[:, :-1]).square().sum() + 0.5 * RHO1 * (Z[1:] - Z[:-1]).square().sum()
    return f0, (Z - G)[mask].norm()


def exact(case, seed):
    out = []
    for q, (n1, n2, n3, r, _) in enumerate(shapes(case)):
        G, mask, Y0, X0 = tensor(n1, n2, n3, r, real_type(case), case["observed"], seed + 7919 * q)
        G, Y0, X0 = G.double(), Y0.double(), X0.double()
        if case["kind"] == "grad":
            Xt, Yt = spectrum(X0), spectrum(Y0)
            Z = spatial(Xt @ Yt, n3)
            E = torch.where(mask, Z - G, torch.zeros_like(Z))
            d = Z[1:] - Z[:-1]
            loss = 0.5 * E.square().sum() + 0.5 * RHO1 * d.square().sum()
            E[1:] += RHO1 * d
            E[:-1] -= RHO1 * d
            Et = spectrum(E)
            return {"loss": loss, "dX": spatial(Et @ Yt.mH, n3), "dY": spatial(Xt.mH @ Et, n3)}
        W, Xt, Yt, changes = completion(G, mask, Y0, case["iters"])
        if case["kind"] == "batch":
            out.append(flat(W))
            continue
        got = {"W": flat(W)}
        if case["kind"] == "iterate":
            got["X"], got["Y"] = flat(spatial(Xt, n3)), flat(spatial(Yt, n3))
        else:
            f0, resid = objective(W, Xt, Yt, G, mask)
            got["f0"] = float(f0)
            if case["kind"] == "complete":
                got["resid_obs"] = float(resid)
                if case["eps"] > 0:
                    got["changes"] = [float(v) for v in changes]
        return got
    return out
