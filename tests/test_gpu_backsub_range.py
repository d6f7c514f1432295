"""Back-substitution over the whole range of its type, and over many tiles (needs a GPU).

Multiplying the input by a power of two multiplies every intermediate value by it, exactly, as long
as none of them overflows or becomes subnormal.  So the result of a scaled input is the scaled
result, bit for bit: up to the largest representable result (sums that overflow before it does
would show), and down to inputs of 2^-80 in float32.
"""
import math

import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

SINGLE = [("ultra2ultra", (1.25, 0.25)), ("ultra2ultra", (1.01, 0.01)),
          ("jac2jac", (1.5, 0.25, 0.5, 0.25)), ("jac2jac", (0.3, 1.6, 0.3, 0.6)),
          ("jac2jac", (3.5, 0.25, 2.5, 0.25)), ("jac2jac", (0.2, -0.5, -0.8, -0.5))]
CHAIN = [("ultra2ultra", (2.25, 0.25)), ("jac2jac", (2.5, 1.25, 0.5, 0.25))]


@pytest.fixture(scope="module")
def tdh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07486_gb300 as m
    from paper_1604_07486_gb300 import build
    build.build()
    return m


def _input(n, dtype):
    import torch
    x = np.round(workloads.coefficients(n, 2, decay=0.5, seed=n) * 2.0 ** 12) * 2.0 ** -12
    return torch.tensor(x, dtype=dtype, device="cuda")


@pytest.mark.parametrize("kind,params", SINGLE + CHAIN)
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_no_overflow_before_the_result(tdh, kind, params, prec):
    import torch
    top = 126 if prec == "fp32" else 1022
    for n in (3, 700, 4097, 16384):
        plan = tdh.Plan(kind, n, prec=prec, params=params)
        x = _input(n, plan.dtype)
        for fn in (plan.execute, plan.adjoint):
            y = fn(x)
            big = max(float(y.abs().max()), float(x.abs().max()))
            s = 2.0 ** (top - math.ceil(math.log2(big)))
            assert torch.equal(fn(x * s), y * s), (n, s)


@pytest.mark.parametrize("kind,params", SINGLE)
def test_no_loss_at_small_inputs(tdh, kind, params):
    import torch
    for n in (700, 16384):
        plan = tdh.Plan(kind, n, prec="fp32", params=params)
        x = _input(n, plan.dtype)
        for fn in (plan.execute, plan.adjoint):
            assert torch.equal(fn(x * 2.0 ** -68), fn(x) * 2.0 ** -68), n


@pytest.mark.parametrize("n,prec,params", [((1 << 24) + 4100, "fp32", (1.25, 0.25)),
                                           ((1 << 24) + 1, "fp32", (2.25, 0.25)),
                                           ((1 << 23) + 2049, "fp64", (1.25, 0.25))])
def test_many_tiles(tdh, n, prec, params):
    """From 4097 tiles on their sums are scanned once per vector.  C^(l+1) -> C^(l) is
    x_j = (l + j)/l sum_{i >= j, i = j mod 2} c_i: componentwise error at most 34 roundings (as for
    fewer tiles) and one for every addition of the scan, 17 + 8 + 17 more; chains of two
    factors (float32: pairs of floats) at most twice one rounding plus the reference's own."""
    import torch
    u = 2.0 ** (-24 if prec == "fp32" else -53)
    plan = tdh.Plan("ultra2ultra", n, prec=prec, params=params)
    x = torch.randn(1, n, dtype=plan.dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(1))

    def steps(v, transpose):
        lams = [params[0] - 1 - i for i in range(round(params[0] - params[1]))]
        for lam in (lams[::-1] if transpose else lams):
            w = (np.arange(n) + np.longdouble(lam)) / np.longdouble(lam)
            v = v * w if transpose else v
            out = np.empty_like(v)
            for e in range(2):
                p = v[:, e::2]
                out[:, e::2] = np.cumsum(p, 1) if transpose else np.cumsum(p[:, ::-1], 1)[:, ::-1]
            v = out if transpose else out * w
        return v

    xd = x.double().cpu().numpy().astype(np.longdouble)
    c = 2 if params[0] - params[1] > 1 else 34 + 42
    for fn, tr in ((plan.execute, False), (plan.adjoint, True)):
        y = fn(x).double().cpu().numpy()
        err = np.abs(y - steps(xd, tr))
        assert np.all(err <= c * u * steps(np.abs(xd), tr)), float((err / (u * steps(np.abs(xd), tr))).max())
