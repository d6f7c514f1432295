"""Back-substitution as weighted prefix sums (needs a GPU): the inverse sparse factors of
Sec. 5.2 / 5.3 Case 1 against the double-double oracle, at the edges of their tiles.

The inverse of an unflipped factor has positive entries, so |A| |alpha| is the oracle applied to
|alpha| (for a flipped one, to (-1)^k |alpha_k|, up to sign), and every rounding is bounded
componentwise by it, u = 2^-24 (2^-53 in float64):
  one factor, in its own precision: two rounded table entries, two products and at most 29
  additions on any path through the thread, warp, block and tile sums: 34 u, and in float64 some
  16 u more for each table's Gamma ratio;
  float32 chains (pairs of floats): one rounding at the end, u, doubled for the rest.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

# float32 tiles hold 4096 coefficients, float64 and the unaligned paths fewer per access
SIZES = [1, 2, 3, 5, 63, 1024, 2047, 4096, 4097, 8190]
SINGLE = [("ultra2ultra", (1.25, 0.25)), ("jac2jac", (1.5, 0.25, 0.5, 0.25)),
          ("jac2jac", (0.3, 1.6, 0.3, 0.6))]
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


def _matrix(kind, params, n):
    """A [n][n] from the oracle (its dense product on unit vectors)."""
    if kind == "ultra2ultra":
        return oracle.matvec(oracle.ULTRA, params, np.eye(n)).T
    return np.stack([oracle.jac2jac(v, *params) for v in np.eye(n)]).T


def _check(tdh, kind, params, n, prec, c):
    import torch
    x = workloads.coefficients(n, 3, decay=0.5, seed=n)
    u = 2.0 ** (-24 if prec == "fp32" else -53)
    if prec == "fp32":
        x = x.astype(np.float32).astype(np.float64)
    plan = tdh.Plan(kind, n, prec=prec, params=params)
    xt = torch.tensor(x, dtype=plan.dtype, device="cuda")
    if n <= 2100:
        A = _matrix(kind, params, n)
        cases = [(plan.execute, x @ A.T, np.abs(x) @ np.abs(A).T),
                 (plan.adjoint, x @ A, np.abs(x) @ np.abs(A))]
    elif kind == "ultra2ultra":  # positive entries: the oracle on |x| bounds the terms
        m = lambda v, t: oracle.matvec(oracle.ULTRA, params, v, transpose=t)
        cases = [(plan.execute, m(x, False), m(np.abs(x), False)),
                 (plan.adjoint, m(x, True), m(np.abs(x), True))]
    else:
        s = (-1.0) ** np.arange(n) if params[1] != params[3] and params[0] == params[2] else 1.0
        m = lambda v: np.stack([oracle.jac2jac(r, *params) for r in v])
        cases = [(plan.execute, m(x), np.abs(m(s * np.abs(x))))]
    for fn, ref, size in cases:
        y = fn(xt).double().cpu().numpy()
        # the reference itself is rounded to (and, formed from the matrix, summed in) float64
        bound = c * u * size + 4 * n ** 0.5 * 2.0 ** -53 * size
        assert np.all(np.abs(y - ref) <= bound), (np.abs(y - ref) / (u * size + 1e-300)).max()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind,params", SINGLE, ids=["ultra", "jacobi", "jacobi-reflected"])
@pytest.mark.parametrize("prec,c", [("fp32", 34), ("fp64", 66)])
def test_single_factor(tdh, kind, params, n, prec, c):
    _check(tdh, kind, params, n, prec, c)


@pytest.mark.parametrize("n", [1, 3, 1024, 2047, 2048])
@pytest.mark.parametrize("kind,params", CHAIN, ids=["ultra-two", "jacobi-both-parameters"])
def test_float32_chain_rounds_once(tdh, kind, params, n):
    _check(tdh, kind, params, n, "fp32", 2)


@pytest.mark.parametrize("a", [4.0, 7.0, 30.0])
def test_large_parameters_match_the_oracle(tdh, a):
    """Parameters on both sides of the prefix sums' range (ln W spans about (a + 1) ln n; the
    affine scan takes over above 40): the stated tolerances, in proportion to the output."""
    import torch
    n, params = 700, (a + 0.5, 0.25, a - 0.5, 0.25)
    x = workloads.coefficients(n, 2, decay=1.0, seed=3)
    ref = np.stack([oracle.jac2jac(v, *params) for v in x])
    for prec, tol in (("fp32", 5e-6), ("fp64", 1e-12)):
        plan = tdh.Plan("jac2jac", n, prec=prec, params=params)
        y = plan.execute(torch.tensor(x, dtype=plan.dtype, device="cuda")).double().cpu().numpy()
        l1 = np.abs(x).sum(axis=1, keepdims=True)
        kappa = max(1.0, float((np.abs(ref).max(axis=1, keepdims=True) / l1).max()))
        assert (np.abs(y - ref) / l1).max() <= tol * kappa
