"""The FFT form (needs a GPU): every kind of Toeplitz-dot-Hankel step on an FFT schedule asked for
(executes take the hierarchical product otherwise), within one cluster and in several passes, dense,
transposed, ragged, with targeted factors and on the tensor cores.

Tolerance: max |y - ref| <= tol ||alpha||_1 kappa as stated (float32 5e-6, split bfloat16 1e-5,
float64 1e-12; kappa of tests/conditioning.py), and for plans with a target that of the target.
"""
import numpy as np
import pytest

import oracle
import workloads
from conditioning import kappa

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 5e-6, "bf16x3": 1e-5}


@pytest.fixture(scope="module")
def tdh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07486_gb300 as m
    from paper_1604_07486_gb300 import build
    build.build()
    return m


def _rows(n, count=96):
    if n <= 6000:
        return np.arange(n)
    return np.unique(np.r_[np.arange(32), n - 1 - np.arange(32),
                           np.random.default_rng(7).integers(0, n, count)])


def _oracle(kind, params, x, rows, transpose):
    if kind == "leg2cheb":
        return oracle.matvec(oracle.LEG2CHEB, None, x, rows=rows, transpose=transpose)
    if kind == "cheb2leg":
        return oracle.matvec(oracle.CHEB2LEG, None, x, rows=rows, transpose=transpose)
    if kind == "ultra2ultra":
        return oracle.matvec(oracle.ULTRA, params, x, rows=rows, transpose=transpose)
    if kind == "jac2jac" and params[1] == params[3]:
        return oracle.matvec(oracle.JAC, params[:3], x, rows=rows, transpose=transpose)
    if transpose:
        return None
    f = {"jac2jac": oracle.jac2jac, "jac2cheb": oracle.jac2cheb, "cheb2jac": oracle.cheb2jac}[kind]
    return f(x, *params, rows=rows)


def _check(tdh, plan, kind, params, x, prec, tol=None, seed=0):
    import torch
    n = x.shape[1]
    rows = _rows(n)
    xt = torch.tensor(x, dtype=plan.dtype, device="cuda")
    xr = xt.double().cpu().numpy()
    scale = kappa(kind, params) if params else 1.0
    l1 = np.abs(xr).sum(axis=1)
    for fn, tr in ((plan.execute, False), (plan.adjoint, True)):
        ref = _oracle(kind, params, xr, rows, tr)
        if ref is None:
            continue
        y = fn(xt).double().cpu().numpy()[:, rows]
        err = (np.abs(y - ref).max(axis=1) / l1).max()
        assert err <= (tol or TOL[prec]) * scale, (kind, params, n, prec, tr, err)


KINDS = [("ultra2ultra", (0.2, 0.9)), ("ultra2ultra", (0.9, 0.2)), ("ultra2ultra", (0.3, 2.6)),
         ("jac2jac", (0.05, 0.3, 0.95, 0.3)), ("jac2jac", (-0.75, -0.5, -0.25, -0.5)),
         ("jac2jac", (0.2, 0.3, 0.2, 0.9)), ("jac2jac", (0.1, -0.3, 0.6, 0.2)),
         ("jac2cheb", (0.3, 0.2)), ("cheb2jac", (0.3, 0.2))]


@pytest.mark.parametrize("kind,params", KINDS)
@pytest.mark.parametrize("prec,n", [("fp32", 63), ("fp32", 5001), ("fp64", 1000), ("fp64", 5001),
                                    ("bf16x3", 3000)])
def test_kinds(tdh, kind, params, prec, n):
    plan = tdh.Plan(kind, n, prec=prec, params=params)
    plan.set_schedule(0)
    _check(tdh, plan, kind, params, workloads.coefficients(n, 3, decay=1.0, seed=n), prec)


@pytest.mark.parametrize("kind,params,n,prec", [
    ("leg2cheb", (), 1 << 20, "fp32"), ("leg2cheb", (), 1 << 23, "fp32"),
    ("cheb2leg", (), 70001, "fp64"), ("leg2cheb", (), 1 << 20, "fp64"),
    ("jac2jac", (0.1, 0.3, 0.4, 0.3), 1 << 20, "fp32"), ("leg2cheb", (), 200000, "bf16x3")])
def test_multipass(tdh, kind, params, n, prec):
    """FFTs beyond one cluster: up to 512 slices, rows all over the vector."""
    plan = tdh.Plan(kind, n, prec=prec, params=params)
    plan.set_schedule(0)
    assert plan.schedules()[0]["C"] > 8
    _check(tdh, plan, kind, params, workloads.coefficients(n, 1, decay=1.0, seed=3), prec)


@pytest.mark.parametrize("n_max", [700, 2439, 5000])
@pytest.mark.parametrize("kind", ["leg2cheb", "cheb2leg"])
@pytest.mark.parametrize("prec", ["fp32", "fp64", "bf16x3"])
def test_ragged_lengths_that_are_no_powers_of_two(tdh, prec, kind, n_max):
    """The length classes share one set of factors, as long as the longest class reads (rows past
    their end made such plans' results NaN)."""
    import torch
    lengths = np.array([n_max, 1, n_max - 1, 64, n_max // 2 + 1, 0, 257, 2])
    x, offs = workloads.ragged_coefficients(np.minimum(lengths, n_max), decay=1.0, seed=n_max)
    plan = tdh.Plan(kind, n_max, prec=prec, ragged=True)
    plan.set_schedule(0)
    y = plan.execute_ragged(torch.tensor(x, dtype=plan.dtype, device="cuda"),
                            torch.tensor(offs, device="cuda")).double().cpu().numpy()
    for v in range(len(lengths)):
        a, b = int(offs[v]), int(offs[v + 1])
        if b > a:
            ref = _oracle(kind, (), x[None, a:b], np.arange(b - a), False)[0]
            assert np.abs(y[a:b] - ref).max() <= TOL[prec] * np.abs(x[a:b]).sum(), (v, b - a)
    assert plan.status() == set()


@pytest.mark.parametrize("kind,params,n,target", [
    ("leg2cheb", (), 8192, 2.5e-6), ("cheb2leg", (), 8192, 1e-6), ("leg2cheb", (), 1000, 1e-3),
    ("ultra2ultra", (0.3, 0.8), 4096, 1e-9), ("jac2jac", (0.1, 0.2, 0.6, 0.2), 4096, 1e-9)])
def test_targeted_factors(tdh, kind, params, n, target):
    """The truncated factors of a targeted plan meet their target for every input, and are what the
    FFT form multiplies with: its error on unit vectors is between 1e-4 of the target and it."""
    import torch
    plan = tdh.Plan(kind, n, prec="fp64", tol=target, params=params, target=True)
    plan.set_schedule(0)
    ks = np.unique(np.r_[0:8, np.random.default_rng(5).integers(0, n, 40), n - 4:n])
    x = np.zeros((len(ks), n))
    x[np.arange(len(ks)), ks] = 1.0
    ref = _oracle(kind, params, x, None, False)
    y = plan.execute(torch.tensor(x, device="cuda")).cpu().numpy()
    err = np.abs(y - ref).max()
    assert 1e-4 * target <= err <= target + 1e-12, (err, plan.K)


@pytest.mark.parametrize("n,ragged", [(65536, False), (4096, True)])
def test_split_bfloat16_after_autotune(tdh, n, ragged):
    """Autotune keeps the hierarchical product where it is the faster form; the tensor-core FFTs run
    when their schedule is set, before it or after."""
    import torch
    plan = tdh.Plan("leg2cheb", n, prec="bf16x3", ragged=ragged)
    plan.autotune(4)
    x = workloads.coefficients(n, 2, decay=0.5, seed=12)
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    tree = plan.execute(xt)
    plan.set_schedule(0)
    assert not torch.equal(plan.execute(xt), tree)
    _check(tdh, plan, "leg2cheb", (), x, "bf16x3")
    if ragged:
        offs = torch.tensor([0, 1000, n], device="cuda")
        y = plan.execute_ragged(xt[0].contiguous(), offs).double().cpu().numpy()
        for a, b in ((0, 1000), (1000, n)):
            ref = oracle.matvec(oracle.LEG2CHEB, None, x[0, a:b])
            assert np.abs(y[a:b] - ref).max() <= TOL["bf16x3"] * np.abs(x[0, a:b]).sum()
    assert plan.status() == set()
