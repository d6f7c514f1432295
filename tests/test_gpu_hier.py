"""The hierarchical Toeplitz-dot-Hankel product and the direct one (needs a GPU) against the
oracle's dense product and against the FFT schedules of the same plan.

Sizes sit at the edges of the tree: one coefficient, a leaf of 32 packed indices and its neighbours,
the boxes of 128, 512 and 2048, odd lengths (the last pair half empty) and batches around the
vector groups of a warp.  Tolerances: the stated ones, max |y - ref| <= tol ||alpha||_1 kappa
(float32 5e-6, float64 1e-12; kappa of tests/conditioning.py), and for the errors against
64 bits the claim of the path itself -- float32 far fields to 2e-8 of the result and float64 to
1e-14, componentwise sums otherwise: at most 64 roundings of sum |A_jk| |alpha_k| in the norm.
"""
import numpy as np
import pytest

import oracle
import workloads
from conditioning import kappa

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "fp32": 5e-6}
U = {"fp64": 2.0 ** -53, "fp32": 2.0 ** -24}
FAR = {"fp64": 1e-14, "fp32": 2.5e-8}


@pytest.fixture(scope="module")
def tdh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07486_gb300 as m
    from paper_1604_07486_gb300 import build
    build.build()
    return m


KINDS = {
    "leg2cheb": (oracle.LEG2CHEB, None),
    "cheb2leg": (oracle.CHEB2LEG, None),
    "ultra_up": (oracle.ULTRA, (0.2, 0.9)),
    "ultra_down": (oracle.ULTRA, (0.9, 0.2)),
    "jacobi": (oracle.JAC, (0.05, 0.3, 0.95, 0.3)),
    "jacobi_row0": (oracle.JAC, (-0.75, -0.5, -0.25, -0.5)),
    "laguerre": (oracle.LAG, (0.3, -0.2)),
}
NAMES = {"leg2cheb": "leg2cheb", "cheb2leg": "cheb2leg", "ultra_up": "ultra2ultra",
         "ultra_down": "ultra2ultra", "jacobi": "jac2jac", "jacobi_row0": "jac2jac",
         "laguerre": "lag2lag"}
SIZES = [1, 2, 63, 64, 65, 128, 129, 191, 257, 1023, 2049, 4095, 4097, 8200]


def _check(tdh, name, n, batch, prec):
    import torch
    okind, params = KINDS[name]
    x = workloads.coefficients(n, batch, decay=0.5, seed=n + batch)
    if prec == "fp32":
        x = x.astype(np.float32).astype(np.float64)
    plan = tdh.Plan(NAMES[name], n, prec=prec, params=params or ())
    xt = torch.tensor(x, dtype=plan.dtype, device="cuda")
    sgn = -1.0 if name == "ultra_up" else 1.0
    for fn, tr in ((plan.execute, False), (plan.adjoint, True)):
        y = fn(xt).double().cpu().numpy()
        ref = oracle.matvec(okind, params, x, transpose=tr)
        l1 = np.abs(x).sum(axis=1)
        scale = kappa(NAMES[name], params) if params and NAMES[name] != "lag2lag" else 1.0
        assert (np.abs(y - ref).max(axis=1) / l1).max() <= TOL[prec] * scale, (name, n, tr)
        # off the diagonal every entry of these kinds has one sign, the diagonal the other or
        # the same: sum |A||x| is at most |A|x|| plus twice the diagonal's part
        size = np.abs(oracle.matvec(okind, params, np.abs(x), transpose=tr))
        diag = oracle.entries(okind, params, n)[np.arange(n), np.arange(n)] if n <= 300 else None
        if diag is not None:
            size = size + 2 * np.abs(diag) * np.abs(x)
            err = np.linalg.norm(y - ref, axis=1)
            assert np.all(err <= (64 * U[prec] + FAR[prec]) * np.linalg.norm(size, axis=1)), \
                (name, n, tr, (err / np.linalg.norm(size, axis=1)).max())


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("name", sorted(KINDS))
def test_matches_oracle(tdh, name, n):
    _check(tdh, name, n, 3, "fp32")
    _check(tdh, name, n, 3, "fp64")


@pytest.mark.parametrize("batch", [1, 2, 5, 12, 17, 33, 70])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_vector_groups(tdh, batch, prec):
    _check(tdh, "cheb2leg", 3001, batch, prec)
    _check(tdh, "jacobi", 1300, batch, prec)


def test_short_batches(tdh):
    """Where the direct product takes two vectors per CTA for want of shared memory, and its
    last sizes before the tree."""
    for name, n, batch in (("cheb2leg", 5900, 3), ("cheb2leg", 5900, 4), ("cheb2leg", 5400, 4),
                           ("jacobi", 4400, 3), ("cheb2leg", 400, 70)):
        _check(tdh, name, n, batch, "fp64")
        _check(tdh, name, n, batch, "fp32")


def test_long_vectors_match_the_fft_schedule(tdh):
    """Several 2048-boxes (the top level's exchange) and the deepest tree, against the FFT schedule
    of the same plan: both within the stated tolerance, so within twice of each other."""
    import torch
    for kind, params, n, batch in (("leg2cheb", (), 131072 + 77, 2), ("cheb2leg", (), 65536, 20),
                                   ("jac2jac", (0.1, 0.3, 0.4, 0.3), 1 << 17, 17)):
        x = torch.tensor(workloads.coefficients(n, batch, decay=0.5, seed=5), device="cuda")
        for prec in ("fp32", "fp64"):
            plan = tdh.Plan(kind, n, prec=prec, params=params)
            xp = x.to(plan.dtype)
            y, g = plan.execute(xp).double(), plan.adjoint(xp).double()
            plan.set_schedule(0)
            yf, gf = plan.execute(xp).double(), plan.adjoint(xp).double()
            l1 = x.abs().sum(dim=1, keepdim=True)
            for a, b in ((y, yf), (g, gf)):
                assert float(((a - b).abs() / l1).max()) <= 2 * TOL[prec], (kind, prec)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_ragged_edges(tdh, prec):
    """Lengths at the tree's edges in one ragged batch, each against the oracle; vectors that
    share a group with longer ones do not see them."""
    lengths = np.array([0, 1, 2, 63, 64, 65, 127, 129, 1000, 4096, 4097, 5000, 3, 0, 64] * 3)
    _ragged(tdh, lengths, 5000, prec)
    # a few short vectors (float64: the FFT schedules), and the same plan with more of them
    _ragged(tdh, np.array([0, 1, 700, 64, 1000]), 1000, prec)
    _ragged(tdh, np.array([1000, 700, 64, 0] * 20), 1000, prec)


def _ragged(tdh, lengths, n_max, prec):
    import torch
    x, offs = workloads.ragged_coefficients(lengths, decay=0.5, seed=9)
    plan = tdh.Plan("cheb2leg", n_max, prec=prec, ragged=True)
    y = plan.execute_ragged(torch.tensor(x, dtype=plan.dtype, device="cuda"),
                            torch.tensor(offs, device="cuda")).double().cpu().numpy()
    for v in range(len(lengths)):
        a, b = int(offs[v]), int(offs[v + 1])
        if b > a:
            ref = oracle.matvec(oracle.CHEB2LEG, None, x[a:b])
            assert np.abs(y[a:b] - ref).max() <= TOL[prec] * np.abs(x[a:b]).sum(), (v, b - a)
    assert plan.status() == set()


@pytest.mark.parametrize("n", [5, 1000, 20001])
def test_bf16x3_plans_run_it_in_float32(tdh, n):
    """Split-bfloat16 plans: the float32 plan's results bit for bit (dense, transpose, ragged)
    until an FFT schedule is set, whose results differ and stay within the stated tolerance."""
    import torch
    a = tdh.Plan("leg2cheb", n, prec="bf16x3", ragged=True)
    b = tdh.Plan("leg2cheb", n, prec="fp32", ragged=True)
    x = torch.tensor(workloads.coefficients(n, 9, decay=0.5, seed=4), dtype=torch.float32,
                     device="cuda")
    offs = torch.arange(10, device="cuda") * n
    y = a.execute(x)
    assert torch.equal(y, b.execute(x)) and torch.equal(a.adjoint(x), b.adjoint(x))
    assert torch.equal(a.execute_ragged(x.flatten(), offs), b.execute_ragged(x.flatten(), offs))
    a.set_schedule(0)
    z = a.execute(x)
    assert n < 64 or not torch.equal(z, y)
    assert float(((z - y).abs().amax(1) / x.abs().sum(1)).max()) <= 5e-6 + TOL["fp32"]


def test_unaligned_rows_and_nonfinite_inputs(tdh):
    """Odd lengths put every other vector at an odd offset; a NaN reaches exactly the outputs
    that depend on it (same parity, lower index) and no other vector."""
    import torch
    n = 3001
    plan = tdh.Plan("leg2cheb", n, prec="fp32")
    x = torch.tensor(workloads.coefficients(n, 9, decay=0.5, seed=2), dtype=torch.float32,
                     device="cuda")
    y = plan.execute(x)
    k = 1500
    z = x.clone()
    z[4, k] = float("nan")
    w = plan.execute(z)
    keep = torch.arange(9, device="cuda") != 4
    assert torch.equal(w[keep], y[keep])
    bad = torch.isnan(w[4]).cpu().numpy()
    assert bad[0:k + 1:2].all() and not bad[1::2].any()
    # a leaf's near field covers its right neighbour: nothing past the NaN's own leaf is touched
    assert not bad[(k // 64 + 1) * 64:].any()
