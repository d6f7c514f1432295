"""The hierarchical product's tree (needs a GPU): sizes at the edges of its boxes in batches large
enough that the direct product does not take them, forward and transposed, vector groups of the
wide far-field kernel, chunks of vectors, and inputs that only the far field sees.

Bound, as in the direct product's test: off the diagonal every entry of these kinds has one sign,
so sum |A_jk| |alpha_k| is at most |A| |alpha| plus twice the diagonal's part; a result is within 64
roundings of it and the far field's claim (float32 2.5e-8, float64 1e-14), in the norm.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

U = {"fp64": 2.0 ** -53, "fp32": 2.0 ** -24}
FAR = {"fp64": 1e-14, "fp32": 2.5e-8}
KINDS = {"leg2cheb": ("leg2cheb", oracle.LEG2CHEB, None),
         "cheb2leg": ("cheb2leg", oracle.CHEB2LEG, None),
         "ultra": ("ultra2ultra", oracle.ULTRA, (0.9, 0.2)),
         "jacobi": ("jac2jac", oracle.JAC, (0.05, 0.3, 0.95, 0.3))}


@pytest.fixture(scope="module")
def tdh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07486_gb300 as m
    from paper_1604_07486_gb300 import build
    build.build()
    return m


def _check_vectors(name, x, y, picks, prec, tr, rows=None):
    """Rows `rows` (all if None) of the vectors `picks` against the oracle."""
    _, okind, params = KINDS[name]
    n = x.shape[1]
    r = np.arange(n) if rows is None else rows
    ref = oracle.matvec(okind, params, x[picks], rows=r, transpose=tr)
    size = np.abs(oracle.matvec(okind, params, np.abs(x[picks]), rows=r, transpose=tr))
    t, h, d1, d2 = oracle.split(okind, params, n)
    diag = np.abs(d1 * t[0] * h[::2] * d2)
    if name == "cheb2leg":
        diag[0] = 1.0
    size = size + 2 * diag[r] * np.abs(x[picks][:, r])
    err = np.linalg.norm(y[np.ix_(picks, r)] - ref, axis=1)
    assert np.all(err <= (64 * U[prec] + FAR[prec]) * np.linalg.norm(size, axis=1)), \
        (name, n, prec, tr, (err / np.linalg.norm(size, axis=1)).max())


# packed lengths just above one, two and four boxes of 32, 128, 512 and 2048, and odd ones between
# (two channels: n = 2 m)
@pytest.mark.parametrize("n", [130, 150, 257, 300, 514, 516, 1030, 1537, 2049, 2060, 4100, 8195])
@pytest.mark.parametrize("name", sorted(KINDS))
def test_tree_at_box_edges(tdh, name, n):
    import torch
    kind, _, params = KINDS[name]
    for prec in ("fp32", "fp64"):
        # past the direct product's limit: lane operations, as it counts them, above 1e8
        channels = 1 if kind == "jac2jac" else 2
        m = (n + channels - 1) // channels
        batch = max(12, int(1e8 / (channels * m / 4 * (5 * (m / 2 + 16) + 640))) + 1)
        x = workloads.coefficients(n, batch, decay=0.5, seed=n)
        if prec == "fp32":
            x = x.astype(np.float32).astype(np.float64)
        plan = tdh.Plan(kind, n, prec=prec, params=params or ())
        xt = torch.tensor(x, dtype=plan.dtype, device="cuda")
        picks = np.unique([0, 1, batch // 2, batch - 1])
        for fn, tr in ((plan.execute, False), (plan.adjoint, True)):
            y = fn(xt).double().cpu().numpy()
            _check_vectors(name, x, y, picks, prec, tr)


@pytest.mark.parametrize("batch", [1, 3000])
def test_leading_entry_is_exact(tdh, batch):
    """C_0 = 1 for every parameter, A_00 = 1: the float32 tables hold s_0 and h_0 as powers of two and
    what was taken out of them in D1, whose first entry is then one too, so the constant is
    converted exactly (direct product and tree, forward and transposed)."""
    import torch
    n = 150
    for params in ((0.05, 1.04), (0.488, 1.297), (0.9, 0.2), (0.3, 0.8), (100.2, 100.7), (0.7, 0.25)):
        plan = tdh.Plan("ultra2ultra", n, prec="fp32", params=params)
        x = torch.zeros(batch, n, device="cuda")
        x[:, 0] = 1.0
        for fn in (plan.execute, plan.adjoint):
            assert (fn(x)[:, 0] == 1.0).all(), (params, float(fn(x)[0, 0]) - 1)


@pytest.mark.parametrize("kind", ["leg2cheb", "cheb2leg", "jacobi"])
def test_wide_far_field_and_top_exchange(tdh, kind):
    """Float32 against float64 of the same input, in the norm of the result: inputs that live only in
    the last box of 2048 of long vectors (forward; the first for the transpose), rows two boxes and
    more away, so that every value comes through the exchange of the 2048-boxes -- by itself
    (>= 32 boxes) and within the far kernel -- and through each of its smaller levels; batches of one
    vector group and of the 16-vector far CTAs.  Bound: 64 roundings of |A| |alpha| and the
    interpolation's 2.5e-8; the entries here have one sign, so |A| |alpha| is A |alpha|."""
    import torch
    name, _, params = KINDS[kind]
    channels = 1 if kind == "jacobi" else 2
    for n, batch in ((channels * 2048 * 40 + 77, 3), (channels * 2048 * 5 + 1, 40),
                     (channels * 2048 * 2 + 9, 200)):
        lo = tdh.Plan(name, n, prec="fp32", params=params or ())
        hi = tdh.Plan(name, n, prec="fp64", params=params or ())
        g = torch.Generator("cuda").manual_seed(n)
        far = torch.randn(batch, n, device="cuda", generator=g)
        for size in (2048, 512, 128, 32):
            w = channels * size
            if 3 * w >= n:  # no rows that far away
                continue
            for tr in (False, True):
                x = torch.zeros_like(far)
                keep = slice(n - w, n) if not tr else slice(0, w)
                x[:, keep] = far[:, keep]
                fn, ref = (lo.adjoint, hi.adjoint) if tr else (lo.execute, hi.execute)
                rows = slice(0, n - 3 * w) if not tr else slice(3 * w, n)
                y, r = fn(x).double()[:, rows], ref(x.double())[:, rows]
                a = ref(x.double().abs())[:, rows]
                err = (y - r).norm(dim=1) / a.norm(dim=1)
                assert float(err.max()) <= 64 * U["fp32"] + FAR["fp32"], (n, size, tr, float(err.max()))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_chunks_of_vectors(tdh, prec):
    """More vectors than one pass of the tree takes (about 1 GB of moments): those on both sides of
    the cut, dense and ragged, against the oracle, and the same vector everywhere the same."""
    import torch
    n, batch = 300, 330000 if prec == "fp64" else 1300000
    x = workloads.coefficients(n, 50, decay=0.5, seed=1)
    if prec == "fp32":
        x = x.astype(np.float32).astype(np.float64)
    plan = tdh.Plan("cheb2leg", n, prec=prec, ragged=True)
    base = torch.tensor(x, dtype=plan.dtype, device="cuda")
    big = base.repeat((batch + 49) // 50, 1)[:batch]
    offs = torch.arange(batch + 1, device="cuda") * n
    for tr, y in ((False, plan.execute(big)), (True, plan.adjoint(big)),
                  (False, plan.execute_ragged(big.flatten(), offs).reshape(batch, n))):
        first = y[:50].double().cpu().numpy()
        _check_vectors("cheb2leg", x, first, np.arange(50), prec, tr)
        assert all(torch.equal(y[k:k + 50], y[:50]) for k in range(0, batch - 50, 50 * 800))
        assert torch.equal(y[batch - 50:], y[:50])
    assert plan.status() == set()
