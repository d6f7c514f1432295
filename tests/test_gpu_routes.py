"""Which form a call takes (hierarchical product, direct product, FFT schedules, sums or affine
scans), and what it needs for that (needs a GPU): a plan that stays usable when a call fails
half-way, scratch that is bounded, results that do not depend on how a call was cut up.

Tolerances: the stated ones (float32 5e-6, float64 1e-12 of ||alpha||_1) unless a test says
otherwise.
"""
import numpy as np
import pytest

import oracle
import workloads

pytestmark = pytest.mark.gpu

NOMEM = -3
TOL = {"fp64": 1e-12, "fp32": 5e-6, "bf16x3": 1e-5}


@pytest.fixture(scope="module")
def tdh():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1604_07486_gb300 as m
    from paper_1604_07486_gb300 import build
    build.build()
    yield m
    m.inject_alloc_failure(0)


@pytest.mark.parametrize("n,prec", [(4096, "fp32"), (700, "fp32"), (9000, "fp64")])
def test_autotune_that_fails_leaves_the_plan_usable(tdh, n, prec):
    """Every allocation of autotune in turn (a spread of them) fails: the plan goes on giving the
    results it gave before, bit for bit, ragged and dense; a whole autotune's choice stays within
    the tolerance for every length class."""
    import torch
    lengths = np.array([n, 1, 100, 0, 257, n // 2, n // 3, 64])
    x, offs = workloads.ragged_coefficients(lengths, decay=1.0, seed=5)
    ot = torch.tensor(offs, device="cuda")
    made, failed = None, 0
    for k in [0] + list(range(1, 30)):
        plan = tdh.Plan("leg2cheb", n, prec=prec, ragged=True)
        xt = torch.tensor(x, dtype=plan.dtype, device="cuda")
        dense = xt[:n].reshape(1, n).clone()
        before = plan.execute_ragged(xt, ot), plan.execute(dense), plan.adjoint(dense)
        if k == 0:
            a0 = tdh.alloc_stats()[0]
            plan.autotune(6)
            made = tdh.alloc_stats()[0] - a0
            y = plan.execute_ragged(xt, ot).double().cpu().numpy()
            for v in range(len(lengths)):
                a, b = int(offs[v]), int(offs[v + 1])
                if b > a:
                    ref = oracle.matvec(oracle.LEG2CHEB, None, x[a:b])
                    assert np.abs(y[a:b] - ref).max() <= TOL[prec] * np.abs(x[a:b]).sum()
        else:
            at = 1 + (k - 1) * int(0.85 * made) // 28  # (a choice of schedule costs a few)
            tdh.inject_alloc_failure(at)
            try:
                plan.autotune(6)
                raised = False
            except tdh.TdhError as e:
                assert e.code == NOMEM, at
                raised = True
            tdh.inject_alloc_failure(0)
            failed += raised
            after = plan.execute_ragged(xt, ot), plan.execute(dense), plan.adjoint(dense)
            if raised:
                assert all(torch.equal(a, b) for a, b in zip(before, after)), at
        assert plan.status() == set()
        plan.close()
    assert failed >= 20


@pytest.mark.parametrize("n", [1, 64, 128, 129, 256, 257, 512, 513, 3000])
@pytest.mark.parametrize("kind", ["leg2cheb", "cheb2leg"])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_small_ragged_calls(tdh, prec, kind, n):
    """Ragged calls on both sides of the one-launch sort's limit (4096 vectors) agree with
    the oracle and take no more launches than they need."""
    import torch
    okind = oracle.LEG2CHEB if kind == "leg2cheb" else oracle.CHEB2LEG
    plan = tdh.Plan(kind, n, prec=prec, ragged=True)
    for batch in (1, 9, 4096, 4097):
        lengths = np.random.default_rng(batch).integers(0, n + 1, batch)
        lengths[0] = n
        x, offs = workloads.ragged_coefficients(lengths, decay=0.5, seed=n)
        xt, ot = torch.tensor(x, dtype=plan.dtype, device="cuda"), torch.tensor(offs, device="cuda")
        c0 = tdh.launch_count()
        y = plan.execute_ragged(xt, ot).double().cpu().numpy()
        launches = tdh.launch_count() - c0
        far = 3 if n > 128 else 1  # moments, far and near field, or the near field alone
        assert launches == (1 if batch <= 4096 else 3) + far, (batch, launches)
        for v in np.r_[0:min(batch, 40), batch - 1]:
            a, b = int(offs[v]), int(offs[v + 1])
            if b > a:
                ref = oracle.matvec(okind, None, x[a:b])
                assert np.abs(y[a:b] - ref).max() <= TOL[prec] * np.abs(x[a:b]).sum()
    assert plan.status() == set()


def test_small_ragged_calls_report_bad_input(tdh):
    """The one-launch sort records what the three launches do: vectors out of range are left
    unwritten (LENGTH), overlapping input and output convert nothing (ALIAS)."""
    import torch
    n = 64
    plan = tdh.Plan("leg2cheb", n, prec="fp32", ragged=True)
    offs = torch.tensor([0, 64, 200, 190, 254], device="cuda")  # too long; decreasing
    x = torch.randn(300, device="cuda")
    y = torch.full_like(x, -7.0)
    plan.execute_ragged(x, offs, out=y)
    assert plan.status() == {"LENGTH"}
    assert (y[64:190] == -7).all() and (y[:64] != -7).all() and (y[190:254] != -7).all()
    buf = torch.randn(400, device="cuda")
    keep = buf.clone()
    plan.execute_ragged(buf[:300], torch.tensor([0, 64, 128], device="cuda"), out=buf[32:332])
    assert plan.status() == {"ALIAS"} and torch.equal(buf, keep)


def test_laguerre_route_and_accuracy(tdh):
    """Laguerre changes below one: one FFT pair where that is the faster or the more exact form
    (float32 up to 4096 coefficients, float64), the tree beyond.  Float64 FFT errors are at most
    64 roundings of the result in the norm (an FFT pair of 2^15 points rounds about 2 log2 L u);
    the interpolation's are 2e-14 and would not pass."""
    import torch
    for n, prec, launches in ((4096, "fp32", 1), (4097, "fp32", 3), (4096, "bf16x3", 3)):
        plan = tdh.Plan("lag2lag", n, prec=prec, params=(0.3, -0.2))
        x = torch.randn(64, n, dtype=plan.dtype, device="cuda")
        c0 = tdh.launch_count()
        plan.execute(x)
        assert tdh.launch_count() - c0 == launches, (n, prec)
    n = 9001
    rows = np.unique(np.r_[0:64, np.random.default_rng(0).integers(0, n, 300), n - 64:n])
    x = np.random.default_rng(3).standard_normal((2, n))
    for params in ((0.3, -0.2), (100.5, 100.1), (0.5, 0.25)):
        plan = tdh.Plan("lag2lag", n, prec="fp64", params=params)
        for fn, tr in ((plan.execute, False), (plan.adjoint, True)):
            y = fn(torch.tensor(x, device="cuda")).cpu().numpy()[:, rows]
            ref = oracle.matvec(oracle.LAG, params, x, rows=rows, transpose=tr)
            assert np.linalg.norm(y - ref) <= 64 * 2.0 ** -53 * np.linalg.norm(ref), (params, tr)


def test_chain_scratch_is_bounded(tdh):
    """Float32 chains take at most about 1 GB of scratch however large the batch (the pairs of floats
    between two inverse factors of 512 x 2^20 would take 4 GB), and cut batches give what whole
    ones do: every vector's sums are its own, bit for bit."""
    import torch
    n, batch = 1 << 20, 512
    plan = tdh.Plan("ultra2ultra", n, prec="fp32", params=(2.25, 0.25))
    x = torch.randn(batch, n, device="cuda")
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    for fn in (plan.execute, plan.adjoint):
        fn(x, out=y)
        torch.cuda.synchronize()
        assert free0 - torch.cuda.mem_get_info()[0] <= 3 << 29
        for v in (0, 127, 128, 300, batch - 1):
            assert torch.equal(fn(x[v:v + 1]), y[v:v + 1]), v


@pytest.mark.parametrize("kind,params", [("jac2jac", (0.1, -0.3, 0.6, 0.2)),
                                         ("jac2jac", (2.5, 1.25, -0.3, -0.4)),
                                         ("leg2cheb", ())])
def test_executes_get_by_with_less_scratch(tdh, kind, params):
    """A scratch allocation that fails is tried again with fewer vectors at a time: chains (before:
    in place) and the tree both still convert the batch."""
    import torch
    n, batch = 5000, 3000
    plan = tdh.Plan(kind, n, prec="fp32", params=params)
    x = torch.randn(batch, n, device="cuda") / torch.arange(1, n + 1, device="cuda")
    ref = plan.execute(x), plan.adjoint(x)
    for k in (1, 2, 3):
        for fn, r in zip((plan.execute, plan.adjoint), ref):
            tdh.inject_alloc_failure(k)
            y = fn(x)
            tdh.inject_alloc_failure(0)
            scale = r.abs().amax(1) + x.abs().sum(1)
            assert float(((y - r).abs().amax(1) / scale).max()) <= 2 * TOL["fp32"], k
    torch.cuda.synchronize()
    assert tdh.alloc_stats()[2] == 0


def test_plans_keep_only_their_rank(tdh):
    """A plan whose factorisation fills its first 64 terms starts again with room for kmax; it keeps
    the terms it took, and at most 64 MB of spare rows."""
    import torch
    n = 20000
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    plan = tdh.Plan("jac2jac", n, prec="fp64", params=(10.2, 3.0, 10.9, 3.0), kmax=1000)
    torch.cuda.synchronize()
    held = free0 - torch.cuda.mem_get_info()[0]
    assert plan.K > 64
    assert held <= 8 * n * plan.K + (64 << 20) + (32 << 20), (held, plan.K)


@pytest.mark.parametrize("kind,params", [("leg2cheb", ()), ("cheb2leg", ()),
                                         ("jac2jac", (0.1, -0.3, 0.6, 0.2))])
def test_factorisation_without_all_blocks_resident(tdh, kind, params):
    """The factorisation's one launch gives up when its blocks cannot meet (here: a bounded wait that
    the test hook makes run out) and goes launch by launch: same pivots, factors and ranks."""
    import torch
    n = 5000
    sym = tdh.symbols("leg2cheb", n)[1]
    u0, p0 = tdh.pchol(sym, n, 0, 1e-13)
    want = [tdh.Plan(kind, n, prec=prec, params=params).K for prec in ("fp32", "fp64")]
    few = tdh.Plan(kind, n, prec="fp64", params=params, kmax=3).K
    tdh.inject_tc_stall(True)
    try:
        u1, p1 = tdh.pchol(sym, n, 0, 1e-13)
        plans = [tdh.Plan(kind, n, prec=prec, params=params) for prec in ("fp32", "fp64")]
        assert tdh.Plan(kind, n, prec="fp64", params=params, kmax=3).K == few == 3
    finally:
        tdh.inject_tc_stall(False)
    assert torch.equal(p0, p1) and torch.equal(u0, u1)
    assert [p.K for p in plans] == want
    x = torch.tensor(workloads.coefficients(n, 2, decay=1.0, seed=2), device="cuda")
    plans[1].set_schedule(0)  # (the FFT form multiplies with the factors)
    ref = tdh.Plan(kind, n, prec="fp64", params=params)
    ref.set_schedule(0)
    assert torch.equal(plans[1].execute(x), ref.execute(x))


def test_large_kmax_asks_for_no_more_rows_than_steps(tdh):
    """The factorisation takes at most 1024 steps, so a larger kmax asks for 1024 rows (here it would
    be 320 GB)."""
    n = 200000
    plan = tdh.Plan("jac2jac", n, prec="fp64", params=(10.2, 3.0, 10.9, 3.0), kmax=10 ** 9)
    assert 64 < plan.K <= 1024
