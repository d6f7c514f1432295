"""The conversions a user of the library runs, as measurable cases.

``listed()`` names the workloads; ``draw()`` gives more of the same ranges.  ``prepare()``
holds what a program keeps (the plan, the coefficients on the GPU), ``run()`` is one pass
through the public API, ``exact()`` the same result in 64-bit arithmetic from the closed forms
of the conversion matrices (Townsend, Webb & Olver, arXiv:1604.07486, Eqs. (2), (11), (13) and
Sec. 5.3) with numpy and torch alone.

Inputs follow the paper's experiments: alpha_k = z_k (k+1)^(-decay), z_k iid standard normal.
"""
import math

import numpy as np
import torch

import paper_1604_07486_gb300 as tdh
from paper_1604_07486_gb300.autograd import convert

DTYPE = {"fp32": torch.float32, "bf16x3": torch.float32, "fp64": torch.float64}
PARAMS = ("p0", "p1", "p2", "p3")


def listed():
    return [
        # the smallest call: one short vector in double precision (a function approximated by
        # about a thousand terms, converted once); launches and latency
        dict(name="leg2cheb_n1024_b1_fp64", op="execute", kind="leg2cheb", n=1024, batch=1,
             prec="fp64", decay=1.0),
        # one long vector: a single function resolved to 2^16 terms
        dict(name="leg2cheb_n65536_b1_fp32", op="execute", kind="leg2cheb", n=65536, batch=1,
             prec="fp32", decay=0.5),
        # the paper's headline conversion over a full batch (the default benchmark, one way)
        dict(name="leg2cheb_n65536_b256_fp32", op="execute", kind="leg2cheb", n=65536, batch=256,
             prec="fp32", decay=0.5),
        # the way back, at a length and a batch that are no powers of two
        dict(name="cheb2leg_n40001_b100_fp32", op="execute", kind="cheb2leg", n=40001, batch=100,
             prec="fp32", decay=1.0),
        # a batch in double precision: spectral solvers that need full accuracy
        dict(name="leg2cheb_n65536_b32_fp64", op="execute", kind="leg2cheb", n=65536, batch=32,
             prec="fp64", decay=0.5),
        # the split-bfloat16 option
        dict(name="leg2cheb_n65536_b64_bf16x3", op="execute", kind="leg2cheb", n=65536, batch=64,
             prec="bf16x3", decay=0.5),
        # thousands of functions of uneven degree in one call (degrees log-uniform, 64..65535)
        dict(name="ragged_4096_fp32", op="ragged", kind="leg2cheb", n=65536, batch=4096,
             nmin=64, prec="fp32", decay=1.0),
        # the conversion as a layer of a trained model: forward, loss, backward
        dict(name="train_n8192_b1024_fp32", op="train", kind="leg2cheb", n=8192, batch=1024,
             prec="fp32", decay=1.0),
        # very long vectors, no parity structure: two Toeplitz-dot-Hankel steps
        dict(name="jac2jac_n2p20_b16_fp32", op="execute", kind="jac2jac", n=1 << 20, batch=16,
             prec="fp32", decay=1.0, p0=0.1, p1=-0.3, p2=0.0, p3=0.0, tol=1e-13),
        # raising the ultraspherical parameter by one (differentiation and multiplication in
        # ultraspherical spectral methods), and lowering it again by back-substitution
        dict(name="ultra_up_n2p20_b16_fp32", op="execute", kind="ultra2ultra", n=1 << 20,
             batch=16, prec="fp32", decay=1.0, p0=0.25, p1=1.25, tol=1e-13),
        dict(name="ultra_down_n2p20_b16_fp32", op="execute", kind="ultra2ultra", n=1 << 20,
             batch=16, prec="fp32", decay=1.0, p0=1.25, p1=0.25, tol=1e-13),
        # a one-off conversion: build the plan, convert one vector, release the plan
        dict(name="one_off_leg2cheb_n65536_fp32", op="one_off", kind="leg2cheb", n=65536,
             batch=1, prec="fp32", decay=0.5),
    ]


def _log_int(rng, lo, hi):
    """An integer log-uniform in [lo, hi]; now and then a power of two."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.25:
        v = 1 << int(round(math.log2(v)))
    return max(lo, min(hi, v))


def draw(rng):
    op = rng.choice(["execute"] * 6 + ["adjoint"] * 2 + ["ragged", "ragged", "train", "one_off"])
    prec = "fp32"
    if op in ("execute", "adjoint"):
        prec = rng.choice(["fp32", "fp32", "fp64", "bf16x3"])
        kind = rng.choice(["leg2cheb", "leg2cheb", "cheb2leg", "ultra2ultra", "jac2jac"])
    elif op == "ragged":
        kind = rng.choice(["leg2cheb", "cheb2leg"])
    else:
        kind = "leg2cheb"
    top = 1 << 16
    if kind in ("ultra2ultra", "jac2jac") and prec == "fp32":
        top = 1 << 20
    case = dict(op=op, kind=kind, n=_log_int(rng, 64, top), prec=prec,
                decay=rng.choice([0.5, 1.0, 1.5]) if kind == "leg2cheb" else 1.0)
    # the whole batch: at most 2^24 coefficients (2^20 in double precision)
    room = (1 << 20 if prec == "fp64" else 1 << 24) // case["n"]
    case["batch"] = 1 if op == "one_off" else _log_int(rng, 1, max(1, min(room, 4096)))
    if op == "ragged":
        case["nmin"] = _log_int(rng, 1, case["n"])
        case["batch"] = max(2, case["batch"])
    if kind == "ultra2ultra":
        p0 = round(rng.uniform(0.2, 0.8), 3)
        step = rng.choice([1.0, -1.0, 2.0, 0.0])  # whole steps up and down, or a fraction
        case["p0"] = p0 + max(0.0, -step)
        case["p1"] = p0 + max(0.0, step) if step else p0 + round(rng.uniform(0.1, 0.9), 3)
    if kind == "jac2jac":
        case["p0"], case["p1"] = (round(rng.uniform(-0.4, 0.0), 3) for _ in range(2))
        case["p2"] = case["p0"] + round(rng.uniform(0.1, 0.9), 3)
        case["p3"] = case["p1"] + round(rng.uniform(0.1, 0.9), 3)
    return case


def _lengths(case):
    """Vector lengths: degrees log-uniform between the shortest and the longest."""
    rng = np.random.default_rng(0)
    u = rng.uniform(math.log(case["nmin"]), math.log(case["n"]), size=case["batch"])
    lengths = np.clip(np.floor(np.exp(u)).astype(np.int64), case["nmin"], case["n"])
    lengths[rng.integers(case["batch"])] = case["n"]
    return lengths


def _normal(count, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)
    return torch.randn(count, generator=g, device="cuda", dtype=torch.float64)


def _inputs(case, seed):
    """(values in the plan's type, host offsets or None)."""
    dt = DTYPE[case["prec"]]
    if case["op"] == "ragged":
        lengths = _lengths(case)
        offsets = np.zeros(lengths.size + 1, dtype=np.int64)
        np.cumsum(lengths, out=offsets[1:])
        k = torch.arange(int(offsets[-1]), device="cuda")
        k -= torch.repeat_interleave(torch.from_numpy(offsets[:-1]).cuda(),
                                     torch.from_numpy(lengths).cuda())
        z = _normal(int(offsets[-1]), seed)
        return (z * (k + 1.0).double() ** -case["decay"]).to(dt), offsets
    k = torch.arange(case["n"], device="cuda", dtype=torch.float64)
    z = _normal(case["batch"] * case["n"], seed).reshape(case["batch"], case["n"])
    return (z * (k + 1.0) ** -case["decay"]).to(dt), None


def _params(case):
    return tuple(case[p] for p in PARAMS if p in case)


def _plan(case):
    return tdh.Plan(case["kind"], case["n"], prec=case["prec"], tol=case.get("tol"),
                    params=_params(case), ragged=case["op"] == "ragged")


def _target(case, seed):
    """What a training step fits the converted coefficients to (squared error)."""
    return _inputs(case, seed + 1000003)[0]


def prepare(case, seed):
    x, offsets = _inputs(case, seed)
    state = dict(case=case, x=x)
    if case["op"] != "one_off":
        state["plan"] = _plan(case)
    if case["op"] == "ragged":
        state["offsets"] = torch.from_numpy(offsets).cuda()
    if case["op"] == "train":
        state["target"] = _target(case, seed)
    return state


def run(state):
    op, x = state["case"]["op"], state["x"]
    if op == "execute":
        return state["plan"].execute(x)
    if op == "adjoint":
        return state["plan"].adjoint(x)
    if op == "ragged":
        return state["plan"].execute_ragged(x, state["offsets"])
    if op == "train":
        a = x.detach().requires_grad_(True)
        b = convert(a, state["plan"])
        ((b - state["target"]) ** 2).sum().backward()
        return {"beta": b.detach(), "grad": a.grad}
    # one-off: a plan may be released only when its work is done
    plan = _plan(state["case"])
    y = plan.execute(x)
    torch.cuda.current_stream().synchronize()
    plan.close()
    return y


def work(case):
    """Each coefficient read once and written once; a conversion matrix in its most compact
    (data-sparse) form takes about log2 n multiply-adds per coefficient, a banded one two."""
    size = 8 if case["prec"] == "fp64" else 4
    if case["op"] == "ragged":
        coeffs = float(case["batch"]) * case["n"] * _mean_fraction(case)
    else:
        coeffs = float(case["batch"]) * case["n"]
    passes = 2 if case["op"] == "train" else 1
    banded = case["kind"] == "ultra2ultra" and float(case["p1"] - case["p0"]).is_integer()
    per = 4.0 if banded else 2.0 * math.log2(case["n"])
    return {"bytes": 2.0 * size * coeffs * passes, "flops": per * coeffs * passes}


def _mean_fraction(case):
    """Mean length of a ragged batch over its longest (log-uniform lengths)."""
    lo, hi = float(case["nmin"]), float(case["n"])
    return 1.0 if hi <= lo else (hi - lo) / math.log(hi / lo) / hi


# ------------------------------------------------------------------- 64-bit reference


def _gamma_ratio(z0, a, b, count):
    """Gamma(z + a) / Gamma(z + b), z = z0, z0 + 1, ..., by its first-order recurrence in
    extended precision."""
    z = np.arange(count - 1, dtype=np.longdouble) + np.longdouble(z0)
    r = np.ones(count, dtype=np.longdouble)
    r[1:] = np.cumprod((z + np.longdouble(a)) / (z + np.longdouble(b)))
    return r * np.longdouble(math.gamma(z0 + a) / math.gamma(z0 + b))


def _cuda64(v):
    return torch.from_numpy(np.asarray(v, dtype=np.float64)).cuda()


def _toeplitz_hankel_dense(s, h, v, transpose, rows=1024):
    """w_a = sum_{b >= a} s[b-a] h[a+b] v_b (or its transpose) for v [count][batch]."""
    m = v.shape[0]
    w = torch.zeros_like(v)
    pad = torch.cat([torch.zeros(m, dtype=s.dtype, device="cuda"), s[:m]])
    for a0 in range(0, m, rows):
        r = min(rows, m - a0)
        # rows a0+r-1 ... a0 (last first), columns a0 ... m-1: s[b - a] at pad[m + b - a]
        c = m - a0
        t = pad.as_strided((r, c), (1, 1), m - r + 1).flip(0)
        a = t * h.as_strided((r, c), (1, 1), h.storage_offset() + 2 * a0)
        if transpose:
            w[a0:] += a.T @ v[a0:a0 + r]
        else:
            w[a0:a0 + r] = a @ v[a0:]
    return w


def _toeplitz_hankel_fft(s, h, v, transpose):
    """The same through H ~ sum_r u_r u_r^T (pivoted Cholesky run to its rounding floor) and
    zero-padded FFTs, in complex128: O(n log n) terms for vectors too long to do densely."""
    m = v.shape[0]
    d = h[0:2 * m - 1:2].clone()
    top, u = float(d.max()), []
    for _ in range(96):
        p = int(torch.argmax(d))
        if float(d[p]) <= 1e-17 * top:
            break
        col = h[p:p + m].clone()
        for ur in u:
            col -= ur * ur[p]
        if float(col[p]) <= 0.0:
            break
        col /= math.sqrt(float(col[p]))
        u.append(col)
        d = (d - col * col).clamp_min_(0.0)
        d[p] = 0.0
    size = 1 << (2 * m - 1).bit_length()
    f = torch.fft.rfft(s[:m], size)[:, None]
    f = f if transpose else f.conj()
    w = torch.zeros_like(v)
    for ur in u:
        y = torch.fft.rfft(v * ur[:, None], size, dim=0)
        w += torch.fft.irfft(y * f, size, dim=0)[:m] * ur[:, None]
    return w


def _product(s, h, v, transpose):
    dense = v.shape[0] <= 1 << 15
    return (_toeplitz_hankel_dense if dense else _toeplitz_hankel_fft)(s, h, v, transpose)


def _parity_step(lam, hank, d1, d2, x, transpose):
    """diag(d1) (T o H) diag(d2) x, T_jk = lam[(k-j)/2] for even k - j, H_jk = hank[(j+k)/2]
    (hank holds whole and half arguments: hank[e] for parity e)."""
    din, dout = (d1, d2) if transpose else (d2, d1)
    v = x * din[:, None]
    w = torch.empty_like(v)
    for e in range(min(2, x.shape[0])):
        part = v[e::2].contiguous()
        w[e::2] = _product(lam, hank[e], part, transpose)
    return w * dout[:, None]


def _jacobi_step(a, b, g, n, x, transpose):
    """P^(a,b) -> P^(g,b), |a - g| < 1 (Sec. 5.3)."""
    s = g + b + 1.0
    k = np.arange(n, dtype=np.longdouble)
    d1 = _cuda64((2 * k + s) * _gamma_ratio(0.0, s, b + 1.0, n))
    d2 = _cuda64(_gamma_ratio(0.0, b + 1.0, a + b + 1.0, n))
    t = _cuda64(_gamma_ratio(0.0, a - g, 1.0, n) / math.gamma(a - g))
    h = _cuda64(_gamma_ratio(0.0, a + b + 1.0, s + 1.0, 2 * n))
    din, dout = (d1, d2) if transpose else (d2, d1)
    return _product(t, h, x * din[:, None], transpose) * dout[:, None]


def _convert(case, n, x, transpose):
    """A x (or A^T x) in 64 bits for the columns of x [n][batch]."""
    kind, p = case["kind"], _params(case)
    m = (n + 1) // 2
    j = torch.arange(n, device="cuda", dtype=torch.float64)
    if kind == "leg2cheb":
        lam = _cuda64(_gamma_ratio(0.0, 0.5, 1.0, 2 * m + 1))
        d1 = torch.full((n,), 2.0 / math.pi, dtype=torch.float64, device="cuda")
        d1[0] = 1.0 / math.pi
        return _parity_step(lam, [lam, lam[1:]], d1, torch.ones_like(d1), x, transpose)
    if kind == "cheb2leg":
        t = _cuda64(_gamma_ratio(0.0, -0.5, 1.0, m))
        h = _cuda64(np.concatenate([[1.0], _gamma_ratio(1.0, 0.0, 1.5, 2 * m + 1)]))
        d2 = -0.25 * j
        d2[0] = -1.0 / math.sqrt(math.pi)
        return _parity_step(t, [h, h[1:]], j + 0.5, d2, x, transpose)
    if kind == "ultra2ultra":
        diff = p[1] - p[0]
        if abs(diff - round(diff)) < 1e-12:
            return _ultra_whole(p[0], int(round(diff)), j[:, None], x, transpose)
        c = math.gamma(p[1]) / (math.gamma(p[0]) * math.gamma(-diff))
        t = _cuda64(c * _gamma_ratio(0.0, -diff, 1.0, m))
        h = _cuda64(_gamma_ratio(0.0, p[0], p[1] + 1.0, 2 * m + 1))
        # (the sign of 1/Gamma(-diff) goes to T; H is positive)
        return _parity_step(t, [h, h[1:]], j + p[1], torch.ones_like(j), x, transpose)
    # Jacobi: second parameter in the reflected frame, then the first
    a, b, g, d = p
    sign = torch.ones(n, 1, dtype=torch.float64, device="cuda")
    sign[1::2] = -1.0
    if transpose:
        y = _jacobi_step(a, d, g, n, x, True)
        return sign * _jacobi_step(b, a, d, n, sign * y, True)
    y = sign * _jacobi_step(b, a, d, n, sign * x, False)
    return _jacobi_step(a, d, g, n, y, False)


def _ultra_whole(lam, steps, j, x, transpose):
    """C^(lam) -> C^(lam + steps): each factor is (c_j' - c_{j+2}'), c' = lam/(lam+j) c; its
    inverse a suffix sum over every other index."""
    def shift(v, by):
        out = torch.zeros_like(v)
        if by > 0:
            out[:-by] = v[by:]
        else:
            out[-by:] = v[:by]
        return out

    def sums(v, suffix):
        out = torch.empty_like(v)
        for e in range(2):
            part = v[e::2]
            out[e::2] = part.flip(0).cumsum(0).flip(0) if suffix else part.cumsum(0)
        return out

    pars = [lam + i if steps > 0 else lam - 1 - i for i in range(abs(steps))]
    y = x
    for l in (reversed(pars) if transpose else pars):
        c = l / (l + j)
        if steps > 0:
            y = c * (y - shift(y, -2)) if transpose else c * y - shift(c * y, 2)
        else:
            y = sums(y / c, False) if transpose else sums(y, True) / c
    return y


def exact(case, seed):
    x, offsets = _inputs(case, seed)
    if case["op"] == "ragged":
        # pad to the longest; A is upper triangular and its leading block does not depend on
        # n, so zero padding leaves each vector's result as its first entries
        if float(case["batch"]) * case["n"] > 1 << 30:
            return None
        y = torch.empty(x.shape[0], dtype=torch.float64, device="cuda")
        lengths = np.diff(offsets)
        order = np.argsort(lengths, kind="stable")
        lo = 0
        while lo < order.size:  # groups of lengths within a factor of two
            top = max(2 * int(lengths[order[lo]]), 64)
            hi = int(np.searchsorted(lengths[order], top, side="right"))
            grp = order[lo:hi]
            n = int(lengths[grp].max())
            v = torch.zeros(len(grp), n, dtype=torch.float64, device="cuda")
            for i, g in enumerate(grp):
                v[i, :lengths[g]] = x[offsets[g]:offsets[g + 1]]
            w = _convert(case, n, v.T.contiguous(), False).T
            for i, g in enumerate(grp):
                y[offsets[g]:offsets[g + 1]] = w[i, :lengths[g]]
            lo = hi
        return y
    v = x.double().T.contiguous()
    n = case["n"]
    if case["op"] == "train":
        b = _convert(case, n, v, False)
        g = 2.0 * (b - _target(case, seed).double().T)
        return {"beta": b.T.contiguous(), "grad": _convert(case, n, g, True).T.contiguous()}
    return _convert(case, n, v, case["op"] == "adjoint").T.contiguous()
