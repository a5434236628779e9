"""Performance cases: the calls that a user of qless makes, over the range they are made in.

Inputs are X = G S with G i.i.d. N(0,1) and S = V diag(sigma) W^T (sigma geometric from 1 to
1/kappa), the shape of the paper's synthetic workloads, column-major on the GPU.  A pass is
one call of the package's public Python functions with the outputs and the workspace that a
program keeps between calls; every result of the call is returned whole.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2603_20889_gb300 as q

_METHODS = {"tsqr": q.QL_TSQR, "cholqr2": q.QL_CHOLQR2, "svqb2": q.QL_SVQB2, "scholqr3": q.QL_SCHOLQR3}


def listed():
    return [
        # the smallest serving request (2^12 rows, few columns, odd sizes): launches and latency
        {"name": "tsqr_4099x5", "op": "tsqr", "m": 4099, "n": 5, "dtype": "f64", "kappa": 1e2},
        # the plain single matrix of the paper's problem statement, by both of its methods
        {"name": "tsqr_131072x8", "op": "tsqr", "m": 131072, "n": 8, "dtype": "f64", "kappa": 1.0},
        {"name": "cholqr2_131072x8", "op": "cholqr2", "m": 131072, "n": 8, "dtype": "f64", "kappa": 1.0},
        # the narrow, memory-heavy end of the condition sweep
        {"name": "tsqr_33554432x4", "op": "tsqr", "m": 1 << 25, "n": 4, "dtype": "f64", "kappa": 1e4},
        # the widest single matrices: largest serving request, both methods
        {"name": "tsqr_4194304x64", "op": "tsqr", "m": 1 << 22, "n": 64, "dtype": "f64", "kappa": 1e4},
        {"name": "cholqr2_4194304x64", "op": "cholqr2", "m": 1 << 22, "n": 64, "dtype": "f64", "kappa": 1e4},
        # block orthogonalisation inside an eigensolver: SVQB2 of a mid-size block
        {"name": "svqb2_1000000x32", "op": "svqb2", "m": 1000000, "n": 32, "dtype": "f64", "kappa": 1e4},
        # single-pass least squares on FP32-stored data
        {"name": "lstsq_f32_16777216x31", "op": "lstsq", "m": 1 << 24, "n": 31, "dtype": "f32", "kappa": 1e3,
         "method": "tsqr"},
        # an ill-conditioned block of ragged height (columns not 16-byte aligned)
        {"name": "scholqr3_300007x24", "op": "scholqr3", "m": 300007, "n": 24, "dtype": "f64", "kappa": 1e8},
        # the explicit Q of a factored block
        {"name": "q_from_r_8388608x16", "op": "q_from_r", "m": 1 << 23, "n": 16, "dtype": "f64", "kappa": 1e4},
        # a matrix wider than one panel: projections, TSQR panels and Q
        {"name": "qr_wide_524288x128", "op": "qr_wide", "m": 1 << 19, "n": 128, "dtype": "f64", "kappa": 1e3},
        # many uneven problems of both kinds and storages in one batched call
        {"name": "batch_96", "op": "batch", "count": 96, "mix": 7, "max_log2_m": 20},
    ]


# ranges of the drawn cases, per operation: rows, columns (both over their logarithm) and
# the largest condition number
_RANGES = {
    "tsqr": (1 << 12, 1 << 25, 1, 64, 1e6),
    "cholqr2": (1 << 12, 1 << 25, 1, 64, 1e4),
    "svqb2": (1 << 12, 1 << 24, 2, 64, 1e4),
    "lstsq": (1 << 12, 1 << 24, 1, 63, 1e4),
    "scholqr3": (1 << 12, 1 << 22, 2, 64, 1e8),
    "q_from_r": (1 << 12, 1 << 23, 1, 64, 1e4),
    "qr_wide": (1 << 14, 1 << 19, 65, 200, 1e3),
}


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["tsqr", "tsqr", "tsqr", "cholqr2", "cholqr2", "svqb2", "lstsq", "scholqr3", "q_from_r",
                     "qr_wide", "batch"])
    if op == "batch":
        return {"op": op, "count": _log_int(rng, 8, 96), "mix": rng.randrange(1 << 20), "max_log2_m": 20}
    mlo, mhi, nlo, nhi, kmax = _RANGES[op]
    while True:
        m, n = _log_int(rng, mlo, mhi), _log_int(rng, nlo, nhi)
        if rng.random() < 0.5:  # half of the matrices have 16-byte aligned columns in both storages
            m = (m + 3) // 4 * 4
        if m * n <= 1 << 28 and m * n * n <= 1 << (33 if op == "qr_wide" else 34):
            break
    case = {"op": op, "m": m, "n": n, "dtype": "f64" if rng.random() < 0.7 else "f32",
            "kappa": 10.0 ** rng.uniform(0.0, math.log10(kmax))}
    if op == "lstsq":
        case["method"] = rng.choice(["tsqr", "tsqr", "cholqr2"])
    return case


# ------------------------------------------------------------------ inputs


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _mixing(n, kappa, seed):
    """S = V diag(sigma) W^T, V and W random orthogonal."""
    rng = np.random.default_rng([n, seed])
    V, _ = np.linalg.qr(rng.standard_normal((n, n)))
    W, _ = np.linalg.qr(rng.standard_normal((n, n)))
    s = kappa ** (-np.arange(n) / max(n - 1, 1))
    return (V * s) @ W.T


def _matrix(m, n, kappa, dtype, gen, seed):
    """(X, S): X = G S as an m x n column-major view, in `dtype`."""
    S = _mixing(n, kappa, seed)
    Gt = torch.randn((n, m), dtype=torch.float64, device="cuda", generator=gen)
    Xt = torch.as_tensor(S.T.copy(), device="cuda") @ Gt
    del Gt
    return Xt.to(dtype).T, S


def _rhs(A, gen):
    """b = A x* + 1e-6 N(0,1) in A's dtype."""
    xs = torch.randn(A.shape[1], dtype=torch.float64, device="cuda", generator=gen)
    b = torch.zeros(A.shape[0], dtype=torch.float64, device="cuda")
    for j in range(A.shape[1]):
        b += A[:, j].double() * xs[j]
    b += 1e-6 * torch.randn(A.shape[0], dtype=torch.float64, device="cuda", generator=gen)
    return b.to(A.dtype)


def _square(n):
    return torch.empty((n, n), dtype=torch.float64, device="cuda").T


def _dtype(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _shapes(case):
    """The problems of a batch: (m, n, dtype, kind, kappa) each."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        m = int(round(2.0 ** rng.uniform(10.0, case["max_log2_m"])))
        n = rng.randint(4, 48)
        out.append((m, n, "f64" if rng.random() < 0.7 else "f32", 1 if rng.random() < 0.2 else 0,
                    10.0 ** rng.uniform(0.0, 6.0)))
    return out


def _batch_inputs(case, seed):
    gen = _generator(seed)
    out = []
    for i, (m, n, dt, kind, kappa) in enumerate(_shapes(case)):
        X, _ = _matrix(m, n, kappa, torch.float64 if dt == "f64" else torch.float32, gen, seed * 1009 + i)
        out.append((X, _rhs(X, gen) if kind else None, kind, kappa))
    return out


def _inputs(case, seed):
    gen = _generator(seed)
    X, S = _matrix(case["m"], case["n"], case["kappa"], _dtype(case), gen, seed)
    if case["op"] == "lstsq":
        return X, _rhs(X, gen)
    if case["op"] == "q_from_r":
        # the triangle of S, scaled by sqrt(m): X R^-1 is orthonormal up to G's sampling
        R = np.linalg.qr(S, mode="r") * math.sqrt(case["m"])
        R *= np.sign(np.diag(R))[:, None]
        return X, torch.as_tensor(np.ascontiguousarray(np.triu(R).T), device="cuda").T
    return X, None


def prepare(case, seed):
    op = case["op"]
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    if op == "batch":
        # the triangles, the solutions (48 + 1 entries at most) and the statuses in one buffer each
        probs, keep, off, count = [], [], 0, case["count"]
        R = torch.zeros(sum((n + kind) ** 2 for _, n, _, kind, _ in _shapes(case)), dtype=torch.float64, device="cuda")
        x = torch.zeros((count, 49), dtype=torch.float64, device="cuda")
        infos = torch.zeros((count, 2), dtype=torch.int32, device="cuda")
        for i, (X, b, kind, kappa) in enumerate(_batch_inputs(case, seed)):
            n = X.shape[1]
            probs.append(q.Problem(m=X.shape[0], n=n, ld=X.stride(1), X=X.data_ptr(),
                                   dtype=q.QL_F64 if X.dtype == torch.float64 else q.QL_F32, kind=kind,
                                   b=b.data_ptr() if kind else None, R=R[off:].data_ptr(),
                                   x=x[i].data_ptr() if kind else None, info=infos[i].data_ptr(),
                                   method_hint=q.QL_AUTO, kappa_hint=kappa))
            keep.append((X, b))
            off += (n + kind) ** 2
        arr = (q.Problem * count)(*probs)
        nb = q.load_library().ql_batch_workspace_bytes(count, arr)
        return {"op": op, "probs": probs, "keep": keep, "out": [R, x, infos],
                "ws": torch.empty(nb, dtype=torch.uint8, device="cuda")}
    m, n = case["m"], case["n"]
    X, other = _inputs(case, seed)
    st = {"op": op, "X": X, "info": info}
    code = q.QL_F64 if case["dtype"] == "f64" else q.QL_F32
    if op == "lstsq":
        st.update(b=other, method=_METHODS[case["method"]], ws=q.workspace(q.QL_AUTO, m, n, code))
    elif op == "q_from_r":
        st.update(R=other, Q=torch.empty((n, m), dtype=X.dtype, device="cuda").T)
    elif op == "qr_wide":
        nb = q.load_library().ql_qr_wide_workspace_bytes(m, n, code)
        st.update(R=_square(n), Q=torch.empty((n, m), dtype=X.dtype, device="cuda").T,
                  ws=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    else:
        st.update(R=_square(n), ws=q.workspace(_METHODS[op], m, n, code))
    return st


def run(state):
    op = state["op"]
    if op == "batch":
        q.batch_qless(state["probs"], ws=state["ws"])
        return state["out"]
    X, info = state["X"], state["info"]
    if op == "tsqr":
        R, info = q.tsqr_qless(X, R=state["R"], info=info, ws=state["ws"])
        return [R, info]
    if op == "cholqr2":
        R, info = q.cholqr2_qless(X, R=state["R"], info=info, ws=state["ws"])
        return [R, info]
    if op == "scholqr3":
        R, info = q.scholqr3_qless(X, R=state["R"], info=info, ws=state["ws"])
        return [R, info]
    if op == "svqb2":
        R, _, info = q.svqb_qless(X, R=state["R"], info=info, ws=state["ws"])
        return [R, info]
    if op == "lstsq":
        x, rn, _, info = q.lstsq_qless(X, state["b"], method=state["method"], info=info, ws=state["ws"])
        return [x, rn, info]
    if op == "q_from_r":
        Q, info = q.q_from_r(X, state["R"], Q=state["Q"], info=info)
        return [Q, info]
    Q, R, info = q.qr_wide(X, R=state["R"], Q=state["Q"], info=info, ws=state["ws"])
    return [Q, R, info]


# ------------------------------------------------------------------ work and exact results


# flops per m n^2: Householder R; Gram, then Gram plus the product with R1^-1 or B1 per later pass
_FLOPS = {"tsqr": 2.0, "lstsq": 2.0, "cholqr2": 5.0, "svqb2": 6.0, "scholqr3": 8.0, "q_from_r": 1.0, "qr_wide": 4.0}


def work(case):
    if case["op"] == "batch":
        by = fl = 0.0
        for m, n, dt, kind, _ in _shapes(case):
            c = n + kind
            by += m * c * (8 if dt == "f64" else 4) + 8.0 * c * c
            fl += 2.0 * m * c * c
        return {"bytes": by, "flops": fl}
    m, n, s = case["m"], case["n"], 8 if case["dtype"] == "f64" else 4
    cols = n + 1 if case["op"] == "lstsq" else n
    by = float(m) * cols * s + 8.0 * (cols if case["op"] == "lstsq" else n * n)
    if case["op"] in ("q_from_r", "qr_wide"):
        by += float(m) * n * s
    return {"bytes": by, "flops": _FLOPS[case["op"]] * m * cols * cols}


def _r64(*parts):
    """R (nonnegative diagonal) of [parts...] side by side, by QR of row blocks in float64."""
    m, n = parts[0].shape[0], sum(p.shape[1] for p in parts)
    step = max(1 << 14, (1 << 24) // n)
    rs = []
    for i in range(0, m, step):
        blk = torch.cat([p[i:i + step].double() for p in parts], dim=1)
        rs.append(torch.linalg.qr(blk, mode="r")[1])
    R = torch.linalg.qr(torch.cat(rs), mode="r")[1] if len(rs) > 1 else rs[0]
    return torch.triu(R * torch.where(torch.diagonal(R) < 0, -1.0, 1.0)[:, None])


def _lstsq64(A, b):
    R = _r64(A, b[:, None])
    n = A.shape[1]
    x = torch.linalg.solve_triangular(R[:n, :n], R[:n, n:], upper=True)[:, 0]
    return R, x, R[n, n].reshape(1)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        rs, xs = [], torch.zeros((case["count"], 49), dtype=torch.float64, device="cuda")
        for i, (X, b, kind, _) in enumerate(_batch_inputs(case, seed)):
            if kind:
                R, x, rho = _lstsq64(X, b)
                xs[i, :len(x) + 1] = torch.cat([x, rho])
            else:
                R = _r64(X)
            rs.append(R.T.reshape(-1))
        return [torch.cat(rs), xs, None]
    X, other = _inputs(case, seed)
    if op == "lstsq":
        _, x, rho = _lstsq64(X, other)
        return [x, rho, None]
    if op == "q_from_r":
        return [torch.linalg.solve_triangular(other, X.double(), upper=True, left=False), None]
    if op == "qr_wide":
        Q, R = torch.linalg.qr(X.double())
        s = torch.where(torch.diagonal(R) < 0, -1.0, 1.0)
        return [Q * s, torch.triu(R * s[:, None]), None]
    return [_r64(X), None]
