"""The exact Gram route on long inputs (full groups of tiles, sets of sums and emptied 128-bit sums
in every column class), the Householder tiles behind it, and the single calls' chains of dependent
launches under capture and side by side on streams."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2603_20889_gb300 import synth

from test_gpu_exact_gram import gram_error, row_error

pytestmark = pytest.mark.gpu


def r_of_gram(C):
    """R of an integer Gram matrix (nested lists of int), Cholesky in 400-bit fixed point."""
    from math import isqrt

    n, bits = len(C), 400
    S = [[v << bits for v in row] for row in C]
    R = np.zeros((n, n))
    for k in range(n):
        r = [isqrt(S[k][k] << bits)] * (k + 1) + [0] * (n - k - 1)
        for j in range(k + 1, n):
            r[j] = (S[k][j] << bits) // r[k]
        for i in range(k + 1, n):
            for j in range(i, n):
                S[i][j] -= r[i] * r[j] >> bits
        R[k, k:] = [v / (1 << bits) for v in r[k:]]
    return R


@pytest.mark.parametrize("m,n,ld", [((1 << 24) - 37, 4, 1 << 24), (1 << 24, 8, 1 << 24), ((1 << 24) - 37, 8, 1 << 24),
                                    (1 << 24, 16, 1 << 24), ((1 << 24) - 5, 31, 1 << 24), ((1 << 23) - 9, 64, 1 << 23)])
def test_every_read_out_of_a_long_input(m, n, ld):
    """2^50 X = 2^40 A + B, A and B integers below 2^12: exact in FP64 and in the fixed point, C from three
    exact FP64 products.  More tiles per CTA than a read-out and than the 128-bit sums take; R rounds
    once per entry."""
    import torch

    import paper_2603_20889_gb300 as q

    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    A, B = (torch.randint(-4095, 4096, (n, m), device="cuda", generator=g).double() for _ in range(2))
    buf = torch.zeros((n, ld), dtype=torch.float64, device="cuda")
    buf[:, :m] = (A * 2.0 ** 40 + B) * 2.0 ** -50  # inside the double-float range
    AA, AB, BB = ((U @ V.T).cpu().numpy() for U, V in ((A, A), (A, B), (B, B)))  # below 2^48
    del A, B
    C = [[(int(AA[i, j]) << 80) + ((int(AB[i, j]) + int(AB[j, i])) << 40) + int(BB[i, j]) for j in range(n)]
         for i in range(n)]
    ref = r_of_gram(C) * 2.0 ** -50
    X = buf[:, :m].T
    R, info = q.tsqr_qless(X)
    assert info.cpu().tolist() == [0, 0] and row_error(R.cpu().numpy(), ref) <= 2.0 ** -52
    if n > 4:
        x, rn, Rext, info = q.lstsq_qless(X[:, : n - 1], X[:, n - 1], want_rext=True)
        assert info.cpu().tolist() == [0, 0] and row_error(Rext.cpu().numpy(), ref) <= 2.0 ** -52
    Rc, _ = q.cholqr2_qless(X)
    assert torch.equal(R, Rc)


@pytest.mark.parametrize("n", [3, 4])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_tile_edges_of_the_four_column_class(n, dtype):
    import torch

    import paper_2603_20889_gb300 as q

    for m, pad in ((1023, 1), (1024, 0), (1025, 3), (3077, 3), (5 * 1024 - 1, 1), (5 * 1024 + 1, 7)):
        X = synth.conditioned(m, n, 100.0, seed=m + n, dtype=dtype)
        buf = torch.zeros((n, m + pad), dtype=torch.float64 if dtype == np.float64 else torch.float32, device="cuda")
        buf[:, :m] = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        ref = oracle.householder_r(X.astype(np.float64))
        calls = [q.cholqr2_qless, q.scholqr3_qless] + ([q.tsqr_qless] if m >= 4096 else [])
        for fn in calls:
            R, info = fn(buf[:, :m].T)
            assert info.cpu().tolist() == [0, 0]
            assert oracle.rel_err(R.cpu().numpy(), ref) <= oracle.tolerance(n, 100.0), m


CHILD = """
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np, torch
import oracle, paper_2603_20889_gb300 as q
from paper_2603_20889_gb300 import synth
for n, log2m in ((4, 22), (8, 20), (16, 19), (24, 18), (32, 18), (40, 17), (64, 17)):
    X, R0 = synth.hadamard_exact_case(1 << log2m, n, 1e4, seed=n)
    R, info = q.tsqr_qless(torch.from_numpy(np.ascontiguousarray(X.T)).cuda().T)
    assert info.cpu().tolist() == [0, 0], n
    err = oracle.rel_err(R.cpu().numpy(), R0)
    assert err <= oracle.tolerance(n, 1e4), (n, err)
    print(n, err)
"""


def test_householder_tiles_of_every_class_over_many_tiles():
    """The tiles that the exact pass falls back to, three row tiles per CTA and more (with the
    tensor-core Gram kernels off every TSQR call runs on them), against an exact R."""
    root = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..")
    p = subprocess.run([sys.executable, "-c", CHILD, root], env=dict(os.environ, QL_GRAM_SIMT="1"), capture_output=True,
                       text=True, timeout=600)
    assert p.returncode == 0, p.stdout + p.stderr


def test_batch_redo_that_leaves_the_double_float_range():
    """A nearly dependent column with light rows at the end (lost to the fixed point: the tiles redo
    the problem), the last of them below the tiles' range in a whole chunk but not in a whole chunk
    of the exact launch: one CTA refactors the problem in FP64."""
    import torch

    import paper_2603_20889_gb300 as q

    m, n = 1 << 18, 6
    X = synth.gaussian(m, n, seed=11)
    X[:, 4] = X[:, 0] + 1e-4 * X[:, 4]
    X[-6000:] *= 2.0 ** -45
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    outs, probs = [], []
    for k in range(3):
        R = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        info = torch.full((2,), -1, dtype=torch.int32, device="cuda")
        outs.append((R, info))
        probs.append(q.Problem(m=m, n=n, ld=m, X=Xd.data_ptr(), dtype=q.QL_F64, kind=0, b=None, R=R.data_ptr(), x=None,
                               info=info.data_ptr(), method_hint=q.QL_TSQR, kappa_hint=0.0))
    q.batch_qless(probs)
    torch.cuda.synchronize()
    ref = oracle.householder_r(X)
    for R, info in outs:
        R = R.cpu().numpy().T
        assert info.cpu().tolist() == [0, 0] and gram_error(R, X) <= 1e-13 * n
        assert oracle.rel_err(R, ref) <= oracle.tolerance(n, 1e5)


def single_calls(q, torch):
    """(name, call into kept outputs, outputs, inputs) of every single entry point, on routes that end
    early and on ones that run their gated launches."""
    out = []
    for k, (m, n) in enumerate(((20000, 3), (4099, 5), (30000, 8), (9000, 40), (50000, 1))):
        X = torch.from_numpy(np.ascontiguousarray(synth.conditioned(m, n, 50.0, seed=k).T)).cuda().T
        heavy = X.clone()
        heavy[0] *= 2.0 ** 30  # light rows below: Householder tiles, or the Gram methods' passes
        b = X.sum(1) + 1.0
        for name, A in (("plain", X), ("heavy", heavy)):
            R = torch.empty((n, n), dtype=torch.float64, device="cuda").T
            info = torch.zeros(2, dtype=torch.int32, device="cuda")
            for fn, code in ((q.tsqr_qless, q.QL_TSQR), (q.cholqr2_qless, q.QL_CHOLQR2), (q.scholqr3_qless, q.QL_SCHOLQR3)):
                R, info, ws = torch.empty_like(R), torch.zeros_like(info), q.workspace(code, m, n, q.QL_F64)
                out.append((f"{fn.__name__} {m}x{n} {name}",
                            lambda s, fn=fn, A=A, R=R, info=info, ws=ws: fn(A, R=R, info=info, ws=ws, stream=s), (R, info)))
            R, info, ws = torch.empty_like(R), torch.zeros_like(info), q.workspace(q.QL_SVQB2, m, n, q.QL_F64)
            out.append((f"svqb {m}x{n} {name}",
                        lambda s, A=A, R=R, info=info, ws=ws: q.svqb_qless(A, R=R, info=info, ws=ws, stream=s), (R, info)))
            if n < 40:
                keep, info, ws = [], torch.zeros_like(info), q.workspace(q.QL_AUTO, m, n, q.QL_F64)

                def ls(s, A=A, b=b, keep=keep, info=info, ws=ws):
                    keep[:] = q.lstsq_qless(A, b, info=info, ws=ws, stream=s)[:2]

                out.append((f"lstsq {m}x{n} {name}", ls, (keep, info)))
    return out


def snapshot(outs):
    a, info = outs
    return [t.clone() for t in (a if isinstance(a, list) else [a])] + [info.clone()]


def same(a, b):  # equal entries, NaN where a breakdown is reported
    return bool(((a == b) | ((a != a) & (b != b))).all())


def test_single_calls_under_capture():
    """Every call captured by itself and replayed twice gives the bits of the direct call."""
    import torch

    import paper_2603_20889_gb300 as q

    s = torch.cuda.Stream()
    for name, call, outs in single_calls(q, torch):
        with torch.cuda.stream(s):
            call(s)
        torch.cuda.synchronize()
        want = snapshot(outs)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call(s)
        for _ in range(2):
            for t in (outs[0] if isinstance(outs[0], list) else [outs[0]]) + [outs[1]]:
                t.fill_(-3)
            g.replay()
            torch.cuda.synchronize()
            assert all(same(a, b) for a, b in zip(snapshot(outs), want)), name


def test_single_calls_side_by_side_on_streams():
    """The calls, each with its own outputs and workspace, over three streams at once: the bits of the
    calls one after the other."""
    import torch

    import paper_2603_20889_gb300 as q

    calls = single_calls(q, torch)
    main = torch.cuda.current_stream()
    want = []
    for _, call, outs in calls:
        call(main)
        torch.cuda.synchronize()
        want.append(snapshot(outs))
    streams = [torch.cuda.Stream() for _ in range(3)]
    for _ in range(5):
        for k, (_, call, outs) in enumerate(calls):
            with torch.cuda.stream(streams[k % 3]):
                call(streams[k % 3])
        torch.cuda.synchronize()
        for (name, _, outs), w in zip(calls, want):
            assert all(same(a, b) for a, b in zip(snapshot(outs), w)), name
