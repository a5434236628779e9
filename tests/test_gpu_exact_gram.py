"""The exact Gram route (n >= 2): tile edges, column classes, scale changes, zero and
dependent columns, unaligned columns, and the hand-over to the Householder tiles.

Tolerance.  X is rounded to 2^-56 of each column's largest entry and everything after that is
exact to 2^-100, so ||R - R_ref|| <= (2^-55 kappa + 2^-52) ||R_ref|| n; the bound of the other
parity tests, 1e-13 n kappa, is far above it.  R^T R is compared with X^T X formed in FP64 by
row blocks (rounding below 1e-14 n of the column norms).
"""
import numpy as np
import pytest

import oracle
from paper_2603_20889_gb300 import synth

pytestmark = pytest.mark.gpu


def tsqr(X, pad=0):
    import torch

    import paper_2603_20889_gb300 as q

    m, n = X.shape
    buf = torch.zeros((n, m + pad), dtype=torch.float64 if X.dtype == np.float64 else torch.float32, device="cuda")
    buf[:, :m] = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    R, info = q.tsqr_qless(buf[:, :m].T)
    return R.cpu().numpy(), info.cpu().tolist()


def gram_error(R, X):
    G = X.astype(np.float64).T @ X.astype(np.float64)
    d = np.sqrt(np.diag(G))
    return np.abs((R.T @ R - G) / np.where(d > 0, d, 1)[:, None] / np.where(d > 0, d, 1)[None, :]).max()


@pytest.mark.parametrize("n", [2, 4, 5, 8, 9, 16, 17, 32, 33, 64])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_tile_edges_against_oracle(n, dtype):
    kt = 4096 // (4 if n <= 4 else 8 if n <= 8 else 16 if n <= 16 else 32 if n <= 32 else 64)
    for m, pad in ((n, 0), (kt - 1, 1), (kt, 0), (kt + 1, 2), (3 * kt + 5, 3)):
        X = synth.conditioned(max(m, n), n, 100.0, seed=m + n, dtype=dtype)
        R, info = tsqr(X, pad)
        assert info == [0, 0]
        ref = oracle.householder_r(X.astype(np.float64))
        # a square Gaussian X may be far worse conditioned than its mixing matrix
        kappa = max(100.0, np.linalg.cond(X.astype(np.float64)))
        assert oracle.rel_err(R, ref) <= oracle.tolerance(n, kappa), (m, pad)


@pytest.mark.parametrize("n,log2m", [(3, 19), (8, 18), (16, 17), (32, 16), (64, 16)])
def test_many_tiles_per_cta_exact_r(n, log2m):
    X, R0 = synth.hadamard_exact_case(1 << log2m, n, 1e4, seed=n)
    R, info = tsqr(X)
    assert info == [0, 0]
    assert oracle.rel_err(R, R0) <= 1e-15  # R0 is exact; R rounds once per entry


@pytest.mark.parametrize("n,m", [(4, 500002), (5, 200001), (16, 100003), (32, 60002), (64, 40000)])
def test_growing_rows_raise_the_column_scales(n, m):
    X = synth.gaussian(m, n, seed=n) * np.exp2(np.floor(24.0 * np.arange(m) / m))[:, None]
    R, info = tsqr(X)
    assert info == [0, 0]
    assert gram_error(R, X) <= 1e-14 * n


@pytest.mark.parametrize("n", [6, 24, 40])
def test_zero_and_far_apart_entries(n):
    X = synth.gaussian(5000, n, seed=3)
    X[:, 2] = 0.0                      # a zero column stays on the exact route
    X[::7, 1] *= 2.0 ** -30            # entries far below the column's scale
    X[::3, 3] = 0.0
    R, info = tsqr(X)
    assert info == [0, 0] and R[2, 2] == 0.0 and np.all(R[2, 3:] == 0.0)
    assert gram_error(R, X) <= 1e-14 * n


@pytest.mark.parametrize("n", [4, 8, 20, 64])
def test_dependent_columns_go_to_householder(n):
    X = synth.gaussian(3000, n, seed=5)
    X[:, n - 1] = X[:, 0]              # pivot exactly zero: the Householder tiles redo the call
    R, info = tsqr(X)
    assert info == [0, 0] and np.all(np.isfinite(R)) and np.all(np.diag(R) >= 0.0)
    assert R[n - 1, n - 1] <= 1e-12 * R[0, 0]
    assert gram_error(R, X) <= 1e-13 * n


def test_very_ill_conditioned_matches_oracle():
    for kappa in (1e9, 1e12, 1e14):    # the last one below the pivot limit of the exact route
        X = synth.conditioned(4000, 12, kappa, seed=9)
        R, info = tsqr(X)
        assert info == [0, 0]
        assert oracle.rel_err(R, oracle.householder_r(X)) <= oracle.tolerance(12, kappa)


@pytest.mark.parametrize("n", [4, 7, 16, 33])
@pytest.mark.parametrize("kappa,rank_tol", [(1e3, 0.0), (1e3, 1e-4), (1e7, 0.0)])
def test_svqb2_with_and_without_z_agree(n, kappa, rank_tol):
    """Z forces both eigensolves; without it the exact pass may answer, but not where an
    eigenvalue is truncated (kappa^-2 < rank_tol, or kappa^2 n 2^-52 > 1)."""
    import torch

    import paper_2603_20889_gb300 as q

    X = synth.conditioned(6000, n, kappa, seed=n)
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().T
    Rz, Z, iz = q.svqb_qless(Xd, rank_tol=rank_tol, want_z=True)
    R, _, i = q.svqb_qless(Xd, rank_tol=rank_tol)
    assert i.cpu().tolist() == iz.cpu().tolist()
    assert oracle.rel_err(R.cpu().numpy(), Rz.cpu().numpy()) <= 2 * oracle.tolerance(n, min(kappa, 1e6))


@pytest.mark.parametrize("n", [3, 6, 20, 40])
def test_gram_methods_against_oracle_on_both_sides_of_the_limits(n):
    import torch

    import paper_2603_20889_gb300 as q

    for kappa, fn in ((1e2, q.cholqr2_qless), (1e6, q.cholqr2_qless), (1e2, q.scholqr3_qless),
                      (1e8, q.scholqr3_qless), (1e10, q.scholqr3_qless)):
        X = synth.conditioned(5001, n, kappa, seed=n + 1)
        Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().T
        R, info = fn(Xd)
        assert info.cpu().tolist() == [0, 0]
        assert oracle.rel_err(R.cpu().numpy(), oracle.householder_r(X)) <= oracle.tolerance(n, kappa)


def test_gram_methods_still_report_breakdowns():
    import torch

    import paper_2603_20889_gb300 as q

    X = synth.gaussian(4000, 10, seed=1)
    X[:, 6] = 0.0                      # zero column: not the exact route's to answer here
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().T
    assert q.cholqr2_qless(Xd)[1].cpu().tolist() == [q.QL_ERR_NOT_SPD, 7]
    assert q.scholqr3_qless(Xd)[1].cpu().tolist() == [q.QL_ERR_NOT_SPD, 1007]


@pytest.mark.parametrize("hint", ["tsqr", "auto", "cholqr2"])
def test_batch_of_every_class_and_every_way_out(hint):
    """One batch: every column class and both storages on the exact launch, and problems that
    its last launch redoes (dependent columns, data out of the double-float range)."""
    import torch

    import paper_2603_20889_gb300 as q

    mats, keep, probs = [], [], []
    for k, n in enumerate([1, 2, 3, 4, 6, 8, 13, 16, 20, 32, 40, 64, 9, 30]):
        m = [3001, 40000, 2048][k % 3]
        X = synth.conditioned(m, n, 10.0 ** (k % 4), seed=k, dtype=np.float32 if k % 3 == 2 else np.float64)
        if n == 13 and hint != "cholqr2":
            X[:, 7] = X[:, 2]                      # pivot zero
        if n == 20:
            X = X * 2.0 ** 70                      # beyond the range check
        if n == 9:
            X[:, 4] *= 0.0 if hint != "cholqr2" else 1.0
        if n == 30:
            X = synth.conditioned(m, n, 1e8, seed=k)   # beyond Cholesky-QR2's pivot limit
        mats.append(X)
        d = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
        R = torch.zeros((n, n), dtype=torch.float64, device="cuda")
        info = torch.full((2,), -1, dtype=torch.int32, device="cuda")
        keep.append((d, R, info))
        probs.append(q.Problem(m=m, n=n, ld=m, X=d.data_ptr(), dtype=q.QL_F64 if X.dtype == np.float64 else q.QL_F32,
                               kind=0, b=None, R=R.data_ptr(), x=None, info=info.data_ptr(),
                               method_hint={"tsqr": q.QL_TSQR, "auto": q.QL_AUTO, "cholqr2": q.QL_CHOLQR2}[hint],
                               kappa_hint=1e4))
    q.batch_qless(probs)
    torch.cuda.synchronize()
    for X, (_, R, info) in zip(mats, keep):
        n = X.shape[1]
        R = R.cpu().numpy().T
        assert info.cpu().tolist() == [0, 0], n
        assert np.all(np.diag(R) >= 0.0) and gram_error(R, X) <= 1e-13 * n, n
        if n not in (9, 13):
            kappa = 1e8 if n == 30 else 1e3
            assert oracle.rel_err(R, oracle.householder_r(X.astype(np.float64))) <= oracle.tolerance(n, kappa), n


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("n,m", [(1, 4099), (2, 700000), (3, 4099), (3, 700000), (3, 700003), (7, 350000), (15, 150000)])
def test_right_hand_side_rows_stay_with_their_rows(n, m, dtype):
    # repeated on data that stays in L2, where a copy into a stage follows its release soonest: one
    # 16-byte piece of a column read from another tile changes the Gram matrix by about 2 / m
    import torch

    import paper_2603_20889_gb300 as q

    X = synth.gaussian(m, n + 1, seed=m + n).astype(dtype)
    A = torch.from_numpy(np.ascontiguousarray(X[:, :n].T)).cuda().T
    b = torch.from_numpy(np.ascontiguousarray(X[:, n])).cuda()
    for _ in range(12):
        x, rn, R, info = q.lstsq_qless(A, b, want_rext=True)
        assert info.cpu().tolist() == [0, 0]
        assert gram_error(R.cpu().numpy(), X) <= 1e-14 * (n + 1)
        assert rn.item() == R[n, n].item()


def r_of_integers(X):
    """R of X with integer entries: the Gram matrix in integers, Cholesky in 400-bit fixed point."""
    from math import isqrt

    n, bits = X.shape[1], 400
    cols = [[int(v) for v in X[:, j].tolist()] for j in range(n)]
    S = [[sum(a * b for a, b in zip(cols[i], cols[j])) << bits if j >= i else 0 for j in range(n)] for i in range(n)]
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


def row_error(R, ref):
    return (np.abs(R - ref).max(axis=1) / np.abs(ref).max(axis=1)).max()


def heavy_rows(m, n, where, log2w):
    """Rows of N(0,1) (integers up to 2^53) under a few rows 2^log2w times as large."""
    X = np.rint(np.random.default_rng(m + n).standard_normal((m, n)) * 2.0 ** 50)
    if where == "parallel":  # every fourth row along one direction, in half of the columns
        X[::4] = 0.0
        X[::4, : (n + 1) // 2] = np.rint(np.linspace(1.0, 2.0, (n + 1) // 2) * 2.0 ** 30) * 2.0 ** (20 + log2w)
        return X
    X[{"first": [0, 1], "last": [m - 1], "spread": list(range(5, m, m // 2))}[where]] *= 2.0 ** log2w
    return X


@pytest.mark.parametrize("where", ["first", "last", "spread", "parallel"])
@pytest.mark.parametrize("m,n,log2w", [(16384, 3, 30), (16385, 3, 24), (16384, 8, 30), (4096, 14, 24), (70000, 14, 30)])
def test_light_rows_under_heavy_ones(m, n, log2w, where):
    """R row by row, against exact integers: no further off than the Householder tiles (the
    workspace-free entry) by more than a factor of two, or than 2^-44 n: 48-bit entries, a few
    roundings of that size per column.  Gram calls of up to 8 columns: 2^-44 n."""
    import ctypes

    import torch

    import paper_2603_20889_gb300 as q

    X = heavy_rows(m, n, where, log2w) * 2.0 ** -50
    ref = r_of_integers(X * 2.0 ** 50) * 2.0 ** -50
    Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda().T
    Rh = torch.zeros((n, n), dtype=torch.float64, device="cuda").T
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    L = q.load_library()
    assert L.ql_tsqr_qless_noalloc(m, n, Xd.data_ptr(), q.QL_F64, m, Rh.data_ptr(), n, info.data_ptr(),
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == q.QL_OK
    bound = max(n * 2.0 ** -44, 2.0 * row_error(Rh.cpu().numpy(), ref))
    R, info = q.tsqr_qless(Xd)
    assert info.cpu().tolist() == [0, 0] and row_error(R.cpu().numpy(), ref) <= bound
    if n == 3 and where != "parallel":  # kappa of the others is beyond the Gram methods
        R, info = q.cholqr2_qless(Xd)
        assert info.cpu().tolist() == [0, 0] and row_error(R.cpu().numpy(), ref) <= n * 2.0 ** -44


@pytest.mark.parametrize("m,n", [(20000, 3), (3001, 5), (5000, 8), (2000, 16), (1500, 33), (900, 64)])
def test_numerically_dependent_columns(m, n):
    """A pivot below 2^-96 of its column gives a zero row, as the Householder tiles give; one of about
    2^-86 is resolved where X itself is exact in the fixed point (integers below 2^47: an error of
    n 2^-117 in the Schur complement, 2^-25 of that pivot at 64 columns)."""
    import torch

    import paper_2603_20889_gb300 as q

    X = np.random.default_rng(n).integers(-7, 8, (m, n)).astype(np.float64)
    k = n // 2 + 1
    Xs = X.copy()
    Xs[:, k] = 0.3 * X[:, 0] + X[:, k - 1] / 3.0  # rounded sums: dependent to 2^-53
    R, info = tsqr(Xs)
    assert info == [0, 0] and np.all(R[k, k:] == 0.0)
    assert gram_error(R, Xs) <= 1e-13 * n
    X[:, k] += X[:, 0] * 2.0 ** 43
    ref = r_of_integers(X)
    R, info = tsqr(X)
    assert info == [0, 0] and row_error(R, ref) <= 2.0 ** -24
    if n < 64:
        A = torch.from_numpy(np.ascontiguousarray(Xs.T)).cuda().T
        b = torch.from_numpy(np.random.default_rng(1).standard_normal(m)).cuda()
        x, rn, _, info = q.lstsq_qless(A, b)
        assert info.cpu().tolist() == [q.QL_ERR_NOT_SPD, k + 1] and bool(torch.isnan(x).all())


@pytest.mark.parametrize("m,n", [(20000, 2), (3000, 7), (2000, 20), (1000, 63), (6, 6), (40, 40)])
def test_consistent_least_squares(m, n):
    """b = A 1 up to the rounding of its entries: x to kappa 2^-50, the residual norm to 2^-52 ||b||."""
    import torch

    import paper_2603_20889_gb300 as q

    A = synth.conditioned(m, n, 10.0, seed=n) if m > n else np.eye(n) + 0.25 * np.triu(np.ones((n, n))) / n
    b = A @ np.ones(n)
    x, rn, _, info = q.lstsq_qless(torch.from_numpy(np.ascontiguousarray(A.T)).cuda().T, torch.from_numpy(b).cuda())
    assert info.cpu().tolist() == [0, 0]
    assert np.abs(x.cpu().numpy() - 1.0).max() <= 100 * n * 2.0 ** -50
    assert 0.0 <= rn.item() <= 4 * n * 2.0 ** -52 * np.linalg.norm(b)


@pytest.mark.parametrize("n,rows", [(3, 4096), (4, 4096), (5, 5), (40, 40)])
def test_both_sides_of_the_routes_line(n, rows):
    """One row below the line the Householder tiles answer, at the line the exact pass; with fewer
    rows than columns the rows of R past the last one are zero."""
    for m in (rows - 1, rows, rows + 1):
        X = synth.gaussian(m, n, seed=m)
        R, info = tsqr(X)
        assert info == [0, 0] and gram_error(R, X) <= 1e-13 * n
        assert np.all(R[m:] == 0.0)


@pytest.mark.parametrize("n,rows", [(2, 8192), (3, 8192), (4, 2048), (5, 2048), (7, 8)])
def test_both_sides_of_the_routes_line_least_squares(n, rows):
    import torch

    import paper_2603_20889_gb300 as q

    for m in (rows - 1, rows, rows + 1):
        A, b, _ = synth.lstsq_case(m, n, 10.0, seed=m)
        x_ref, rho_ref, _, _ = oracle.lstsq(A, b)
        x, rn, _, info = q.lstsq_qless(torch.from_numpy(np.ascontiguousarray(A.T)).cuda().T, torch.from_numpy(b).cuda())
        assert info.cpu().tolist() == [0, 0]
        kappa = max(10.0, np.linalg.cond(A))
        assert np.linalg.norm(x.cpu().numpy() - x_ref) <= oracle.tolerance(n, kappa) * kappa * np.linalg.norm(x_ref)
        assert abs(rn.item() - rho_ref) <= oracle.tolerance(n, kappa) * np.linalg.norm(b)


def test_batch_across_the_tiles_line():
    """Both sides of the batch's line between Householder tiles and the exact launch, in one call
    and with every problem on one side; least squares among them."""
    import torch

    import paper_2603_20889_gb300 as q

    small = [(3001, 1), (70000, 1), (50000, 2), (16383, 4), (4096, 8), (1023, 16), (5, 9), (300, 3), (0, 4)]
    large = [(16384, 3), (4097, 8), (4097, 5), (1024, 16), (200, 17), (3000, 40)]
    for shapes in (small, large, small + large, small + large + [(1 << 21, 1)]):
        probs, keep = [], []
        for k, (m, n) in enumerate(shapes):
            X = synth.gaussian(max(m, 1), n, seed=k)[:m]
            ls = k % 3 == 1 and m > n + 1
            Xd = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
            b = torch.from_numpy(synth.gaussian(max(m, 1), 1, seed=k + 50)[:, 0].copy()).cuda()
            R = torch.zeros((n + ls, n + ls), dtype=torch.float64, device="cuda")
            x = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
            info = torch.full((2,), -1, dtype=torch.int32, device="cuda")
            keep.append((X, b, ls, Xd, R, x, info))
            probs.append(q.Problem(m=m, n=n, ld=max(m, 1), X=Xd.data_ptr(), dtype=q.QL_F64, kind=int(ls),
                                   b=b.data_ptr() if ls else None, R=R.data_ptr(), x=x.data_ptr() if ls else None,
                                   info=info.data_ptr(), method_hint=q.QL_AUTO, kappa_hint=0.0))
        q.batch_qless(probs)
        torch.cuda.synchronize()
        for X, b, ls, _, R, x, info in keep:
            m, n = X.shape
            full = np.column_stack([X, b.cpu().numpy()[:m]]) if ls else X
            R = R.cpu().numpy().T
            assert info.cpu().tolist() == [0, 0], (m, n)
            assert gram_error(R, full) <= 1e-13 * (n + 1), (m, n)
            if ls:
                assert x[n].item() == R[n, n]


@pytest.mark.parametrize("n,m", [(3, 20000), (8, 4097), (20, 5000), (64, 3000)])
def test_cholqr2_between_its_limits_and_a_breakdown(n, m):
    """kappa = 3e7 (pivots of about 2^-50): FP64 Cholesky of C answers, and R comes from the fixed-point
    factorisation of the same C as TSQR's, 2^-99 / 2^-50 off.  A dependent column still breaks down
    or is answered by the passes."""
    import torch

    import paper_2603_20889_gb300 as q

    Xd = torch.from_numpy(np.ascontiguousarray(synth.conditioned(m, n, 3e7, seed=n).T)).cuda().T
    R, info = q.cholqr2_qless(Xd)
    Rt, _ = q.tsqr_qless(Xd)
    assert info.cpu().tolist() == [0, 0]
    assert row_error(R.cpu().numpy(), Rt.cpu().numpy()) <= 2.0 ** -46
    Xd[:, n - 1] = 0.0
    assert q.cholqr2_qless(Xd)[1].cpu().tolist() == [q.QL_ERR_NOT_SPD, n]
