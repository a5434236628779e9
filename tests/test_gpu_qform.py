"""Q = X R^-1 and the two-phase projection: values at the edges of the FP32 range, row counts
around the kernels' blocks, the smallest and the largest of their column classes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def col_major(X, ld):
    import torch

    m, n = X.shape
    buf = torch.zeros((n, ld), dtype=torch.float64 if X.dtype == np.float64 else torch.float32, device="cuda")
    buf[:, :m] = torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    return buf[:, :m].T


@pytest.mark.parametrize("n", [1, 8, 13, 33])
@pytest.mark.parametrize("m,ld", [(64, 64), (129, 131), (1000, 1000)])
def test_fp32_subnormals_keep_their_value(m, n, ld):
    """R = I: every product is by 1 or 0 and every sum with 0, so Q is X to the bit."""
    import torch

    import paper_2603_20889_gb300 as q

    X = np.random.default_rng(n).integers(1, 1 << 23, (m, n)).astype(np.float32) * np.float32(2.0 ** -149)
    X[::2] *= -1.0
    X[:, n // 2] = 1.5  # an ordinary column beside them
    Xd = col_major(X, ld)
    Q, info = q.q_from_r(Xd, torch.eye(n, dtype=torch.float64, device="cuda").T)
    assert info.cpu().tolist() == [0, 0]
    assert np.array_equal(Q.cpu().numpy().view(np.int32), X.view(np.int32))


@pytest.mark.parametrize("n", [1, 8, 16, 33, 64])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_few_rows_spread_over_the_sms(n, dtype):
    """Row counts on both sides of a block and of a warp per CTA.  Entries and products hold 48 bits
    (FP32 results 24), so |Q - X M| <= (n 2^-44 + u) |X| |M| with M = R^-1 in FP64."""
    import torch

    import paper_2603_20889_gb300 as q

    rng = np.random.default_rng(n)
    R = np.triu(rng.standard_normal((n, n)) / n) + 2.0 * np.eye(n)
    M = np.linalg.inv(R)
    u = 2.0 ** -24 if dtype == np.float32 else 2.0 ** -53
    for m, ld in ((1, 1), (63, 64), (65, 65), (1000, 1000), (9729, 9731), (30002, 30002)):
        X = rng.standard_normal((m, n)).astype(dtype)
        Q, info = q.q_from_r(col_major(X, ld), torch.from_numpy(np.ascontiguousarray(R.T)).cuda().T)
        assert info.cpu().tolist() == [0, 0]
        X = X.astype(np.float64)
        assert np.all(np.abs(Q.cpu().numpy() - X @ M) <= (n * 2.0 ** -44 + u) * (np.abs(X) @ np.abs(M))), m


@pytest.mark.parametrize("n,bad", [(1, 1), (8, 8), (40, 17)])
def test_first_zero_pivot_is_reported(n, bad):
    import torch

    import paper_2603_20889_gb300 as q

    R = np.eye(n)
    R[bad - 1:, bad - 1:] = 0.0
    Q, info = q.q_from_r(col_major(np.ones((200, n)), 200), torch.from_numpy(np.ascontiguousarray(R.T)).cuda().T)
    assert info.cpu().tolist() == [q.QL_ERR_NOT_SPD, bad] and bool(torch.isnan(Q).all())


@pytest.mark.parametrize("k,n", [(1, 1), (8, 9), (64, 3), (33, 64)])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_projection_of_few_rows(k, n, dtype):
    """Row counts on both sides of the tiles, out of place and in place.  W and C to 48-bit products
    and the storage's rounding: |C - Y^T X| and |W - (X - Y Y^T X)| <= 8 k (m 2^-47 + u) max|X|."""
    import torch

    import paper_2603_20889_gb300 as q

    rng = np.random.default_rng(k + n)
    u = 2.0 ** -24 if dtype == np.float32 else 2.0 ** -53
    for m, ld in ((k, k), (65, 65), (129, 131), (1000, 1000), (9729, 9730)):
        if m < k:
            continue
        Y = np.linalg.qr(rng.standard_normal((m, k)))[0].astype(dtype)
        X = rng.standard_normal((m, n)).astype(dtype)
        Yd, Xd = col_major(Y, ld), col_major(X, ld)
        W, C = q.project_out(Yd, Xd)
        Wi, Ci = q.project_out(Yd, Xd, W=Xd)
        assert torch.equal(W, Wi) and torch.equal(C, Ci)
        Y, X = Y.astype(np.float64), X.astype(np.float64)
        C0 = Y.T @ X
        W0 = X - Y @ C0
        C1 = Y.T @ W0  # Y is orthonormal to its storage's rounding only
        tol = 8 * k * (m * 2.0 ** -47 + u) * np.abs(X).max()
        assert np.abs(C.cpu().numpy() - (C0 + C1)).max() <= tol, m
        assert np.abs(W.cpu().numpy() - (W0 - Y @ C1)).max() <= tol, m
