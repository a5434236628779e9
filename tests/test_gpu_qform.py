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
