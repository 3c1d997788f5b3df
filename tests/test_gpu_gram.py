"""Gram matrices of FP32 blocks: FP32 sums over 16 rows, FP64 sums of those, at the
edges of its tiles and row ranges and in its symmetric and general form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

K24 = 2.0 ** -24


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


def _t(x):
    import torch
    return torch.as_tensor(x, device="cuda:0")


@pytest.mark.parametrize("pair", [False, True])
def test_sums_beyond_16_rows_are_fp64(g, pair):
    """Sums of 16 rows of 2^48, 2^24 and three ones in one range of rows: exact in
    FP64, while neither one FP32 number nor the sum of two holds the result."""
    n, k = 10000, 16                       # ranges of 80 rows
    A = np.zeros((n, k))
    A[0], A[16] = 2.0 ** 24, 2.0 ** 12
    A[[32, 48, 64]] = 1.0
    G = g.selftest_gram(_t(A), _t(A) if pair else None).cpu().numpy()
    assert np.all(G == 2.0 ** 48 + 2.0 ** 24 + 3)


@pytest.mark.parametrize("n,k", [(1, 1), (17, 3), (33, 48), (100, 49), (1024, 80), (5184, 160), (5000, 97)])
def test_gram_against_fp64(g, n, k):
    rng = np.random.default_rng(n + k)
    A, B = (rng.standard_normal((n, k)).astype(np.float32).astype(np.float64) for _ in range(2))
    for X, got in ((A, g.selftest_gram(_t(A))), (B, g.selftest_gram(_t(A), _t(B)))):
        # 16 roundings of FP32 sums; the FP64 ones are far below
        assert np.all(np.abs(got.cpu().numpy() - A.T @ X) <= 17 * K24 * (np.abs(A).T @ np.abs(X)))
