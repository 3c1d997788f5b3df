"""The row-block passes of the projector's small bases (k <= 96, n <= 2048) at the
edges of their blocks and of their range, and the general path just beyond it,
through the ordered CholQR2: the same bounds as the CholQR2 kernel test."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


@pytest.mark.parametrize("n,k", [(31, 16), (32, 17), (33, 33), (65, 48), (97, 96), (1025, 80), (2047, 95),
                                 (2048, 96), (2049, 96), (300, 97)])
def test_single_precision_orthonormal_basis(g, n, k):
    import torch
    rng = np.random.default_rng(n + k)
    Y = rng.standard_normal((n, k)) * np.logspace(0, -2, k)[rng.permutation(k)]
    Y[:, k - 2] = 0.0
    rank = min(n, k - 1)
    Q = g.selftest_orth(torch.as_tensor(Y, device="cuda:0"), "fp32").cpu().numpy()
    eps = 1.2e-7
    norms = np.linalg.norm(Q, axis=0)
    live = norms > 0.5
    assert np.all(norms[~live] == 0.0) and live.sum() == rank
    Ql = Q[:, live]
    assert np.abs(Ql.T @ Ql - np.eye(rank)).max() <= 50 * eps * k
    assert np.abs(Y - Ql @ (Ql.T @ Y)).max() <= 1e3 * eps * np.abs(Y).max()
