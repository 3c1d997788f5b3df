"""The FP64 refinement of a single-precision SVD on matrices of low rank with a tail
at rounding level, as the Rayleigh-Ritz matrices of product-like states are: the
tail's directions are arbitrary, but the factors stay bounded and the singular
values exact to FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def low_rank(k, seed):
    rng = np.random.default_rng(1000 * k + seed)
    rng.standard_normal((3, k, k))
    u, v = (np.linalg.qr(rng.standard_normal((k, k)))[0] for _ in range(2))
    return u[:, :5] @ np.diag([1, 0.3, 0.1, 1e-3, 1e-4]) @ v[:5] + 1e-16 * rng.standard_normal((k, k))


@pytest.mark.parametrize("k,seeds", [(80, range(4)), (112, range(8, 12)), (160, range(6, 12))])
def test_low_rank_with_a_tail(k, seeds):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    for seed in seeds:
        X = low_rank(k, seed)
        S, L, Q = (t.cpu().numpy() for t in g.selftest_svd_refined(torch.as_tensor(X, device="cuda:0")))
        # columns of orthonormal matrices, the tail's to a first approximation only
        assert np.abs(L).max() < 2 and np.abs(Q).max() < 2
        # k roundings of 2^-53 in products of unit columns, three of them
        assert np.abs(np.sort(np.abs(S))[::-1] - np.linalg.svd(X, compute_uv=False)).max() <= 3 * k * 2.0 ** -53
