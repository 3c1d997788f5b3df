"""The FP64 product at the edges of its tiles (8 x 8 and 16 x 16 outputs, K
chunks of 32 split over thread groups) against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 33), (7, 9, 31), (8, 8, 32), (9, 17, 65), (16, 4096, 256), (288, 48, 288),
                                   (560, 561, 40), (48, 48, 1000)])
def test_fp64_product(M, N, K):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    A, B = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    C = g.selftest_gemm(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"), "fp64").cpu().numpy()
    # K roundings of the running sum, each at most 2^-53 of sum |a||b|, in either product
    assert np.all(np.abs(C - A @ B) <= 2 * K * 2.0 ** -53 * (np.abs(A) @ np.abs(B)))
