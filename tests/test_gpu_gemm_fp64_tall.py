"""The FP64 product with more row tiles than a grid has along y."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(16 * 65535 + 1, 3, 2), (1200000, 8, 8), (3, 16 * 65535 + 1, 2)])
def test_tall_and_wide_products(M, N, K):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    gen = torch.Generator(device="cuda:0").manual_seed(M)
    A, B = (torch.randint(-8, 9, s, device="cuda:0", generator=gen).double() for s in ((M, K), (K, N)))
    assert torch.equal(g.selftest_gemm(A, B, "fp64"), sum(A[:, k, None] * B[k] for k in range(K)))   # whole numbers
