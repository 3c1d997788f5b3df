"""The FP32-accurate tensor-core product with several tiles of a deep K on each
CTA, where the operand rings run full while a finished tile is stored.  One
operand holds the number of its block of 32 values, so that a value of another
block shows: every product and sum is a whole number of 1/32 and exact."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("colmajor", [False, True])
@pytest.mark.parametrize("coded", ["A", "B"])
@pytest.mark.parametrize("M,N,K", [(4096, 4096, 4096), (6000, 4000, 160)])
def test_no_value_of_another_block(M, N, K, coded, colmajor):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    block = torch.arange(K, dtype=torch.float64, device="cuda:0") // 32 + 1
    A = torch.ones((M, K), dtype=torch.float64, device="cuda:0")
    B = torch.ones((K, N), dtype=torch.float64, device="cuda:0")
    if coded == "A":
        A *= block[None, :] / 32
    else:
        B *= block[:, None] / 32
    C = g.selftest_gemm3x(A, B, colmajor)
    assert bool((C == float(block.sum()) / 32).all())
