"""The FP32-accurate tensor-core product (operands split into TF32 parts,
partial sums of at most 32 terms added in FP32) against FP64, at the edges of
its tiles (128 rows, up to 160 columns, 32 values of K), for both layouts of A
and with K split over CTAs."""
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


def _bound(K):
    """Relative to sum |a||b|: the remainder's truncation to TF32 (2^-23 per
    operand) and the dropped product of remainders (2^-24); four truncated
    additions per 32 terms (2^-23 each); K / 32 FP32 additions (2^-24 each, plus
    up to 16 of the K split)."""
    return (2.5 + 4.0 + 0.5 * (K / 32 + 16)) * 2.0 ** -23


SHAPES = [(128, 160, 32), (4, 1, 4), (132, 17, 36), (124, 159, 28), (256, 161, 100), (260, 321, 8), (1024, 80, 1024),
          (132, 16, 4100), (1300, 40, 64), (640, 640, 4)]


@pytest.mark.parametrize("colmajor", [False, True])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_product_against_fp64(g, M, N, K, colmajor):
    import torch
    rng = np.random.default_rng(M + 7 * N + 31 * K)
    A = rng.standard_normal((M, K)) * np.exp(rng.uniform(-6, 6, (M, 1)))
    B = rng.standard_normal((K, N)) * np.exp(rng.uniform(-6, 6, (1, N)))
    A, B = A.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    C = g.selftest_gemm3x(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"), colmajor).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= _bound(K) * (np.abs(A) @ np.abs(B)))


def test_same_sign_sums_keep_fp32_accuracy(g):
    """All products positive: the tensor core's truncation would shrink a long
    sum by ~3e-8 per instruction; sums of 32 terms keep it below 3e-7."""
    import torch
    rng = np.random.default_rng(5)
    A = rng.uniform(0.5, 1.0, (128, 4096)).astype(np.float32).astype(np.float64)
    B = rng.uniform(0.5, 1.0, (4096, 64)).astype(np.float32).astype(np.float64)
    C = g.selftest_gemm3x(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0")).cpu().numpy()
    assert abs(np.mean(C / (A @ B) - 1.0)) <= 4 * 2.0 ** -23


def test_nan_and_infinity_come_through(g):
    """A non-finite operand makes its row or column non-finite and no other."""
    import torch
    A = np.ones((128, 64))
    B = np.ones((64, 32))
    A[3, 5], A[7, 0], B[9, 11] = np.nan, np.inf, -np.inf
    C = g.selftest_gemm3x(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0")).cpu().numpy()
    bad = np.zeros((128, 32), bool)
    bad[3], bad[7], bad[:, 11] = True, True, True
    assert np.array_equal(~np.isfinite(C), bad)
    assert np.all(C[~bad] == 64.0)


@pytest.mark.parametrize("M,N,K,colmajor", [(8, 8, 6, False), (6, 8, 8, True)])
def test_unaligned_rows_are_refused(g, M, N, K, colmajor):
    import torch
    with pytest.raises(g.KhError) as e:
        g.selftest_gemm3x(torch.ones((M, K), dtype=torch.float64, device="cuda:0"),
                          torch.ones((K, N), dtype=torch.float64, device="cuda:0"), colmajor)
    assert e.value.status == g.KH_EINVAL
