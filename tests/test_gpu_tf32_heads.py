"""Operand splits at the upper end of FP32: values that would round up to infinity as
TF32 stay finite, as in products of the unsplit values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MAX = float(np.finfo(np.float32).max)


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


@pytest.mark.parametrize("colmajor", [False, True])
def test_product_of_the_largest_values(g, colmajor):
    A, B = np.ones((128, 64)), np.full((64, 32), 2.0 ** -20)
    A[3, 5], A[4, 6], A[5, 7] = MAX, -MAX, MAX * (1 - 2.0 ** -11)
    B[9, 11], B[5, 4] = MAX * 2.0 ** -9, 0.0
    C = g.selftest_gemm3x(_t(A), _t(B), colmajor).cpu().numpy()
    assert np.all(np.abs(C - A @ B) <= 2e-6 * (np.abs(A) @ B))


@pytest.mark.parametrize("shape,order", [((64, 32), (1, 0)), ((1024, 2048), (1, 0))])
def test_split_permutation_of_the_largest_values(g, shape, order):
    x = np.ones(shape)
    x[3, 5], x[4, 6], x[8, 1] = MAX, -MAX, np.nan
    y = g.selftest_permute(_t(x), order, 2).cpu().numpy()
    assert np.array_equal(y, x.transpose(order), equal_nan=True)


def test_layered_contraction_of_large_values(g):
    """D = 6 rounds heads to nearest: the largest value against sites of 1e-6."""
    D, nb = 6, 5
    rng = np.random.default_rng(1)
    T = 1e-6 * rng.uniform(0.5, 1.0, (2, D, D, D, D))
    Y = rng.uniform(0.5, 1.0, (nb, D * D, D * D))
    Y[2, 3, 4] = MAX
    out = g.selftest_site_layered(_t(T), _t(Y), npass=3).cpu().numpy()
    TL = T.transpose(1, 2, 0, 3, 4).reshape(D * D, 2, D * D)
    want = np.einsum("bji,ipo,jpq->boq", Y, TL, TL, optimize=True)
    assert np.all(np.abs(out - want) <= 1e-5 * want)
