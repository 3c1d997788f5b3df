"""The FP32-accurate tensor-core product with A column-major and K of any residue,
as the corners and the absorption call it (K = chi): the last step of eight values
then runs past K, where the tensor maps fill in zeros.  And one environment whose
chi is odd, against FP64."""
import numpy as np
import pytest

import kh_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


@pytest.mark.parametrize("M,N,K", [(128, 160, 1), (132, 17, 2), (4, 1, 3), (256, 161, 30), (1200, 1200, 75), (260, 321, 131),
                                   (132, 17, 4099), (128, 16, 4097), (136, 48, 4102)])
def test_any_k_with_a_column_major(g, M, N, K):
    """Bound relative to sum |a||b|: the remainders' truncation to TF32 (2^-23 per
    operand) and the dropped product of remainders (2^-22, each at most 2^-11);
    four truncated additions per 32 terms (2^-23 each); K / 32 FP32 additions
    (2^-24 each, plus up to 16 of the K split)."""
    import torch
    rng = np.random.default_rng(M + 7 * N + 31 * K)
    A = rng.standard_normal((M, K)) * np.exp(rng.uniform(-6, 6, (M, 1)))
    B = rng.standard_normal((K, N)) * np.exp(rng.uniform(-6, 6, (1, N)))
    A, B = A.astype(np.float32).astype(np.float64), B.astype(np.float32).astype(np.float64)
    C = g.selftest_gemm3x(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"), True).cpu().numpy()
    tol = (4.0 + 4.0 + 0.5 * (K / 32 + 16)) * 2.0 ** -23
    assert np.all(np.abs(C - A @ B) <= tol * (np.abs(A) @ np.abs(B)))


def test_environment_with_odd_chi(g):
    """D = 6, chi = 75: the corners' and absorptions' products have K = 75 on the
    tensor cores.  Expectation values agree with the FP64 kind's, which keeps the
    same directions, to FP32 accuracy."""
    import torch
    A, B = kh_inputs.perturbed_product_state(6, seed=5, eps=0.02)
    rng = np.random.default_rng(7)
    ops = rng.standard_normal((4, 16, 16))
    vals = []
    for prec in ("tf32x3", "fp64"):
        ctx = g.Context(6, 75, prec, svd_cut=1e-4, proj_fp64=1, n_slots=1)
        ctx.set_state(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"))
        ctx.ctm_build_composite(0, 0)
        ctx.ctm_sweep(0, 4)
        vals.append(ctx.ctm_expval(0, ops))
        ctx.close()
    assert np.all(np.abs(vals[0] - vals[1]) <= 2e-5 * np.abs(vals[1]).max())
