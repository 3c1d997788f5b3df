"""The environment metric on either side of its dispatch: the last product on the
tensor cores (1e9 flops or more, chi^2 a multiple of 4) and on the CUDA cores,
against the oracle's contraction of the library's own environment."""
import numpy as np
import pytest

import kh_inputs
from oracle import ctmrg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


@pytest.mark.parametrize("D,chi,prec", [(5, 34, "tf32x3"), (5, 36, "tf32x3"), (5, 37, "tf32x3"), (5, 38, "bf16"),
                                        (6, 18, "tf32x3"), (5, 36, "fp32")])
def test_metric_of_the_librarys_environment(g, D, chi, prec):
    """Six operands rounded to FP32 and six products, the longest of chi^2 terms:
    at most (2.5 + 4 + (K / 32 + 16) / 2) 2^-23 of the sum of absolute values each
    on the tensor cores, K 2^-24 on the CUDA cores, so (180 + chi^2 / 2) 2^-23 of the
    metric of absolute values bounds the whole."""
    import torch
    A, B = kh_inputs.random_site_tensors(D, 7)
    ctx = g.Context(D, chi, prec)
    a, b = torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0")
    ctx.set_state(a, b)
    ctx.cost_gradient(2, np.eye(4), a, b, ctm_max_sweeps=2, ctm_min_sweeps=2, ctm_tol=-1.0)
    C, E = (t.cpu().numpy() for t in ctx.ctm_get_env(2))
    N = ctx.ctm_metric(2).cpu().numpy()
    ctx.close()
    E = E.reshape(4, chi, D * D, chi)
    ref = ctmrg.metric(ctmrg.Env(list(C), list(E)), D)
    bound = ctmrg.metric(ctmrg.Env(list(np.abs(C)), list(np.abs(E))), D)
    assert np.all(np.abs(N - ref) <= (180 + chi * chi / 2) * 2.0 ** -23 * bound)
