"""Kernels of the bond update at the sizes where their dispatch changes: the cost
and its gradient (<T'|N|T'>, the normal equations with eight threads an entry
below D = 6 and one from there on, the gradient), and the ALS that runs on them,
with its solve in shared memory and (D = 6) in global memory, against the oracle
on the library's own metric."""
import numpy as np
import pytest

import kh_inputs
from oracle import bond, model, peps

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


def _t(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda:0")


def _state(g, A, B, D, **cfg):
    J, K = model.couplings(0.3 * np.pi)
    gt = model.gate("x", 0.01, J, K)
    ctx = g.Context(D, 8, "fp64", **cfg)
    ctx.set_state(_t(A), _t(B))
    return ctx, gt, peps.composite(A, B, "x", gt)


@pytest.mark.parametrize("D", [1, 2, 3, 5, 6])
def test_cost_and_gradient_on_the_same_metric(g, D):
    """Every number is a nest of sums with at most D^2 + 4 D^2 + 2 D^3 + D^4 / 4 <
    1000 roundings on either side, so 2000 u of the sum of absolute values
    bounds the difference; T' carries 16 more."""
    ctx, gt, Tp = _state(g, *kh_inputs.random_site_tensors(D, 31 + D), D)
    rng = np.random.default_rng(D)
    A2, B2 = (rng.standard_normal((2, 2, D, D, D)) for _ in range(2))
    gA, gB, d, c = ctx.cost_gradient(0, gt, _t(A2), _t(B2), ctm_max_sweeps=2, ctm_tol=-1.0)
    N = ctx.ctm_metric(0).cpu().numpy()
    ctx.close()
    gA_ref, gB_ref = bond.cost_gradient(A2, B2, Tp, N)
    d_ref, c_ref = bond.cost(A2, B2, Tp, N)
    a, b, t, n = (np.abs(x) for x in (A2, B2, Tp, N))
    gA_abs, gB_abs = bond.cost_gradient(a, b, -t, n)              # every term positive
    d_abs, c_abs = bond.cost(a, b, -t, n)
    tol = 2100 * U
    assert np.all(np.abs(gA.cpu().numpy() - gA_ref) <= tol * gA_abs)
    assert np.all(np.abs(gB.cpu().numpy() - gB_ref) <= tol * gB_abs)
    assert abs(c - c_ref) <= tol * c_abs
    assert abs(d - d_ref) <= tol * d_abs


@pytest.mark.parametrize("D", [2, 4, 5, 6])
def test_als_cost_after_three_sweeps(g, D):
    """Three ALS sweeps from the truncated SVD of T' reach the oracle's cost.  The
    library's start comes from single precision (1e-5 in the factors), which the
    sweeps contract: 1e-4 of the cost."""
    ctx, gt, Tp = _state(g, *kh_inputs.perturbed_product_state(D, 51 + D, 0.3), D, als_max_iter=3, als_tol=0.0)
    out = ctx.eefu_apply_gate(0, gt, ctm_max_sweeps=10, ctm_tol=-1.0)
    N = ctx.ctm_metric(0).cpu().numpy()
    ctx.close()
    _, _, info = bond.als(Tp, N, D, tol=0.0, max_iter=3)
    assert out["als_iters"] == 3
    assert abs(out["rel_cost"] - info["rel_cost"]) <= 1e-4 * info["rel_cost"] + 1e-13
