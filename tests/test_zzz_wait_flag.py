"""A tensor-core wait that ran out is reported by every call that hands out or
stores results, before anything else that the unfinished buffers may show.  The
flag is set from the host, as a kernel that gave up would set it.  Collected after
the other library tests."""
import numpy as np
import pytest

import kh_inputs

pytestmark = pytest.mark.gpu


def _context(g, nan=False):
    import torch
    A, B = kh_inputs.perturbed_product_state(2, seed=3, eps=0.05)
    ctx = g.Context(2, 16, "tf32x3", als_max_iter=8)
    ctx.set_state(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"))
    for slot in range(6):
        ctx.ctm_build_composite(slot, slot % 3)
        ctx.ctm_sweep(slot, 2)
    if nan:
        A = A.copy()
        A[0, 0, 0, 0, 0] = np.nan
        ctx.set_state(torch.as_tensor(A, device="cuda:0"), torch.as_tensor(B, device="cuda:0"))
    return ctx


def _calls(g, ctx, path):
    import torch
    gate = g.gate(g.bond_hamiltonian(0, 0.3, 0.7), 0.01)
    A2, B2 = (torch.full((2, 2, 2, 2, 2), 0.3, dtype=torch.float64, device="cuda:0") for _ in range(2))
    return dict(
        env=lambda: ctx.ctm_get_env(0), projectors=lambda: ctx.ctm_projectors(0, 1), metric=lambda: ctx.ctm_metric(0),
        kappa=lambda: ctx.ctm_kappa(0), expval=lambda: ctx.ctm_expval(0, np.eye(16)),
        xi=lambda: ctx.ctm_correlation_length(0, max_iter=8), plaquette=lambda: ctx.flux(0),
        sweep=lambda: ctx.ctm_sweep(0, 2, 1, 0.5), gate=lambda: ctx.eefu_apply_gate(0, gate, 2, 2, -1.0),
        gradient=lambda: ctx.cost_gradient(0, gate, A2, B2, ctm_max_sweeps=0),
        observables=lambda: ctx.observables([np.eye(4)] * 3, ctm_max_sweeps=2, ctm_tol=-1.0),
        save=lambda: ctx.save(path))


CALLS = ("env", "projectors", "metric", "kappa", "expval", "xi", "plaquette", "sweep", "gate", "gradient", "observables",
         "save")


@pytest.mark.parametrize("name,nan", [(n, False) for n in CALLS] + [("gate", True), ("xi", True)])
def test_a_timed_out_wait_is_reported(name, nan, tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    ctx = _context(g, nan)
    if nan and name == "xi":
        ctx.ctm_build_composite(0, 0)
    call = _calls(g, ctx, str(tmp_path / "state.ckpt"))[name]
    assert g.lib().kh_selftest_wait_flag(ctx._ctx, 64) == g.KH_OK
    with pytest.raises(g.KhError) as e:
        call()
    assert e.value.status == g.KH_ETIMEOUT
    assert not (tmp_path / "state.ckpt").exists()
    assert g.lib().kh_selftest_wait_flag(ctx._ctx, 0) == g.KH_OK
    if not nan:
        call()
    ctx.close()
