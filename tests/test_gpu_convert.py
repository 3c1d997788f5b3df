"""The FP64 <-> FP32 conversions in integer arithmetic against the hardware's:
every value is the same, subnormal operands among them; subnormal results, which
are rounded twice, within one unit of their last place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_conversions_are_ieee():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    rng = np.random.default_rng(0)
    with np.errstate(over="ignore"):
        x = np.concatenate([
            rng.standard_normal(4000) * np.exp2(rng.uniform(-160, 140, 4000)),         # through both ends of FP32
            rng.standard_normal(2000) * np.exp2(rng.uniform(-151, -124, 2000)),        # subnormal results
            np.exp2(np.arange(-152.0, 130.0)), 1.5 * np.exp2(np.arange(-152.0, 130.0)),
            (1 + 2.0 ** -24) * np.exp2(np.arange(-150.0, 128.0)),                      # ties of normal results
            (1 + 3 * 2.0 ** -24) * np.exp2(np.arange(-150.0, 128.0)),
            [0.0, np.inf, np.nan, 2.0 ** 128 - 2.0 ** 103, 2.0 ** 128 - 2.0 ** 104, 2.0 ** -1074, 2.0 ** -149,
             2.0 ** -150, 1.0000001 * 2.0 ** -150, 2.0 ** -126 - 2.0 ** -151]])
        x = np.concatenate([x, -x])
        want = x.astype(np.float32).astype(np.float64)
    for got in g.selftest_convert(torch.as_tensor(x, device="cuda:0")):
        got = got.cpu().numpy()
        ok = ~np.isnan(want)
        assert np.array_equal(np.isnan(got), ~ok)
        normal = ok & ~(np.abs(want) < 2.0 ** -126)
        assert np.array_equal(got[normal], want[normal])
        low = ok & ~normal
        assert np.all(np.abs(got[low] - want[low]) <= 2.0 ** -149)
        assert np.array_equal(np.signbit(got[ok]), np.signbit(want[ok]))
