"""The layered site contraction over several tiles per CTA with odd and even
numbers of chunks: the two worker sets take chunks in turn across tiles, so an
odd number exchanges their roles from tile to tile."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (npass, D, p, blocks per tile): 3 or 4 tiles on each of 152 CTAs and a ragged last one
CASES = [(3, 1, 16, 128), (3, 2, 16, 32), (3, 4, 11, 8), (3, 4, 16, 8), (3, 3, 5, 14), (3, 5, 5, 5), (16, 4, 3, 8),
         (16, 2, 16, 32), (1, 3, 16, 14)]


@pytest.mark.parametrize("npass,D,p,bt", CASES)
def test_chunks_over_tiles(npass, D, p, bt):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as g
    nb = bt * 500 + 1
    rng = np.random.default_rng(31 * D + p)
    T = rng.standard_normal((p, D, D, D, D))
    Y = rng.standard_normal((nb, D * D, D * D))
    out = g.selftest_site_layered(torch.as_tensor(T, device="cuda:0"), torch.as_tensor(Y, device="cuda:0"), npass=npass)
    TL = np.ascontiguousarray(T.transpose(1, 2, 0, 3, 4)).reshape(D * D, p, D * D)

    def contract(TL, Y):
        Z = np.einsum("ipo,bji->bjpo", TL, Y, optimize=True).reshape(nb, D * D * p, D * D)
        return np.matmul(Z.transpose(0, 2, 1), TL.reshape(D * D * p, D * D))

    ref, scale = contract(TL, Y), contract(np.abs(TL), np.abs(Y))
    # FP32-level with 3 passes; 2^-11 per rounded factor in TF32; Y, T and Z rounded to 8 bits in BF16
    assert np.all(np.abs(out.cpu().numpy() - ref) <= {3: 1e-5, 1: 3e-3, 16: 8e-3}[npass] * scale)
