"""Axis permutations at the sizes where the tiled kernel takes over (2^21 elements)
and at ragged tiles, against torch: whole numbers, exact in every kind."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("shape,order", [
    ((57, 5, 5, 5, 5, 58), (0, 5, 2, 4, 1, 3)),          # just below the line
    ((61, 5, 5, 5, 5, 63), (0, 5, 2, 4, 1, 3)),          # odd bonds, just above it
    ((4, 4, 101, 4, 4, 103), (2, 5, 1, 4, 0, 3)),
    ((97, 3, 3, 3, 3, 331), (5, 0, 1, 2, 3, 4)),
    ((97, 3, 3, 3, 3, 331), (1, 2, 3, 4, 5, 0)),
    ((1447, 1453), (1, 0)),                              # prime sides: no divisor to split off
    ((1536, 1536), (1, 0)),
    ((2, 1100003), (1, 0)),
    ((8, 8, 8, 8, 8, 8, 8), (6, 0, 2, 4, 1, 3, 5)),
    ((2100001,), (0,)),
])
def test_permutation(g, shape, order, kind):
    import torch
    n = 1
    for d in shape:
        n *= d
    x = (torch.arange(n, dtype=torch.float64, device="cuda:0") * 7919 % 16777213).reshape(shape)
    assert torch.equal(g.selftest_permute(x, order, kind), x.permute(order).contiguous())
