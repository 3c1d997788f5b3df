"""Kernels of the projector in the forms in which it calls them: the SVD asked for its
largest triplets only, the refinement of single-precision factors in place, and
the row-block passes that warm-start a small basis and join a split product."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
K24 = 2.0 ** -24


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1906_02220_gb300 as pkg
    return pkg


def _t(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda:0")


def _matrix(kind, k):
    rng = np.random.default_rng(k)
    X = rng.standard_normal((k, k))
    if kind == "graded":
        q, r = (np.linalg.qr(rng.standard_normal((k, k)))[0] for _ in range(2))
        X = q @ np.diag(10.0 ** -np.linspace(0, 10, k)) @ r
    elif kind == "low rank":
        X = X[:, :7] @ rng.standard_normal((7, k)) + 1e-17 * rng.standard_normal((k, k))
    return X


@pytest.mark.parametrize("kind", ["full", "graded", "low rank"])
@pytest.mark.parametrize("k,n_top", [(16, 5), (17, 8), (48, 24), (64, 24), (65, 64), (96, 1), (112, 40), (112, 112)])
def test_largest_triplets(g, k, n_top, kind):
    """Columns below the n_top largest may stay coupled to each other, so the sum of
    their couplings, not the top triplets, is what is left open.  Backward stable
    to some 10 k roundings."""
    X = _matrix(kind, k)
    S, L, Q = (t.cpu().numpy() for t in g.selftest_svd_top(_t(X), n_top))
    ref = np.linalg.svd(X, compute_uv=False)
    tol = 20 * k * U
    assert np.all(np.diff(S) <= 0)
    assert np.abs(S[:n_top] - ref[:n_top]).max() <= tol * ref[0]
    assert np.abs(Q.T @ Q - np.eye(k)).max() <= tol
    assert np.abs(X @ Q - L * S).max() <= tol * ref[0]
    top = S[:n_top] > 1e-13 * S[0]
    Lt = L[:, :n_top][:, top]
    assert np.abs(Lt.T @ Lt - np.eye(top.sum())).max() <= tol


@pytest.mark.parametrize("k", [5, 16, 33, 80, 112, 160])
def test_refinement_in_place_is_the_same(g, k):
    """The same FP64 factors, rounded once to FP32."""
    X = _matrix("full", k)
    S, L, Q = (t.cpu().numpy() for t in g.selftest_svd_refined(_t(X)))
    s, l, q = (t.cpu().numpy() for t in g.selftest_svd_refined_in_place(_t(X)))
    assert np.array_equal(s, S)
    assert np.array_equal(l, L.astype(np.float32)) and np.array_equal(q, Q.astype(np.float32))


@pytest.mark.parametrize("n,k,dead", [(31, 16, [0]), (33, 17, [3, 16]), (300, 48, list(range(20, 48))), (1024, 80, [79]),
                                      (2048, 96, list(range(0, 96, 3))), (441, 65, []), (100, 33, list(range(33)))])
def test_warm_basis(g, n, k, dead):
    """Live columns stay as they are; the random ones have entries below one and are
    orthogonal to the live ones to FP32 rounding of sums over k and n."""
    rng = np.random.default_rng(n)
    V = np.linalg.qr(rng.standard_normal((n, k)))[0].astype(np.float32).astype(np.float64)
    live = np.ones(k)
    live[dead] = 0.0
    out = g.selftest_warm_basis(_t(V), _t(live)).cpu().numpy()
    on = live > 0
    assert np.array_equal(out[:, on], V[:, on])
    R = out[:, ~on]
    if len(dead):
        norms = np.linalg.norm(R, axis=0)
        assert np.all(norms > 0.1) and np.abs(R).max() < 2
        assert np.linalg.matrix_rank(R) == min(len(dead), n - int(on.sum()))
        if on.any():
            assert np.abs(V[:, on].T @ R).max() <= 4 * k * K24 * norms.max()


@pytest.mark.parametrize("n,k,parts", [(31, 16, 1), (33, 33, 2), (1024, 80, 8), (2048, 96, 24), (441, 65, 3)])
def test_joined_parts(g, n, k, parts):
    rng = np.random.default_rng(parts)
    P = rng.standard_normal((parts, n, k)).astype(np.float32)
    want = np.zeros((n, k), np.float32)
    for p in P:
        want = want + p
    Y, G = (t.cpu().numpy() for t in g.selftest_join_parts(_t(P)))
    assert np.array_equal(Y, want)
    # FP32 sums over 16 rows
    assert np.all(np.abs(G - Y.T @ Y) <= 17 * K24 * (np.abs(Y).T @ np.abs(Y)))
