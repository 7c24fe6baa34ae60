"""GPU: the Rayleigh-Ritz eigensolver of Davidson on its own, on matrices whose diagonal ends
with equal, infinite or NaN entries: its sort must stay a permutation (the indices it leaves
address shared memory), so a matrix that is not finite gives values, not a fault (NaN where
it holds a NaN), and leaves nothing behind for the next call.

Tolerance 1e-13 |G| for finite matrices: cyclic Jacobi in FP64 is backward stable, some 20
sweeps of at most 48 rows are off by ~1e-14."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eig():
    import torch
    assert torch.cuda.is_available()
    from paper_1312_2415_gb300 import binding
    return binding.test_small_eig


def check(eig, G):
    m = len(G)
    w, v = np.linalg.eigvalsh(G), eig(G, m)
    tol = 1e-13 * max(1.0, np.abs(w).max())
    assert np.abs(v[0] - w).max() <= tol
    assert np.abs(v[1] @ v[1].T - np.eye(m)).max() <= 1e-13
    assert np.abs(v[1] @ G - v[0][:, None] * v[1]).max() <= tol


@pytest.mark.parametrize("m", [1, 2, 3, 7, 8, 9, 16, 31, 32, 33, 48])
def test_not_finite_then_finite(eig, m):
    rng = np.random.default_rng(m)
    A = rng.normal(size=(m, m))
    A = A + A.T
    for bad in (np.nan, np.inf, -np.inf):
        for i, j in ((0, 0), (m - 1, m - 1), (m - 1, 0), (m // 2, m // 3)):
            G = A.copy()
            G[i, j] = G[j, i] = bad
            theta, C = eig(G, min(m, 3))
            assert not np.isnan(bad) or np.isnan(theta).all()
    theta, C = eig(np.full((m, m), np.nan), m)
    assert not np.isfinite(theta).any()
    check(eig, A)
    check(eig, np.diag(np.repeat([2.0, -1.0], [m // 2, m - m // 2])))  # equal values
    check(eig, np.zeros((m, m)))
