"""Dense Ritz solves of matrices whose columns nearly vanish below the diagonal
(entries of 1e-150 and 1e-160, whose squares leave the FP64 range) and of whole
matrices far from 1, at the sizes of both tridiagonalisation kernels' rows."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


def _solve(S):
    import torch
    import paper_2111_09039_gb300 as hs
    d = lambda a: torch.as_tensor(a, device="cuda")
    lam, X, _ = hs.ritz(hs.Context(0), d(S), d(np.eye(len(S))))
    return lam.cpu().numpy(), X.cpu().numpy()


def _check(S):
    n, norm = len(S), np.abs(S).max()
    lam, X = _solve(S)
    # numpy on the matrix scaled near 1 (an exact power of two)
    e = np.frexp(norm)[1]
    ref = np.linalg.eigvalsh(np.ldexp(S, -e))
    tol = 4 * max(n, 16) * EPS  # a backward stable solve
    assert np.all(np.isfinite(lam)) and np.all(np.isfinite(X))
    assert np.abs(np.ldexp(lam, -e) - ref).max() <= tol * max(1.0, np.abs(ref).max())
    assert np.abs(X.T @ X - np.eye(n)).max() <= max(tol, 1e-11)
    assert np.abs(np.ldexp(S, -e) @ X - X * np.ldexp(lam, -e)).max() <= tol * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("norm", [1e-8, 1.0, 1e10])
@pytest.mark.parametrize("tiny", [1e-115, 1e-130, 1e-140, 1e-150, 1e-160])
@pytest.mark.parametrize("n", [3, 40, 300])
def test_tiny_couplings(n, tiny, norm):
    rng = np.random.default_rng(n)
    E = rng.uniform(0.5, 1.0, (n, n)) * tiny
    S = np.diag(norm * np.linspace(1.0, 2.0, n)) + np.tril(E, -1) + np.tril(E, -1).T
    _check(S)


@pytest.mark.parametrize("tiny", [1e-149, 1e-154])
def test_block_then_tiny(tiny):
    """An ordinary leading block, tiny couplings to and within the rest."""
    rng = np.random.default_rng(1)
    n, h = 96, 40
    A = rng.standard_normal((n, n)) * tiny
    A[:h, :h] = 1e9 * rng.standard_normal((h, h))
    S = np.tril(A, -1) + np.tril(A, -1).T + np.diag(1e10 * np.linspace(-1.0, 1.0, n))
    _check(S)


@pytest.mark.parametrize("scale", [1e-290, 1e-155, 1e-120, 1e120, 1e150, 1e290])
def test_scales(scale):
    rng = np.random.default_rng(2)
    A = rng.standard_normal((75, 75))
    _check((A + A.T) * scale)
