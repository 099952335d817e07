"""Mixed-path Ritz solves on both sides of the order up to which its products
are FP64 ones (256), at the edges of their tiles (16 rows, 8 columns, 128 terms
per stage), with a reduced mass near I (Newton-Schulz) and away from it (factor,
whose inversion takes tiles of 16, 32 and 64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


SMALL = [3, 8, 9, 16, 17, 65, 127, 128, 129, 255, 256]


@pytest.mark.parametrize("k,near", [(k, True) for k in SMALL] + [(k, False) for k in SMALL + [257, 700]])
def test_ritz(k, near):
    import torch
    import paper_2111_09039_gb300 as hs
    rng = np.random.default_rng(k)
    Q, _ = np.linalg.qr(rng.standard_normal((k, k)))
    w = np.linspace(0.9, 1.1, k) if near else np.geomspace(0.01, 1.0, k)
    M = Q @ np.diag(w) @ Q.T
    if near:  # rows of |M - I| sum to at most 0.4
        E = M - np.eye(k)
        M = np.eye(k) + E * min(1.0, 0.4 / np.abs(E).sum(1).max())
    A = rng.standard_normal((k, k))
    S = A @ A.T / k
    M, S = 0.5 * (M + M.T), 0.5 * (S + S.T)
    d = lambda a: torch.as_tensor(a, device="cuda")
    lam, X, _ = hs.ritz(hs.Context(0), d(S), d(M), tc=True)
    lam, X = lam.cpu().numpy(), X.cpu().numpy()
    cond = 1.0 if near else 100.0
    # backward errors of k eps each of the reduction, the eigensolver and the
    # back transformation, times the condition of M
    tol = 16 * max(k, 16) * EPS * cond
    nS = np.linalg.norm(S, 2)
    assert np.abs(X.T @ M @ X - np.eye(k)).max() <= tol
    assert np.abs(S @ X - M @ X * lam[None, :]).max() <= tol * nS * np.sqrt(cond)
