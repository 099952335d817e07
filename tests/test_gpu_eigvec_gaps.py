"""Eigenvectors of dense symmetric matrices: pairs and triples of eigenvalues at
relative gaps on both sides of the cluster tolerance, and the sizes where the
back transformation changes (blocks of eight reflectors; 128 rows per thread
step; one or two buffers; a few vectors per block of threads)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


def _check(S, ev):
    import torch
    import paper_2111_09039_gb300 as hs
    n = len(ev)
    d = lambda a: torch.as_tensor(a, device="cuda")
    lam, X, _ = hs.ritz(hs.Context(0), d(S), d(np.eye(n)))
    lam, X = lam.cpu().numpy(), X.cpu().numpy()
    # a backward stable solve: n eps ||S|| with a modest factor
    tol = 4 * max(n, 16) * EPS
    norm = np.abs(ev).max()
    assert np.abs(lam - np.sort(ev)).max() <= tol * norm
    assert np.abs(X.T @ X - np.eye(n)).max() <= max(tol, 1e-11)
    assert np.abs(S @ X - X * lam[None, :]).max() <= tol * norm


@pytest.mark.parametrize("gap", [1e-3, 2e-5, 1e-6, 1e-8, 2e-9, 5e-10, 1e-12, 1e-15])
@pytest.mark.parametrize("dense", [True, False])
def test_gaps(gap, dense):
    n = 120
    rng = np.random.default_rng(11)
    ev = np.linspace(-1.0, 1.0, n)
    ev[21] = ev[20] + gap
    ev[51], ev[52] = ev[50] + gap, ev[50] + 2.5 * gap
    ev[80:90] = ev[80] + gap * np.arange(10)
    if dense:
        Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
        S = Q @ np.diag(ev) @ Q.T
        S = 0.5 * (S + S.T)
    else:
        S = np.diag(rng.permutation(ev))
    _check(S, ev)


@pytest.mark.parametrize("n", [2, 3, 8, 9, 10, 17, 128, 129, 153, 305, 384, 385, 769, 1025, 1280, 1537, 1610, 2048, 2049])
def test_sizes(n):
    rng = np.random.default_rng(n)
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    ev = np.sort(rng.uniform(-3.0, 5.0, n))
    S = Q @ np.diag(ev) @ Q.T
    _check(0.5 * (S + S.T), ev)
