"""The FP64 Gram and basis update on seven BF16 digits (the form that large
hsim_gram and hsim_gemm_update calls take), at the edges of its tiles, K
ranges and dispatch, and the inputs that it hands to the FP64 kernels."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def hs():
    import paper_2111_09039_gb300
    return paper_2111_09039_gb300


@pytest.fixture(scope="module")
def ctx(hs):
    return hs.Context(0)


def dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def exact(A, B):
    return (A.astype(np.longdouble).T @ B.astype(np.longdouble)).astype(np.float64)


# an FP64 sum of n terms in any order is within n EPS sum|a||b| of the exact
# one; the digits are within 2^-54 max|a| max|b| per term
def bound(A, B):
    n = A.shape[0]
    return n * (2.0 ** -54 * np.abs(A).max(0)[:, None] * np.abs(B).max(0)[None, :]) + 4 * EPS * (np.abs(A).T @ np.abs(B))


@pytest.mark.parametrize("n,ka,kb", [(1023, 30, 30), (1024, 30, 30), (1025, 23, 64), (4099, 65, 129), (16384, 63, 1),
                                     (32773, 128, 33)])
def test_gram(hs, ctx, n, ka, kb):
    rng = np.random.default_rng(n)
    A, B = rng.standard_normal((n, ka)), rng.standard_normal((n, kb)) * 10.0 ** rng.uniform(-8, 8, (1, kb))
    G = hs.gram(ctx, dev(A), dev(B)).cpu().numpy()
    assert np.all(np.abs(G - exact(A, B)) <= bound(A, B))


@pytest.mark.parametrize("n,k,m", [(1, 41, 50000), (127, 130, 130), (1024, 48, 63), (4097, 41, 65), (70003, 17, 31),
                                   (2049, 300, 7)])
def test_update(hs, ctx, n, k, m):
    rng = np.random.default_rng(n + k)
    s = 10.0 ** rng.uniform(-9, 9, k)   # unequal columns of A against rows of B
    A, B = rng.standard_normal((n, k)) * s, rng.standard_normal((k, m)) / s[:, None]
    C = hs.gemm_update(ctx, dev(A), dev(B)).cpu().numpy()
    rows = rng.choice(n, min(n, 40), replace=False)
    cols = rng.choice(m, min(m, 40), replace=False)
    X, Y = (A[rows] / s).T, s[:, None] * B[:, cols]
    # column k and row k meet at a power of two of s: factors below 2 on each side
    assert np.all(np.abs(C[np.ix_(rows, cols)] - exact(X, Y)) <= 8 * bound(X, Y))


def test_strided_rows(hs, ctx):
    rng = np.random.default_rng(5)
    A, B = rng.standard_normal((3001, 101)), rng.standard_normal((3001, 77))
    G = hs.gram(ctx, dev(A)[:, 3:90], dev(B)[:, 1:]).cpu().numpy()
    assert np.all(np.abs(G - exact(A[:, 3:90], B[:, 1:])) <= bound(A[:, 3:90], B[:, 1:]))
    C = hs.gemm_update(ctx, dev(A)[:, 3:80], dev(B)[5:82, 1:]).cpu().numpy()
    assert np.all(np.abs(C - exact(A[:, 3:80].T, B[5:82, 1:])) <= 8 * bound(A[:, 3:80].T, B[5:82, 1:]))


def test_standing_out_entry(hs, ctx):
    """One entry 1e12 above the rest of its column must not cost the others' bits."""
    rng = np.random.default_rng(6)
    n = 5000
    A, B = rng.standard_normal((n, 40)), rng.standard_normal((n, 40))
    A[17, 3], B[17, :] = 1e12, 0.0
    G = hs.gram(ctx, dev(A), dev(B)).cpu().numpy()
    ref = exact(A, B)
    assert np.all(np.abs(G - ref) <= n * EPS * (np.abs(A).T @ np.abs(B)))


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite(hs, ctx, bad):
    rng = np.random.default_rng(7)
    A, B = rng.standard_normal((2000, 60)), rng.standard_normal((2000, 50))
    A[100, 7] = bad
    B[100, 5] = 0.0
    G = hs.gram(ctx, dev(A), dev(B)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = A.T @ B
    assert np.array_equal(np.isnan(G), np.isnan(ref)) and np.array_equal(np.isinf(G), np.isinf(ref))
    ok = np.isfinite(ref)
    np.testing.assert_allclose(G[ok], ref[ok], rtol=0, atol=1e-10)
    B2 = rng.standard_normal((60, 50))
    B2[7, 5] = 0.0
    C = hs.gemm_update(ctx, dev(A), dev(B2)).cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = A @ B2
    assert np.array_equal(np.isnan(C), np.isnan(ref)) and np.array_equal(np.isinf(C), np.isinf(ref))


def test_zero_columns_and_subnormals(hs, ctx):
    rng = np.random.default_rng(8)
    A, B = rng.standard_normal((3000, 50)), rng.standard_normal((3000, 50))
    A[:, 4] = 0.0
    B[:, 9] = 0.0
    A[:, 11] *= 2.0 ** -1060      # subnormal entries
    B[:, 12] *= 2.0 ** 900
    G = hs.gram(ctx, dev(A), dev(B)).cpu().numpy()
    ref = exact(A, B)
    assert np.all(G[4] == 0.0) and np.all(G[:, 9] == 0.0)
    assert np.all(np.abs(G - ref) <= bound(A, B) + 3000 * 2.0 ** -1074 * np.abs(B).max(0))
