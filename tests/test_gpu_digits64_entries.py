"""Every entry of the FP64 Gram and basis update against the sum of its terms'
magnitudes, on inputs whose maxima say nothing about the other entries (entries
that stand out, graded and disjoint columns), and the update's shapes at the
edges of its tiles and row ranges on the digits.  A call on the digits launches
more than the one kernel of the FP64 form; every test asks."""
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


def on_digits(hs, call):
    before = hs.kernel_launches()
    out = call().cpu().numpy()
    assert hs.kernel_launches() - before > 5, "not on the digits"
    return out


def check(got, X, Y):
    """X, Y: K rows.  FP64 arithmetic in any order: K EPS sum|x||y|, and the
    digits are given entries whose error stays within 64 EPS of it."""
    K = X.shape[0]
    with np.errstate(over="ignore"):
        ref = (X.astype(np.longdouble).T @ Y.astype(np.longdouble))
        mag = np.abs(X).T @ np.abs(Y)
    assert np.all(np.abs(got - ref) <= (max(K, 64) + 1) * EPS * mag)


@pytest.mark.parametrize("side", ["A", "B"])
@pytest.mark.parametrize("x", [1.0, 1e6, 1e12, 1e20, 1e40, 1e200])
def test_update_outlier(hs, ctx, x, side):
    rng = np.random.default_rng(1)
    A, B = rng.standard_normal((400, 200)), rng.standard_normal((200, 200))
    (A if side == "A" else B)[37, 11] = x
    check(on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B))), A.T, B)


@pytest.mark.parametrize("x", [2.0 ** 20, 2.0 ** 60])
def test_update_outlier_row(hs, ctx, x):
    """A whole row of B that stands out and meets a zero of A."""
    rng = np.random.default_rng(2)
    A, B = rng.standard_normal((2000, 200)), rng.standard_normal((200, 10))
    B[0], A[0, 0] = x, 0.0
    check(on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B))), A.T, B)


@pytest.mark.parametrize("off", [0.0, 1e-6, 1e-3, 0.3])
def test_update_near_identity(hs, ctx, off):
    rng = np.random.default_rng(3)
    k = 300
    A = rng.standard_normal((1000, k)) * 10.0 ** rng.uniform(-3, 3, (1000, k))
    B = np.eye(k) + off / np.sqrt(k) * rng.standard_normal((k, k))
    check(on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B))), A.T, B)


@pytest.mark.parametrize("grade", [1e-3, 1e-10, 1e-20])
@pytest.mark.parametrize("alternate", [False, True])
def test_gram_graded(hs, ctx, grade, alternate):
    rng = np.random.default_rng(4)
    n = 4096
    A, B = rng.standard_normal((n, 70)), rng.standard_normal((n, 66))
    small = np.arange(n) % 2 == 1 if alternate else np.arange(n) >= n // 2
    A[small, 3] *= grade          # graded ...
    B[~small, 5] = 0.0            # ... against one that lives on the small half
    check(on_digits(hs, lambda: hs.gram(ctx, dev(A), dev(B))), A, B)


def test_gram_disjoint_and_sparse(hs, ctx):
    rng = np.random.default_rng(5)
    n = 6000
    A, B = rng.standard_normal((n, 80)), rng.standard_normal((n, 80))
    A[n // 2:, 7], B[:n // 2, 9] = 1e-300, 1e-300   # nearly disjoint
    A[:, 70], A[17, 70] = 0.0, 3.0                  # one entry, off the sampled rows
    check(on_digits(hs, lambda: hs.gram(ctx, dev(A), dev(B))), A, B)


@pytest.mark.parametrize("n", [1025, 40001])
def test_gram_outlier(hs, ctx, n):
    rng = np.random.default_rng(6)
    A, B = rng.standard_normal((n, 65)), rng.standard_normal((n, 129))
    A[n - 1, 64], B[0, 128] = 1e15, -1e30
    check(on_digits(hs, lambda: hs.gram(ctx, dev(A), dev(B))), A, B)


@pytest.mark.parametrize("n,k", [(1024, 33), (20000, 70)])
def test_gram_of_one_block(hs, ctx, n, k):
    """Both operands the same buffer: exponents and sums are taken once."""
    A = np.random.default_rng(n).standard_normal((n, k))
    A[n // 3, k // 2] = 1e9
    dA = dev(A)
    check(on_digits(hs, lambda: hs.gram(ctx, dA, dA)), A, A)


@pytest.mark.parametrize("low", [120, 96, 1])
@pytest.mark.parametrize("n", [1024, 4096])
def test_gram_full_digits(hs, ctx, n, low):
    """Every digit of both factors positive and up to its full size, 127: the digit
    sums from D = 4 on pass 2^24 and their partial sums are odd."""
    rng = np.random.default_rng(low)

    def block(k):
        T = np.zeros((n, k), dtype=object)
        for s in range(7):
            T = T * 256 + rng.integers(low, 128, (n, k)).astype(object)
        return np.array([[float(t) for t in row] for row in T]) * 2.0 ** -55   # 53 of the 55 bits

    A, B = block(40), block(33)
    check(on_digits(hs, lambda: hs.gram(ctx, dev(A), dev(B))), A, B)


# one row, tiles of 128 and 64 and their remainders, K steps of 16, two row ranges
# (16 k bytes of digits to a row, 1 GiB to a range)
SHAPES = [(1, 200, 20000), (127, 170, 130), (129, 177, 129), (1024, 165, 63), (4097, 200, 65), (70003, 41, 63),
          (2049, 300, 7), (16500, 4096, 1)]


@pytest.mark.parametrize("n,k,m", SHAPES)
def test_update_shapes(hs, ctx, n, k, m):
    rng = np.random.default_rng(n + k)
    s = 10.0 ** rng.uniform(-9, 9, k)   # unequal columns of A against rows of B
    A, B = rng.standard_normal((n, k)) * s, rng.standard_normal((k, m)) / s[:, None]
    C = on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B)))
    rows = np.unique(np.concatenate([rng.choice(n, min(n, 40), replace=False), [0, n - 1]]))
    cols = np.unique(np.concatenate([rng.choice(m, min(m, 40), replace=False), [0, m - 1]]))
    check(C[np.ix_(rows, cols)], A[rows].T, B[:, cols])


@pytest.mark.parametrize("start,pitch", [(0, 0), (1, 3), (3, 4), (2, 2)])
def test_update_strided(hs, ctx, start, pitch):
    rng = np.random.default_rng(7)
    A, B = rng.standard_normal((3001, 190 + pitch)), rng.standard_normal((200, 76 + pitch))
    a, b = slice(start, start + 180), slice(start, start + 70)
    C = on_digits(hs, lambda: hs.gemm_update(ctx, dev(A)[:, a], dev(B)[5:185, b]))
    check(C, A[:, a].T, B[5:185, b])


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("where", [(100, 7), (1999, 199)])
def test_update_nonfinite(hs, ctx, bad, where):
    rng = np.random.default_rng(8)
    A, B = rng.standard_normal((2000, 200)), rng.standard_normal((200, 130))
    A[where] = bad
    B[where[1], 5] = 0.0
    C = on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B)))
    with np.errstate(invalid="ignore"):
        ref = A @ B
    assert np.array_equal(np.isnan(C), np.isnan(ref)) and np.array_equal(np.isinf(C), np.isinf(ref))
    keep = np.arange(2000) != where[0]
    check(C[keep], A[keep].T, B)


def test_zero_rows_and_columns(hs, ctx):
    rng = np.random.default_rng(9)
    A, B = rng.standard_normal((2000, 200)), rng.standard_normal((200, 130))
    A[5], A[:, 9], B[7], B[:, 3] = 0.0, 0.0, 0.0, 0.0
    A[11] *= 2.0 ** -1050               # subnormal entries
    C = on_digits(hs, lambda: hs.gemm_update(ctx, dev(A), dev(B)))
    assert np.all(C[5] == 0.0) and np.all(C[:, 3] == 0.0)
    keep = np.arange(2000) != 11
    check(C[keep], A[keep].T, B)
    assert np.abs(C[11] - (A[11].astype(np.longdouble) @ B)).max() <= 200 * 2.0 ** -1074 * np.abs(B).max()
