"""S X at the widths where the kernel changes (32, 64, 96, 128 columns), with
columns that start off a 16-byte boundary, against the same sums in order."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 31, 32, 33, 64, 65, 96, 97, 127, 128, 129, 160, 193, 225, 256, 300])
@pytest.mark.parametrize("off", [0, 1, 2])
def test_widths(k, off):
    import torch
    import paper_2111_09039_gb300 as hs
    rng = np.random.default_rng(k)
    A = sp.random(517, 403, density=0.02, random_state=rng, format="csr")
    A.data = rng.standard_normal(A.nnz)
    X = rng.standard_normal((403, k + off))
    d = lambda a: torch.as_tensor(a, device="cuda")
    Y = hs.spmm(hs.Context(0), d(A.indptr.astype(np.int32)), d(A.indices.astype(np.int32)), d(A.data), d(X)[:, off:],
                n_cols=403).cpu().numpy()
    # FP64 sums of at most 32 products in the same order: a rounding each
    bound = 34 * 2.0 ** -53 * (abs(A) @ np.abs(X[:, off:]))
    assert np.all(np.abs(Y - A @ X[:, off:]) <= bound)
