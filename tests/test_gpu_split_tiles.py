"""Grams of tall blocks, whose columns are split several tiles of 32 rows per
block of threads: row counts around a tile and around the sizes where the number
of tiles per block changes, odd column counts, pitches and starts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 33, 1000, 38911, 38913, 77857, 155713, 311425])
@pytest.mark.parametrize("k,pitch,off", [(65, 65, 0), (64, 66, 0), (63, 66, 1), (130, 132, 2)])
@pytest.mark.parametrize("digits", [5, 6])
def test_gram(n, k, pitch, off, digits):
    import torch
    import paper_2111_09039_gb300 as hs
    rng = np.random.default_rng(n + k)
    A = torch.as_tensor(rng.standard_normal((n, pitch)), device="cuda")[:, off:off + k]
    B = torch.as_tensor(rng.standard_normal((n, pitch)), device="cuda")[:, off:off + k]
    G = hs.gram_tc(hs.Context(0), A, B, digits=digits).cpu().numpy()
    a, b = A.cpu().numpy(), B.cpu().numpy()
    # a digit operand is within 2^-(8 digits - 1) of its column's maximum; both
    # operands and the digit pairs left out: four such terms per product
    bound = n * 2.0 ** (3 - 8 * digits) * np.abs(a).max(0)[:, None] * np.abs(b).max(0)[None, :]
    ref = a.T @ b
    assert np.all(np.abs(G - ref) <= bound + 4 * n * 2.0 ** -53 * (np.abs(a).T @ np.abs(b)))
