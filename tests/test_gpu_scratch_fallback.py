"""FP64 products where the device has no room for the digits' scratch: the FP64
kernel, which needs none, answers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["gram", "gemm_update"])
def test_no_room_for_digits(op):
    import torch
    import paper_2111_09039_gb300 as hs
    torch.cuda.empty_cache()
    rng = np.random.default_rng(0)
    n, k = 150000, 96
    A = rng.standard_normal((n, k))
    B = A[:, ::-1].copy() if op == "gram" else rng.standard_normal((k, k))
    call = getattr(hs, op)
    d = lambda a: torch.as_tensor(a, device="cuda")
    dA, dB = d(A), d(B)
    ctx = hs.Context(0)
    before = hs.kernel_launches()
    ref = call(ctx, dA, dB)
    digits = hs.kernel_launches() - before
    assert digits > 5
    del ctx                                   # gives its scratch back
    spare = torch.empty(3 * n * k, dtype=torch.float64, device="cuda")   # room for the result
    ctx = hs.Context(0)
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    rest = torch.empty(free - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        del spare
        before = hs.kernel_launches()
        got = call(ctx, dA, dB)
        assert hs.kernel_launches() - before < digits
    finally:
        del rest
        torch.cuda.empty_cache()
    # both within n 2^-53 sum|a||b| of the exact result
    mag = (np.abs(A).T @ np.abs(B)) if op == "gram" else np.abs(A) @ np.abs(B)
    assert np.all(np.abs((got - ref).cpu().numpy()) <= 2.0 * (n if op == "gram" else k) * 2.0 ** -53 * mag)
