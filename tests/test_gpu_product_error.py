"""A tensor-core product that gave up is reported on its own context, once, and on
no other one."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("op", ["gram", "gram_tc", "gemm_update", "gemm_update_tc"])
def test_own_context_only(op):
    import torch
    import paper_2111_09039_gb300 as hs
    a, b = hs.Context(0), hs.Context(0)
    rng = np.random.default_rng(0)
    d = lambda *s: torch.as_tensor(rng.standard_normal(s), device="cuda")
    A, B = d(2048, 200), d(2048, 200) if op.startswith("gram") else d(200, 70)
    call = getattr(hs, op)
    ref = call(a, A, B)
    assert hs.lib().hsim_check_product_error(a.handle) == 0
    torch.testing.assert_close(call(b, A, B), ref, rtol=0, atol=1e-9)
    with pytest.raises(hs.HsimError) as e:
        call(a, A, B)
    assert e.value.name == "HSIM_E_INTERNAL"
    torch.testing.assert_close(call(a, A, B), ref, rtol=0, atol=1e-9)
