"""A solve that fits only without the scratch that a context kept from an earlier
call: it is given back, whichever context holds it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("other", [False, True])
def test_solve_takes_kept_scratch(other):
    import torch
    import paper_2111_09039_gb300 as hs
    torch.cuda.empty_cache()
    mesh, p = synth.bumpy_torus(250, 160, 5), 40
    V = torch.as_tensor(mesh.V, device="cuda")
    ctx = hs.Context(0)

    def prepared():
        h = hs.Hierarchy(ctx, mesh.F, V=mesh.V, p=p, levels=2, start_vertex=1, precision=hs.HSIM_MIXED)
        return (h,) + hs.assemble(ctx, h, V=V)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def solve(h, S, M):
        return hs.solve(ctx, h, S, M, p, 1e-5)[0].cpu().numpy()

    first, second = prepared(), prepared()
    solve(*prepared())             # torch's blocks for the results, module loading
    before = free()
    ref = solve(*first)
    need = before - free()
    assert need > 128 << 20
    holder = hs.Context(0) if other else ctx
    A = torch.randn(163842, 300, dtype=torch.float64, device="cuda")
    hs.gram(holder, A, A)
    del A
    torch.cuda.empty_cache()
    a = free()
    rest = torch.empty(a - (need - (64 << 20)), dtype=torch.uint8, device="cuda")
    try:
        got = solve(*second)
    finally:
        del rest
        torch.cuda.empty_cache()
    np.testing.assert_allclose(got, ref, rtol=1e-6, atol=1e-6)
