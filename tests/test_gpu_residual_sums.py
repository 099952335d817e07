"""The residual that a solve reports against the definition in FP64 on the
returned pairs: column counts around a block of 32, and both row block sizes
(64 rows, 256 from n ceil(p / 32) of 311,296 on)."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import assembly, sim
from synth import meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu,nv,p,levels", [(60, 41, 31, 2), (60, 41, 32, 2), (60, 41, 33, 2),
                                            (97, 83, 65, 2), (250, 160, 230, 2)])
@pytest.mark.parametrize("mixed", [True, False])
def test_reported_residual(nu, nv, p, levels, mixed):
    import torch
    import paper_2111_09039_gb300 as hs
    if not mixed and p > 100:
        pytest.skip("the FP64 path takes the same kernel at the smaller sizes")
    mesh = meshes.bumpy_torus(nu, nv, 5)
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    ctx = hs.Context(0)
    o = hs.default_options()
    o.levels = levels
    o.precision = hs.HSIM_MIXED if mixed else hs.HSIM_FP64
    hier = hs.Hierarchy(ctx, mesh.F, V=mesh.V, p=p, options=o)
    S, M = hs.assemble(ctx, hier, V=d(mesh.V))
    lam, Phi, info = hs.solve(ctx, hier, S, M, p, 1e-4, o)
    m = assembly.lumped_mass(mesh)
    res = sim.residuals(assembly.stiffness(mesh), sp.diags(m), Phi.cpu().numpy(), lam.cpu().numpy(), 1.0 / m)
    # mixed: values truncated to 24 bits (2^-23 each, three factors), sums of
    # 48 terms at most in FP32 before FP64: 3e-6 of the square at the most;
    # FP64: rounding of S Phi against a residual of 1e-5 and more
    rtol = 1e-5 if mixed else 1e-8
    assert abs(info["max_residual"] - res.max()) <= rtol * res.max()
