"""FP64 solve of a mesh with two vertices drawn far out: their masses and
stiffnesses stand out in the lowest columns of M Psi and S Psi (1000 times the
mean), so that some tiles of the reduced matrices go to the FP64 kernel and
others to the digits.  Against the oracle."""
import dataclasses

import numpy as np
import pytest

import synth
from oracle import sim

pytestmark = pytest.mark.gpu


def test_matches_oracle():
    import torch
    import paper_2111_09039_gb300 as hs
    mesh = synth.bumpy_torus(48, 40, 17)
    V = mesh.V.copy()
    V[100] *= 6
    V[777] *= 5
    mesh = dataclasses.replace(mesh, V=V)
    p, tol, start = 60, 1e-10, 7     # 90 columns: two by two tiles
    ctx = hs.Context(0)
    hier = hs.Hierarchy(ctx, mesh.F, V=mesh.V, p=p, levels=2, start_vertex=start)
    S, M = hs.assemble(ctx, hier, V=torch.as_tensor(mesh.V, device="cuda:0"))
    lam, Phi, info = hs.solve(ctx, hier, S, M, p, tol)
    ref = sim.hsim(mesh, p, 2, tol, start)
    got = lam.cpu().numpy()
    assert np.max(np.abs(got - ref.lam[:p]) / np.maximum(np.abs(ref.lam[:p]), ref.lam[1])) < 1e-9
    assert info["max_residual"] < tol
    # M-orthonormal to the rounding of sums of this length
    X, m = Phi.cpu().numpy(), M.cpu().numpy()
    assert np.abs(X.T @ (m[:, None] * X) - np.eye(p)).max() < 1e-10
