"""Eigenvectors of a batch at a loose tolerance against tight FP64 solves of the
same meshes: the angle of every vector to the eigenvectors of its group of close
eigenvalues is within residual over distance to the rest of the spectrum (the
Davis-Kahan bound), for groups from the single vector up."""
import numpy as np
import pytest
import scipy.sparse as sp

import synth
from oracle.assembly import lumped_mass, stiffness

pytestmark = pytest.mark.gpu
P, EXTRA, TOL = 24, 8, 1e-5


def test_angles_within_residual_over_gap():
    import torch
    import paper_2111_09039_gb300 as hs
    ctx = hs.Context(0)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda:0")
    # nu : nv as the radii and little noise: pairs of eigenvalues 1e-4 apart
    items = [synth.bumpy_torus(129, 39, s) for s in (3, 5)] + [m for m, _ in synth.batch(count=3, seed=4, lo=1500, hi=6000)]
    hiers, S, M = [], [], []
    for mesh in items:
        h = hs.Hierarchy(ctx, mesh.F, V=mesh.V, p=P, levels=2, start_vertex=1, precision=hs.HSIM_MIXED)
        s, m = hs.assemble(ctx, h, V=dev(mesh.V))
        hiers.append(h), S.append(s), M.append(m)
    out = hs.solve_batched(ctx, hiers, S, M, P, TOL, options=hs.default_options(precision=hs.HSIM_MIXED, levels=2))
    for mesh, (lam, Phi, _) in zip(items, out):
        lam, Phi = lam.cpu().numpy(), Phi.cpu().numpy()
        K, m = stiffness(mesh), lumped_mass(mesh)
        h = hs.Hierarchy(ctx, mesh.F, V=mesh.V, p=P + EXTRA, levels=2, start_vertex=1)
        s, md = hs.assemble(ctx, h, V=dev(mesh.V))
        ref, Q, _ = hs.solve(ctx, h, s, md, P + EXTRA, 1e-10)
        ref, Q = ref.cpu().numpy(), Q.cpu().numpy()
        R = K @ Phi - (m[:, None] * Phi) * lam
        res = np.sqrt((R * R / m[:, None]).sum(0))     # ||(S - lambda M) phi|| in the norm of M^-1
        cos = Q.T @ (m[:, None] * Phi)
        for i in range(P):
            assert abs(lam[i] - ref[i]) <= res[i] + 1e-9 * ref[-1]
            for width in (0.0, 1e-3, 1e-2, 1e-1):
                group = np.abs(ref - ref[i]) <= width * max(ref[i], ref[1])
                if group[-1]:
                    continue                            # its other end is not known
                dist = np.abs(ref[~group] - lam[i]).min()
                part = Phi[:, i] - Q[:, group] @ cos[group, i]
                angle = np.sqrt((m * part * part).sum())
                # the reference carries its own residual of 1e-10 over the same distance
                assert angle <= 1.01 * res[i] / dist + 1e-9 * ref[-1] / dist + 1e-9, (i, width)
