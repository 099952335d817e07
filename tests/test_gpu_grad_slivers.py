"""Shape gradient on flat triangles (disjoint ones: no sums over corners) against
the derivative of cotangents and area in extended precision.

The unit normal of a triangle of aspect a carries a rounding error of about eps /
a, which no formula on the positions avoids.  Replayed in NumPy, the median error
over random triangles is 0.05 eps / a (obtuse) and 0.13 eps / a (needles) where
the area's derivative is a cross product with the normal, and 0.23 and 0.15 where
it is a difference of edges."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


def reference(x, D, P):
    """Gradient of sum_k cot_k D_k / 2 - A P / 3 by the corners, corner by corner
    from the two edges that leave it."""
    n = np.cross(x[1] - x[0], x[2] - x[0])
    s = np.sqrt((n * n).sum(-1))[:, None]
    n = n / s
    g = [np.zeros_like(x[0]) for _ in range(3)]
    for k in range(3):
        a, b = (k + 1) % 3, (k + 2) % 3
        u, w = x[a] - x[k], x[b] - x[k]
        cot, h = (u * w).sum(-1)[:, None] / s, D[k][:, None] / (2 * s)
        gu, gw = h * (w - cot * np.cross(w, n)), h * (u - cot * np.cross(n, u))
        g[a], g[b], g[k] = g[a] + gu, g[b] + gw, g[k] - gu - gw
    q = -P[:, None] / 6
    g1, g2 = q * np.cross(x[2] - x[0], n), q * np.cross(n, x[1] - x[0])
    return np.stack([g[0] - g1 - g2, g[1] + g1, g[2] + g2], 1)


@pytest.mark.parametrize("aspect", [1e-2, 1e-4, 1e-6])
@pytest.mark.parametrize("foot", [0.4, 1.0])   # obtuse; needle
def test_flat_triangles(aspect, foot):
    import torch
    import paper_2111_09039_gb300 as hs
    rng = np.random.default_rng(3)
    m, p = 5000, 20
    unit = lambda a: a / np.linalg.norm(a, axis=1)[:, None]
    x0, d = rng.standard_normal((m, 3)), unit(rng.standard_normal((m, 3)))
    q = unit(np.cross(d, rng.standard_normal((m, 3))))
    V = np.stack([x0, x0 + 0.01 * d, x0 + 0.01 * (foot * d + aspect * q)], 1)   # m x corner x 3
    F = np.arange(3 * m, dtype=np.int32).reshape(m, 3)
    E, lam, w = rng.standard_normal((3 * m, p)), rng.uniform(1, 50, p), rng.standard_normal(p)
    t = lambda a: torch.as_tensor(a, device="cuda")
    # eigenvectors as the solve returns them: column-major
    g = hs.eig_grad(hs.Context(0), t(V.reshape(-1, 3)), t(F), t(lam), t(np.ascontiguousarray(E.T)).t(), t(w))
    g = g.cpu().numpy().reshape(m, 3, 3)
    L = np.longdouble
    f, wl = E.reshape(m, 3, p).astype(L), (w * lam).astype(L)
    D = [((f[:, (k + 1) % 3] - f[:, (k + 2) % 3]) ** 2 * w.astype(L)).sum(-1) for k in range(3)]
    P = (f ** 2 * wl).sum((-1, -2))
    ref = reference([V[:, k].astype(L) for k in range(3)], D, P)
    err = np.abs(g - ref).max((1, 2)) / np.abs(ref).max((1, 2))
    assert np.median(err) <= (0.11 if foot < 1 else 0.2) * EPS / aspect
