"""Entries of the collocation operators' pairs without a common vertex, against the FP64 oracle:
meshes far from the origin (centroids split on a coarse grid), ragged column blocks, small and
large wavenumbers."""
import numpy as np
import pytest

import synthetic as S
from oracle import assemble

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    from paper_2506_06190_gb300 import build
    build.build()
    import paper_2506_06190_gb300 as nb
    return nb


# Row norms of the error: each of the seven points rounds r (three units of 2^-24 with the
# reciprocal square root, cubed in L: nine), the factors (about ten) and the phase (k r a unit and
# sin and cos four, over |e^{i phase}| = 1), and |D|^2's share is common to the points.
@pytest.mark.parametrize("shift", [0.0, 30.0])
@pytest.mark.parametrize("n_tri,k", [(8, 1.0), (254, 0.05), (258, 4.0), (514, 20.0), (1026, 6.0)])
def test_regular_entries(nb, n_tri, k, shift):
    Vs, F = S.ring_sphere(n_tri)
    V = (S.perturbed_ellipsoid(Vs, 5) if n_tri > 100 else Vs) + shift
    L, R = assemble(V, F, k)
    size = float(np.linalg.norm(V.max(0) - V.min(0)))
    tol = 2.0 ** -24 * (24 + 2 * k * size)
    with nb.Operator.assemble(V, F, k) as op:
        for which, ref in ((0, L), (1, R)):
            got = op.rows(which, 0, op.n)
            far = ~(F[:, None, :, None] == F[None, :, None, :]).any((2, 3))
            err = np.linalg.norm(np.where(far, got - ref, 0), axis=1)
            assert np.max(err / np.linalg.norm(ref, axis=1)) < tol


def _slab(m, gap):
    """Unit square plate of m x m cells, `gap` cells thick, its two sheets triangulated differently."""
    rng = np.random.default_rng(17)
    x, y = np.meshgrid(np.arange(m + 1) / m, np.arange(m + 1) / m, indexing="ij")
    top = np.stack([x, y, np.full_like(x, gap / m)], -1)
    bot = np.stack([x, y, np.zeros_like(x)], -1)
    bot[1:-1, 1:-1, :2] += rng.uniform(-0.3, 0.3, (m - 1, m - 1, 2)) / m
    n = (m + 1) ** 2
    at = lambda i, j: i * (m + 1) + j
    F = []
    for i in range(m):
        for j in range(m):
            a, b, c, d = at(i, j), at(i + 1, j), at(i + 1, j + 1), at(i, j + 1)
            F += [(a, b, c), (a, c, d), (n + a, n + d, n + b), (n + b, n + d, n + c)]
    ring = [at(i, 0) for i in range(m)] + [at(m, j) for j in range(m)] + [at(i, m) for i in range(m, 0, -1)] + [
        at(0, j) for j in range(m, 0, -1)]
    for a, b in zip(ring, ring[1:] + ring[:1]):
        F += [(b, a, n + a), (b, n + a, n + b)]
    return np.concatenate([top.reshape(-1, 3), bot.reshape(-1, 3)]), np.array(F, np.int32)


# Collocation points close to the quadrature points of triangles they share no vertex with. d = D - q
# is formed from parts of 0.4 of a cell rounded at 2^-24, so d is off by 2^-24 x 0.4 / gap of itself
# and L (1/r^3 and two projections) by a few times that: below the 1e-5 of the other rows down to
# 0.02 of a cell, 12 x 2^-24 / gap beyond.
@pytest.mark.parametrize("gap", [0.3, 0.1, 0.05, 0.02, 1e-3, 1e-4])
def test_thin_plate_entries(nb, gap):
    V, F = _slab(11, gap)
    k = 2.0
    L, R = assemble(V, F, k)
    far = ~(F[:, None, :, None] == F[None, :, None, :]).any((2, 3))
    with nb.Operator.assemble(V, F, k) as op:
        for which, ref in ((0, L), (1, R)):
            got = op.rows(which, 0, op.n)
            assert np.isfinite(got[far]).all()
            err = np.linalg.norm(np.where(far, got - ref, 0), axis=1)
            assert np.max(err / np.linalg.norm(ref, axis=1)) < (1e-5 if gap >= 0.02 else 12 * 2.0 ** -24 / gap)
