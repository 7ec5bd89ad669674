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
