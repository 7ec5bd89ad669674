"""Solves with several right-hand sides (one Krylov iteration for all of them, decisions per
right-hand side) against single solves: columns that converge at different iterations, zero
columns, row counts that are no multiple of four, more right-hand sides than fit a block's share."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nb():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    from paper_2506_06190_gb300 import build
    build.build()
    import paper_2506_06190_gb300 as nb
    return nb


def _neumann(V, F, k, m):
    rng = np.random.default_rng(m)
    g = np.stack([S.monopole_neumann(V, F, k * (0.3 + 0.1 * i)) for i in range(m)])
    g[m // 2] = 0
    g[0] = rng.normal(size=g.shape[1]) + 1j * rng.normal(size=g.shape[1])
    return np.ascontiguousarray(g.T)


# Both end at true residuals of a few 1e-6 of ||b||, and ||L^-1|| ||L|| < 20 for these surfaces: the
# solutions agree to 2 x 4e-6 x 20 < 2e-4 of the column's norm.
@pytest.mark.parametrize("prec", ["tf32", "bf16", "fp16"])
@pytest.mark.parametrize("n_tri,m", [(20, 5), (302, 17), (1218, 64), (2434, 33), (514, 128)])
def test_columns_match_single_solves(nb, n_tri, m, prec):
    Vs, F = S.ring_sphere(n_tri)
    V = S.perturbed_ellipsoid(Vs, 9) if n_tri > 100 else Vs
    g = _neumann(V, F, 2.0, m)
    p = {"tf32": nb.PREC_MIXED_TF32, "bf16": nb.PREC_MIXED_BF16, "fp16": nb.PREC_MIXED_FP16}[prec]
    with nb.Operator.assemble(V, F, 2.0, nb.nat_bem_opts_default(prec=p)) as op:
        x, info, st = op.solve(g)
        assert st == nb.NAT_BEM_OK
        x = np.asarray(x)
        assert np.all(x[:, m // 2] == 0)
        for c in {0, 1, m // 2 + 1, m - 1}:
            y, _, st1 = op.solve(g[:, c].copy())
            assert st1 == nb.NAT_BEM_OK
            assert np.linalg.norm(x[:, c] - np.asarray(y).ravel()) < 2e-4 * np.linalg.norm(y)


def test_all_columns_zero(nb):
    V, F = S.ring_sphere(302)
    with nb.Operator.assemble(V, F, 1.0, nb.nat_bem_opts_default(prec=nb.PREC_MIXED_BF16)) as op:
        x, info, st = op.solve(np.zeros((op.n, 9), complex))
        assert st == nb.NAT_BEM_OK and np.all(np.asarray(x) == 0)


# The accurate products read a three-way split of R, then of L, from one buffer. Their errors are a
# few 1e-7 of a column, the solver stops at 1e-6 (floor 4e-6 for single precision): 5e-6 in all.
@pytest.mark.parametrize("m", [32, 33, 64, 65, 128])
def test_right_hand_sides_through_the_split_of_r(nb, m):
    Vs, F = S.ring_sphere(1218)
    V = S.perturbed_ellipsoid(Vs, 9)
    g = _neumann(V, F, 2.0, m)
    with nb.Operator.assemble(V, F, 2.0, nb.nat_bem_opts_default(prec=nb.PREC_MIXED_BF16)) as op:
        for k in (2.0, 1.5):  # the buffer holds the old L's split when the operator changes
            if k != 2.0:
                op.reassemble(k)
            L, R = op.rows(0, 0, op.n).astype(complex), op.rows(1, 0, op.n).astype(complex)
            for cols in (slice(0, m), slice(1, 9), slice(0, m)):  # 8 columns need only L's split
                h = np.ascontiguousarray(g[:, cols])
                x, info, st = op.solve(h)
                assert st == nb.NAT_BEM_OK
                b = R @ h
                res = np.linalg.norm(L @ np.asarray(x) - b, axis=0)
                assert np.max(res - 5e-6 * np.linalg.norm(b, axis=0)) <= 0


def test_fewer_right_hand_sides_after_many(nb):
    """A workspace made for many right-hand sides (n nrhs above 2^20: a larger grid for the Arnoldi
    step) gives fewer of them the bits of a fresh one."""
    Vs, F = S.ring_sphere(5174)
    V = S.perturbed_ellipsoid(Vs, 72)
    rng = np.random.default_rng(73)
    g = (rng.normal(size=(len(F), 208)) + 1j * rng.normal(size=(len(F), 208))).astype(np.complex64)
    few = np.asfortranarray(g[:, :64])
    opts = nb.nat_bem_opts_default(max_iter=80)
    with nb.Operator.assemble(V, F, 2.0, opts) as op:
        fresh, a, _ = op.solve(few)
    with nb.Operator.assemble(V, F, 2.0, opts) as op:
        op.solve(np.asfortranarray(g))
        x, b, st = op.solve(few)
    assert st == nb.NAT_BEM_OK and a.iterations == b.iterations and np.array_equal(x, fresh)
