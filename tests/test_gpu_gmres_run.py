"""Whole GMRES runs in one launch (one right-hand side) against the two-launch iteration and the
FP64 oracle, at the sizes where the split over blocks, warps and stages has edges: fewer rows
than blocks, one row per block, ragged column ranges, the largest sizes the launch takes and the
first ones beyond it."""
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


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


# Both forms end with true residuals of at most a few 1e-6 of ||b|| (the solver's own criterion and
# its residual floor of 4 tol); for these second-kind systems ||L^-1|| ||L|| stays below 20 at the
# wavenumbers used, so the solutions agree to 2 x 4e-6 x 20 < 2e-4; in practice to rounding.
@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("n_tri", [8, 20, 152, 302, 1218, 2434, 5174, 10242, 12290])
def test_run_kernel_matches_two_launch_iteration(nb, monkeypatch, n_tri, prec):
    Vs, F = S.ring_sphere(n_tri)
    V = S.perturbed_ellipsoid(Vs, 31) if n_tri >= 302 else Vs
    k = 0.7 if n_tri < 302 else 3.0
    g = S.monopole_neumann(V, F, k)
    p = {"fp32": nb.PREC_FP32, "bf16": nb.PREC_MIXED_BF16, "fp16": nb.PREC_MIXED_FP16}[prec]
    out = []
    for off in (False, True):
        if off:
            monkeypatch.setenv("NATBEM_NO_RUN_KERNEL", "1")
        with nb.Operator.assemble(V, F, k, nb.nat_bem_opts_default(prec=p)) as op:
            x, info, st = op.solve(g)
            assert st == nb.NAT_BEM_OK
            out.append((x, info.iterations))
    assert abs(out[0][1] - out[1][1]) <= 3
    assert _rel(out[0][0], out[1][0]) < 2e-4


@pytest.mark.parametrize("restart", [3, 17])
def test_run_kernel_restarted_cycles(nb, monkeypatch, restart):
    Vs, F = S.ring_sphere(1500)
    V = S.perturbed_ellipsoid(Vs, 32)
    g = S.monopole_neumann(V, F, 2.0)
    out = []
    for off in (False, True):
        if off:
            monkeypatch.setenv("NATBEM_NO_RUN_KERNEL", "1")
        with nb.Operator.assemble(V, F, 2.0, nb.nat_bem_opts_default(restart=restart)) as op:
            x, info, st = op.solve(g)
            assert st == nb.NAT_BEM_OK and info.refinements >= 2
            out.append(x)
    assert _rel(out[0], out[1]) < 2e-4


def test_run_kernel_second_orthogonalisation_pass(nb):
    """Samples that carry little area make L = I/2 plus a small part: every new vector lies within
    1% of the basis, which takes the second Gram-Schmidt pass in every iteration."""
    from oracle import mc_assemble
    m = 700
    Y, N, _ = S.sphere_samples(m)
    rng = np.random.default_rng(5)
    g = (rng.normal(size=m) + 1j * rng.normal(size=m)).astype(np.complex64)
    L, R = mc_assemble(Y, N, 0.02, 2.0)
    ref = np.linalg.solve(L, R @ g)
    with nb.Operator.assemble_mc(Y, N, 0.02, 2.0) as op:
        x, info, st = op.solve(g)
        assert st == nb.NAT_BEM_OK and info.iterations >= 2
    assert _rel(x, ref) < 1e-5  # FP32 entries (6e-8 each) and a residual of 1e-6 on cond(L) ~ 1


def test_run_kernel_zero_right_hand_side(nb):
    V, F = S.icosphere(2)
    with nb.Operator.assemble(V, F, 1.0) as op:
        x, info, st = op.solve(np.zeros(len(F), np.complex64))
        assert st == nb.NAT_BEM_OK and info.iterations == 0 and not np.any(x)


# A mixed solve with one right-hand side ends below 0.75 tol, not just under tol (unless it stops
# contracting, at wavenumbers whose residual floor is near tol: not these), so its error does not
# hang on how a sweep's end was rounded. ||x|| / ||b|| times ||L^-1|| is about 1.2 here: errors stay
# below 0.75e-6 x 1.2 plus the FP32 operator's own 1e-7.
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_mixed_solves_end_well_below_the_tolerance(nb, oracle_lib, prec):
    p = {"bf16": nb.PREC_MIXED_BF16, "fp16": nb.PREC_MIXED_FP16}[prec]
    opts = nb.nat_bem_opts_default(prec=p)
    jobs = []
    for i in range(16):
        Vs, F = S.ring_sphere(500 + 130 * i)
        V = S.perturbed_ellipsoid(Vs, 60 + i)
        k = 3.0 + 0.35 * i
        jobs.append(dict(V=V, F=F, k=k, neumann=S.monopole_neumann(V, F, k).astype(np.complex64)))
    st, res = nb.nat_bem_run_batch_fused(jobs, opts)
    assert st == nb.NAT_BEM_OK
    for i, (job, r) in enumerate(zip(jobs, res)):
        with nb.Operator.assemble(job["V"], job["F"], job["k"], opts) as op:
            x, info, st = op.solve(job["neumann"])
        assert st == nb.NAT_BEM_OK
        assert max(info.rel_residual, r[2].rel_residual) <= 0.75e-6, (i, info.rel_residual, r[2].rel_residual)
        if i % 5 == 0:
            L, R = oracle_lib.assemble(job["V"], job["F"], job["k"])
            ref = np.linalg.solve(L, R @ job["neumann"].astype(np.complex128))
            assert max(_rel(x, ref), _rel(r[0], ref)) < 1e-6


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_single_solve_after_several_right_hand_sides(nb, prec):
    """A workspace made for several right-hand sides serves one as a fresh one does: the same bits."""
    Vs, F = S.ring_sphere(1218)
    V = S.perturbed_ellipsoid(Vs, 71)
    g = S.monopole_neumann(V, F, 3.0).astype(np.complex64)
    opts = nb.nat_bem_opts_default(prec={"fp32": nb.PREC_FP32, "bf16": nb.PREC_MIXED_BF16}[prec])
    with nb.Operator.assemble(V, F, 3.0, opts) as op:
        fresh, a, _ = op.solve(g)
    with nb.Operator.assemble(V, F, 3.0, opts) as op:
        op.solve(np.asfortranarray(np.stack([g, 2 * g, 1j * g, g, -g, g], 1)))
        x, b, st = op.solve(g)
    assert st == nb.NAT_BEM_OK and a.iterations == b.iterations and np.array_equal(x, fresh)
