"""GPU parity of the far-field pattern (FFAT maps, paper Sec. 3.1 and 5) and of the training
sampler (paper Sec. 3.4) against the FP64 oracle."""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

TOL = 1e-4


@pytest.fixture(scope="module")
def nb():
    import paper_2506_06190_gb300 as nb
    from paper_2506_06190_gb300 import build
    build.build()
    return nb


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def _data(n, nrhs, seed):
    rng = np.random.default_rng(seed)
    p = (rng.normal(size=(n, nrhs)) + 1j * rng.normal(size=(n, nrhs))).astype(np.complex64)
    g = (rng.normal(size=(n, nrhs)) + 1j * rng.normal(size=(n, nrhs))).astype(np.complex64)
    return np.asfortranarray(p), np.asfortranarray(g)


@pytest.mark.parametrize("nrhs", [1, 3, 6])
def test_far_field_matches_oracle(nb, oracle_lib, nrhs):
    Vs, F = S.ring_sphere(1500)
    V = S.perturbed_ellipsoid(Vs, 12)
    k = 3.0
    dirs = oracle_lib.ffat_directions(64, 32)
    P, G = _data(len(F), nrhs, 5)
    with nb.Operator.assemble(V, F, k) as op:
        out = op.far_field(dirs, P if nrhs > 1 else P[:, 0], G if nrhs > 1 else G[:, 0])
    out = np.asarray(out).reshape(len(dirs), nrhs, order="F") if nrhs > 1 else np.asarray(out)[:, None]
    for s in range(nrhs):
        ref = oracle_lib.far_field(V, F, k, dirs, P[:, s].astype(np.complex128), G[:, s].astype(np.complex128))
        assert _rel(out[:, s], ref) < TOL


def test_far_field_of_a_monte_carlo_op(nb, oracle_lib):
    Y, N, A = S.sphere_samples(900, 1.1)
    k = 4.0
    dirs = oracle_lib.ffat_directions(64, 32)
    P, G = _data(900, 1, 6)
    with nb.Operator.assemble_mc(Y, N, A, k) as op:
        out = op.far_field(dirs, P[:, 0], G[:, 0])
    ref = oracle_lib.mc_far_field(Y, N, A, k, dirs, P[:, 0].astype(np.complex128), G[:, 0].astype(np.complex128))
    assert _rel(out, ref) < TOL


def test_ffat_map_of_the_pulsating_sphere(nb):
    """Solve on the GPU, then the 64 x 32 FFAT map: |F| = |p(a)| a for the pulsating sphere."""
    V, F = S.icosphere(3)
    k = 2.0
    g = np.ones(len(F), np.complex64)
    with nb.Operator.assemble(V, F, k) as op:
        p, info, st = op.solve(g)
        assert st == nb.NAT_BEM_OK
        import oracle
        ff = op.far_field(oracle.ffat_directions(64, 32), p, g)
    exact = abs(1.0 / (1j * k - 1.0))
    assert np.max(np.abs(np.abs(ff) - exact)) / exact < 0.03


@pytest.mark.parametrize("nrhs", [1, 2])
def test_training_samples_match_oracle(nb, oracle_lib, nrhs):
    """10,000 samples in the shell 1.5-3 bounding radii about the body (paper Sec. 3.4)."""
    Vs, F = S.ring_sphere(1200)
    V = S.perturbed_ellipsoid(Vs, 13)
    k = 2.5
    lo, hi = V.min(axis=0), V.max(axis=0)
    center, rb = 0.5 * (lo + hi), 0.5 * np.linalg.norm(hi - lo)
    u = np.random.default_rng(7).random((10000, 3))
    P, G = _data(len(F), nrhs, 8)
    with nb.Operator.assemble(V, F, k) as op:
        coords, amp = op.sample_field(u, center, 1.5 * rb, 3.0 * rb, P if nrhs > 1 else P[:, 0],
                                      G if nrhs > 1 else G[:, 0])
    tpr, xyz = oracle_lib.sample_coords(u, center, 1.5 * rb, 3.0 * rb)
    assert np.allclose(coords, tpr, rtol=0, atol=1e-12)
    amp = np.asarray(amp).reshape(10000, nrhs, order="F") if nrhs > 1 else np.asarray(amp)[:, None]
    for s in range(nrhs):
        ref = np.abs(oracle_lib.evaluate(V, F, k, xyz, P[:, s].astype(np.complex128), G[:, s].astype(np.complex128)))
        assert _rel(amp[:, s], ref) < TOL


def test_sampler_rejects_bad_radii(nb):
    V, F = S.icosphere(1)
    with nb.Operator.assemble(V, F, 1.0) as op:
        g = np.ones(len(F), np.complex64)
        with pytest.raises(nb.NatBemError):
            op.sample_field(np.zeros((4, 3)), np.zeros(3), 2.0, 1.0, g, g)


def test_dataset_step_at_full_size(nb, oracle_lib):
    """The dataset workload's configuration (interior-source body, 10240 triangles): the GPU
    solve, then 10,000 shell samples and the 64 x 32 FFAT map; sampled outputs against the
    oracle's field and far field of the same surface data."""
    prob = S.interior_source(n_k=1, ka_range=(6.0, 6.0))
    V, F, k = prob.V, prob.F, float(prob.ks[0])
    g = np.ascontiguousarray(prob.neumann[0][:, 0]).astype(np.complex64)
    lo, hi = V.min(axis=0), V.max(axis=0)
    center, rb = 0.5 * (lo + hi), 0.5 * np.linalg.norm(hi - lo)
    u = np.random.default_rng(70).random((10000, 3))
    dirs = oracle_lib.ffat_directions(64, 32)
    with nb.Operator.assemble(V, F, k) as op:
        p, info, st = op.solve(g)
        assert st == nb.NAT_BEM_OK
        coords, amp = op.sample_field(u, center, 1.5 * rb, 3.0 * rb, p, g)
        ff = op.far_field(dirs, p, g)
    pick = np.random.default_rng(71).choice(10000, 64, replace=False)
    _, xyz = oracle_lib.sample_coords(u[pick], center, 1.5 * rb, 3.0 * rb)
    p64, g64 = p.astype(np.complex128), g.astype(np.complex128)
    ref = np.abs(oracle_lib.evaluate(V, F, k, xyz, p64, g64))
    assert _rel(amp[pick], ref) < TOL
    dpick = np.random.default_rng(72).choice(len(dirs), 48, replace=False)
    ref_ff = oracle_lib.far_field(V, F, k, dirs[dpick], p64, g64)
    assert _rel(ff[dpick], ref_ff) < TOL


# Random surface data: the sum over 302 x 7 terms cancels to its root mean square, so FP32 terms
# (a few 6e-8 each, phases up to k r = 18 rounded at 1e-6) leave at most about 1e-6 x sqrt(N / N_eff)
# ~ 5e-6 of the result; 2e-5 holds for every pass width and remainder.
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 9, 17, 33])
@pytest.mark.parametrize("n_tri,m", [(8, 1), (302, 127), (1218, 129)])
def test_field_and_far_field_pass_widths_and_remainders(nb, oracle_lib, n_tri, m, nrhs):
    Vs, F = S.ring_sphere(n_tri)
    V = S.perturbed_ellipsoid(Vs, 41) + np.array([3.0, -1.0, 0.5])
    k = 2.37
    rng = np.random.default_rng(n_tri + nrhs)
    p, g = ((rng.normal(size=(n_tri, nrhs)) + 1j * rng.normal(size=(n_tri, nrhs))).astype(np.complex64) for _ in range(2))
    pts = S.shell_points(m, 6.0, 9.0, 3)
    dirs = S.fibonacci_points(m, 1.0) if m > 1 else np.array([[0.0, 0.6, 0.8]])
    with nb.Operator.assemble(V, F, k) as op:
        f, far = op.evaluate(pts, p, g), op.far_field(dirs, p, g)
    for s in (0, nrhs - 1):
        ref = oracle_lib.evaluate(V, F, k, pts, p[:, s], g[:, s])
        assert _rel(f[:, s], ref) < 2e-5
        ref = oracle_lib.far_field(V, F, k, dirs, p[:, s], g[:, s])
        assert _rel(far[:, s], ref) < 2e-5


# Field points over the outer quadrature points of some elements, `height` element sizes above them:
# d = D - q comes from parts of about half an element rounded at 2^-24 and the nearest point's term
# goes as 1/d^2, so 4 x 2^-24 / height on top of the 2e-5 of the other field tests.
@pytest.mark.parametrize("nrhs", [1, 3, 9, 20])
@pytest.mark.parametrize("height", [0.3, 0.1, 0.03, 0.01, 1e-3, 1e-4])
def test_field_close_to_quadrature_points(nb, oracle_lib, height, nrhs):
    Vs, F = S.ring_sphere(515 - 1)
    V = S.perturbed_ellipsoid(Vs, 42)
    k = 2.0
    cr = np.cross(V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]])
    size, nrm = np.sqrt(np.linalg.norm(cr, axis=1)), cr / np.linalg.norm(cr, axis=1)[:, None]
    rule, _ = oracle_lib.quad_rule()
    t = np.arange(0, len(F), 3)
    q = 1 + np.arange(len(t)) % 6
    pts = np.einsum("tv,tvd->td", rule[q], V[F[t]]) + height * size[t, None] * nrm[t]
    rng = np.random.default_rng(7)
    p, g = ((rng.normal(size=(len(F), nrhs)) + 1j * rng.normal(size=(len(F), nrhs))).astype(np.complex64)
            for _ in range(2))
    with nb.Operator.assemble(V, F, k) as op:
        f = op.evaluate(pts, p, g)
    assert np.isfinite(f).all()
    for s in (0, nrhs - 1):
        ref = oracle_lib.evaluate(V, F, k, pts, p[:, s], g[:, s])
        assert _rel(f[:, s], ref) < 2e-5 + 4 * 2.0 ** -24 / height


@pytest.mark.parametrize("height", [1e-2, 1e-5, 1e-9])
def test_field_close_to_monte_carlo_samples(nb, oracle_lib, height):
    Y, N, A = S.sphere_samples(900, 1.1)
    p, g = _data(900, 1, 43)
    pts = Y[::7] + height * N[::7]
    with nb.Operator.assemble_mc(Y, N, A, 2.0) as op:
        f = op.evaluate(pts, p[:, 0], g[:, 0])
    assert np.isfinite(f).all()
    ref = oracle_lib.mc_evaluate(Y, N, A, 2.0, pts, p[:, 0].astype(np.complex128), g[:, 0].astype(np.complex128))
    # hi/lo differences resolve 2^-48 of the sphere; normals and weights round at 2^-24
    assert _rel(f, ref) < 2e-5 + 4 * 2.0 ** -48 / height


@pytest.mark.parametrize("shift", [0.0, 500.0])
def test_a_point_does_not_depend_on_the_others(nb, oracle_lib, shift):
    """The same points beside one at 1e30, which once took the low parts of the others' coordinates."""
    Vs, F = S.ring_sphere(600)
    V = S.perturbed_ellipsoid(Vs, 44) + shift
    k = 2.0
    p, g = _data(len(F), 1, 45)
    pts = S.shell_points(128, 1.5, 6.0, 4) + shift
    far = pts.copy()
    far[-1] = 1e30
    with nb.Operator.assemble(V, F, k) as op:
        a, b = op.evaluate(pts, p[:, 0], g[:, 0]), op.evaluate(far, p[:, 0], g[:, 0])
    assert np.array_equal(a[:-1], b[:-1])
    ref = oracle_lib.evaluate(V, F, k, pts, p[:, 0].astype(np.complex128), g[:, 0].astype(np.complex128))
    assert _rel(a, ref) < 2e-5  # as in test_field_and_far_field_pass_widths_and_remainders
