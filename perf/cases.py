"""The measured cases: the work users of this library have it do, over the sizes they do it at.

Each case goes through the package's public entry points. The kinds are

  sweep      one step of a wavenumber sweep: re-assemble the operators of a body at a new k,
             solve for the surface pressure, evaluate the field (collocation form);
  galerkin   the same step in the Galerkin form (P1 pressure, P0 Neumann data);
  mc         the same step on Monte-Carlo surface samples;
  sampler    Poisson-disk samples of a mesh, which the Monte-Carlo form starts from;
  fused      a batch of meshes of uneven size, one wavenumber and right-hand side each;
  requests   a batch of requests of uneven size with several right-hand sides each;
  training   shell samples of |p| and a far-field map for solved surface data;
  field      inference of the neural transfer field.

Bodies are perturbed ellipsoids (radii 1, 0.8, 0.6) on a closed, near-uniform triangulation, the
Neumann data those of monopoles inside the body (one, or three with random strengths per
right-hand side), so the surface pressure is smooth as a vibrating object's is. `exact` states
the same discrete problems in 64-bit torch, assembled and solved without the package.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_2506_06190_gb300 as nb

PREC = {"fp32": 0, "bf16": 2}
LEVELS = (8, 16, 32, 64)  # grid cells per axis of the neural field's four levels
WIDTH = 128


def listed():
    return [
        # the smallest body in use, a pulsating-sphere sized check: a pass of many short kernels
        dict(name="sweep_1280", kind="sweep", tri=1280, ka=2.0, nrhs=1, points=256, prec="fp32"),
        # a mid-sized object (the plate of the paper's examples) in plain single precision
        dict(name="sweep_5174", kind="sweep", tri=5174, ka=8.0, nrhs=1, points=1024, prec="fp32"),
        # the headline: one wavenumber of an interior-source body, mixed precision
        dict(name="sweep_10240_bf16", kind="sweep", tri=10240, ka=10.0, nrhs=1, points=1024, prec="bf16"),
        # modal transfer: all modes of one body at one wavenumber; the largest operator
        dict(name="modal_20480_bf16", kind="sweep", tri=20480, ka=6.0, nrhs=64, points=4096, prec="bf16"),
        # data generation over many different bodies, one small solve each
        dict(name="fused_24", kind="fused", jobs=24, lo=500, hi=8000, prec="bf16"),
        # a burst of serving requests, meshes and right-hand sides of every size
        dict(name="requests_6", kind="requests", jobs=6, lo=1000, hi=16000, prec="bf16"),
        # the Monte-Carlo form on about 4000 samples
        dict(name="mc_4096", kind="mc", samples=4096, ka=4.0, points=1024, prec="fp32"),
        # drawing those samples
        dict(name="sampler_32768", kind="sampler", tri=10240, draws=32768),
        # the Galerkin form
        dict(name="galerkin_5120", kind="galerkin", tri=5120, ka=4.0, points=1024, prec="fp32"),
        # training data of one solve: 10,000 shell samples and a 64 x 32 far-field map
        dict(name="training_10240", kind="training", tri=10240, ka=10.0, samples=10000, dirs=2048),
        # neural-field inference: a whole sound field at many listeners, and one frame of a scene
        dict(name="field_4m", kind="field", n=1 << 22, cond=2, out=8, table=18),
        dict(name="field_1000", kind="field", n=1000, cond=2, out=8, table=18),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return n - n % 2


def _ka(rng, tri, most=20.0):
    """A wavenumber with at least six elements per wavelength on a body of `tri` triangles."""
    h = math.sqrt(4.0 * 7.5 / (math.sqrt(3.0) * tri))
    return round(rng.uniform(0.5, min(most, math.pi / (3.0 * h))), 4)


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "modal", "fused", "requests", "mc", "sampler", "galerkin", "training",
                       "field", "field"])
    prec = rng.choice(["fp32", "bf16"])
    if kind == "sweep":
        tri = _even(_log_int(rng, 320, 12000))
        return dict(kind="sweep", tri=tri, ka=_ka(rng, tri), nrhs=1, points=_log_int(rng, 100, 4096), prec=prec)
    if kind == "modal":
        tri = _even(_log_int(rng, 1000, 12000))
        return dict(kind="sweep", tri=tri, ka=_ka(rng, tri, 15.0), nrhs=_log_int(rng, 2, 64),
                    points=_log_int(rng, 100, 4096), prec=prec)
    if kind == "fused":
        lo = _log_int(rng, 500, 1500)
        return dict(kind="fused", jobs=rng.randint(4, 24), lo=lo, hi=_log_int(rng, 2 * lo, 8000), prec=prec)
    if kind == "requests":
        lo = _log_int(rng, 1000, 3000)
        return dict(kind="requests", jobs=rng.randint(2, 6), lo=lo, hi=_log_int(rng, 2 * lo, 12000), prec="bf16")
    if kind == "mc":
        return dict(kind="mc", samples=_log_int(rng, 500, 4096), ka=round(rng.uniform(0.5, 6.0), 4),
                    points=_log_int(rng, 100, 4096), prec=rng.choice(["fp32", "fp32", "bf16"]))
    if kind == "sampler":
        return dict(kind="sampler", tri=_even(_log_int(rng, 500, 20000)), draws=_log_int(rng, 1000, 65536))
    if kind == "galerkin":
        tri = _even(_log_int(rng, 320, 5120))
        return dict(kind="galerkin", tri=tri, ka=_ka(rng, tri, 10.0), points=_log_int(rng, 100, 4096), prec="fp32")
    if kind == "training":
        tri = _even(_log_int(rng, 1000, 20000))
        return dict(kind="training", tri=tri, ka=_ka(rng, tri), samples=_log_int(rng, 500, 20000),
                    dirs=rng.choice([512, 2048, 2049, 8192]))
    return dict(kind="field", n=_log_int(rng, 1, 1 << 22), cond=rng.randint(0, 5), out=rng.choice([1, 3, 8, 32, 64]),
                table=rng.choice([14, 16, 18, 19]))


# ------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=64)
def _sphere(tri):
    """Unit sphere of exactly `tri` (even) near-equilateral triangles: two poles and rings of
    latitude whose vertex counts follow sin(theta), neighbouring rings stitched by angle."""
    total = tri // 2
    h = math.sqrt(16.0 * math.pi / (math.sqrt(3.0) * tri))
    nr = min(max(1, round(math.pi / (h * math.sqrt(0.75))) - 1), max(1, total // 3))
    th = np.pi * np.arange(1, nr + 1) / (nr + 1)
    share = np.cumsum(np.sin(th)) / np.sin(th).sum() * total
    cnt = np.maximum(3, np.diff(np.concatenate([[0], np.round(share)])).astype(int))
    cnt[np.argmax(cnt)] += total - cnt.sum()
    start = np.concatenate([[1], 1 + np.cumsum(cnt)])
    ang = [2 * np.pi * (np.arange(c) + 0.5 * (i % 2)) / c for i, c in enumerate(cnt)]
    V = [np.array([[0.0, 0.0, 1.0]])]
    V += [np.stack([math.sin(t) * np.cos(a), math.sin(t) * np.sin(a), np.full(len(a), math.cos(t))], 1)
          for t, a in zip(th, ang)]
    V = np.concatenate(V + [np.array([[0.0, 0.0, -1.0]])])
    F = [(0, 1 + j, 1 + (j + 1) % cnt[0]) for j in range(cnt[0])]
    for r in range(nr - 1):
        na, nb_ = int(cnt[r]), int(cnt[r + 1])
        a0, b0 = ang[r][0], ang[r + 1]
        off = int(np.argmin((b0 - a0) % (2 * np.pi)))
        lag = float((b0[off] - a0) % (2 * np.pi))
        i = j = 0
        while i < na or j < nb_:
            p, q = start[r] + i % na, start[r + 1] + (off + j) % nb_
            if j >= nb_ or (i < na and 2 * math.pi * (i + 1) / na <= lag + 2 * math.pi * (j + 1) / nb_):
                i += 1
                F.append((p, q, start[r] + i % na))
            else:
                j += 1
                F.append((p, q, start[r + 1] + (off + j) % nb_))
    last, n = start[nr - 1], int(cnt[-1])
    F += [(len(V) - 1, last + (j + 1) % n, last + j) for j in range(n)]
    return V, np.array(F, dtype=np.int32)


def _body(tri, rng):
    """Perturbed ellipsoid: the unit directions scaled by a smooth random radius and the axes."""
    D, F = _sphere(tri)
    q = rng.normal(size=(6, 3))
    q *= rng.uniform(1.0, 6.0, size=(6, 1)) / np.linalg.norm(q, axis=1, keepdims=True)
    amp, ph = 0.05 * rng.normal(size=6), rng.uniform(0.0, 2 * np.pi, 6)
    radius = 1.0 + (np.cos(D @ q.T + ph) * amp).sum(1)
    return D * radius[:, None] * np.array([1.0, 0.8, 0.6]), F


def _triangles(V, F):
    P = V[F]
    cr = np.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    dbl = np.linalg.norm(cr, axis=1)
    return P, P.mean(1), cr / dbl[:, None], 0.5 * dbl


def _sources(rng, nrhs):
    """Monopoles inside the body: positions and their strengths per right-hand side."""
    if nrhs == 1:
        return 0.1 * rng.uniform(-1, 1, (1, 3)), np.ones((1, 1), complex)
    return 0.15 * rng.uniform(-1, 1, (3, 3)), rng.normal(size=(3, nrhs)) + 1j * rng.normal(size=(3, nrhs))


def _monopoles(Y, N, k, at, strength):
    """The monopoles' pressure and its normal derivative at points Y with normals N: (nrhs, n)."""
    d = Y[:, None, :] - at
    r = np.linalg.norm(d, axis=2)
    u = np.exp(1j * k * r) / (4 * np.pi * r)
    du = u * (1j * k - 1 / r) * (d * N[:, None, :]).sum(2) / r
    return (u @ strength).T, (du @ strength).T


def _shell(n, lo, hi, rng):
    d = rng.normal(size=(n, 3))
    return d / np.linalg.norm(d, axis=1, keepdims=True) * rng.uniform(lo, hi, (n, 1))


def _problem(tri, k, nrhs, points, rng):
    V, F = _body(tri, rng)
    _, cen, nrm, _ = _triangles(V, F)
    p, g = _monopoles(cen, nrm, k, *_sources(rng, nrhs))
    return dict(V=V, F=F, p=p.astype(np.complex64), g=g.astype(np.complex64), pts=_shell(points, 2.0, 5.0, rng), k=k)


def _jobs(case, rng):
    """The meshes of a batch: triangle counts spread over the logarithm of the range, a wavenumber
    each, and for requests 1 to 32 right-hand sides; these are the case's, shapes and data the
    seed's."""
    n, pick, out = case["jobs"], np.random.default_rng([case["jobs"], case["lo"], case["hi"]]), []
    for i in range(n):
        tri = _even(int(round(case["lo"] * (case["hi"] / case["lo"]) ** ((i + pick.uniform(0, 1)) / n))))
        nrhs = int(pick.integers(1, 33)) if case["kind"] == "requests" else 1
        h = math.sqrt(4.0 * 7.5 / (math.sqrt(3.0) * tri))
        k = float(pick.uniform(0.5, min(12.0, math.pi / (3.0 * h))))
        out.append(_problem(tri, k, nrhs, 1024, rng))
    return out


def _draws(tri, draws, rng):
    """A mesh, uniform draws on it and the sample radius: 0.7 of the spacing of a hexagonal
    packing of draws / 8 points."""
    V, F = _body(tri, rng)
    area = float(_triangles(V, F)[3].sum())
    return V, F, rng.random((draws, 3)), 0.7 * math.sqrt(2.0 * area / (math.sqrt(3.0) * (draws / 8)))


def _candidates(V, F, u):
    P, _, nrm, area = _triangles(V, F)
    cum = np.cumsum(area)
    t = np.minimum(np.searchsorted(cum, u[:, 0] * cum[-1], side="right"), len(F) - 1)
    s = np.sqrt(u[:, 1])
    b = np.stack([1 - s, s * (1 - u[:, 2]), s * u[:, 2]], 1)
    return (b[:, :, None] * P[t]).sum(1), nrm[t]


def _spaced(x, radius):
    """Greedy choice of points at least `radius` apart, lower indexes first: in rounds, each
    accepting the open points with no open lower-indexed neighbour."""
    y = torch.from_numpy(x).cuda()
    n = len(x)
    idx = torch.arange(n, device="cuda")
    near = torch.cat([torch.cdist(c, y) < radius for c in y.split(4096)])
    open_, taken = torch.ones(n, dtype=torch.bool, device="cuda"), torch.zeros(n, dtype=torch.bool, device="cuda")
    while bool(open_.any()):
        lowest = (near & open_).to(torch.uint8).argmax(1)
        now = open_ & (lowest == idx)
        taken |= now
        open_ &= ~near[now].any(0)
    return taken.cpu().numpy()


def _mc_inputs(case, rng):
    # one body and its samples, as many as they come; the sources and points are the seed's
    V, F, u, radius = _draws(10240, 8 * case["samples"], np.random.default_rng(case["samples"]))
    x, n = _candidates(V, F, u)
    keep = _spaced(x, radius)
    x, n = np.ascontiguousarray(x[keep]), np.ascontiguousarray(n[keep])
    _, g = _monopoles(x, n, case["ka"], *_sources(rng, 1))
    return dict(Y=x, N=n, area=float(_triangles(V, F)[3].sum()), g=g[0].astype(np.complex64),
                pts=_shell(case["points"], 2.0, 5.0, rng))


def _training_inputs(case, rng):
    q = _problem(case["tri"], case["ka"], 1, 1, rng)
    lo, hi = q["V"].min(0), q["V"].max(0)
    m = max(1, math.isqrt(case["dirs"] // 2))
    th = (np.arange(m) + 0.5) * np.pi / m
    cols = -(-case["dirs"] // m)
    T, P = np.meshgrid(th, (np.arange(cols) + 0.5) * 2 * np.pi / cols, indexing="ij")
    dirs = np.stack([np.sin(T) * np.cos(P), np.sin(T) * np.sin(P), np.cos(T)], -1).reshape(-1, 3)[: case["dirs"]]
    return dict(q, u=rng.random((case["samples"], 3)), center=0.5 * (lo + hi), rb=0.5 * float(np.linalg.norm(hi - lo)),
                dirs=np.ascontiguousarray(dirs))


def _field_inputs(case, seed):
    rng = np.random.default_rng(seed)
    tables = [rng.uniform(-1, 1, (min((n + 1) ** 3, 1 << case["table"]), 4)).astype(np.float32) for n in LEVELS]
    outs = [WIDTH] * 4 + [case["out"]]
    weights = [rng.normal(0, math.sqrt(2 / WIDTH), (o, WIDTH)).astype(np.float32) for o in outs]
    biases = [rng.normal(0, 0.05, o).astype(np.float32) for o in outs]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((case["n"], 4 + case["cond"]), generator=gen, device="cuda")
    return dict(n_cond=case["cond"], n_out=case["out"], table_log2=case["table"], tables=tables, weights=weights,
                biases=biases), x


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _opts(case):
    return nb.nat_bem_opts_default(prec=PREC[case["prec"]])


# ------------------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    rng, kind = np.random.default_rng(seed), case["kind"]
    if kind in ("sweep", "galerkin"):
        q = _problem(case["tri"], case["ka"], case.get("nrhs", 1), case["points"], rng)
        make = nb.Operator.assemble if kind == "sweep" else nb.Operator.assemble_galerkin
        g = _cuda(q["g"] if case.get("nrhs", 1) > 1 else q["g"][0])
        return dict(kind=kind, k=case["ka"], g=g, pts=_cuda(q["pts"]),
                    op=make(_cuda(q["V"]), _cuda(q["F"]), 0.75 * case["ka"], _opts(case)))
    if kind == "mc":
        q = _mc_inputs(case, rng)
        return dict(kind=kind, k=case["ka"], g=_cuda(q["g"]), pts=_cuda(q["pts"]),
                    op=nb.Operator.assemble_mc(_cuda(q["Y"]), _cuda(q["N"]), q["area"], 0.75 * case["ka"], _opts(case)))
    if kind == "sampler":
        V, F, u, radius = _draws(case["tri"], case["draws"], rng)
        return dict(kind=kind, V=_cuda(V), F=_cuda(F), u=_cuda(u), radius=radius)
    if kind in ("fused", "requests"):
        jobs = [dict(V=_cuda(q["V"]), F=_cuda(q["F"]), k=q["k"], neumann=_cuda(q["g"]), points=_cuda(q["pts"]))
                for q in _jobs(case, rng)]
        return dict(kind=kind, jobs=jobs, opts=_opts(case))
    if kind == "training":
        q = _training_inputs(case, rng)
        return dict(kind=kind, op=nb.Operator.assemble(_cuda(q["V"]), _cuda(q["F"]), case["ka"]), p=_cuda(q["p"][0]),
                    g=_cuda(q["g"][0]), u=_cuda(q["u"]), dirs=_cuda(q["dirs"]), center=q["center"], rb=q["rb"])
    params, x = _field_inputs(case, seed)
    return dict(kind=kind, field=nb.NatField.from_params(params), x=x)


def run(state):
    kind = state["kind"]
    if kind in ("sweep", "galerkin", "mc"):
        op, g = state["op"], state["g"]
        op.reassemble(state["k"], like=g)
        p, _, _ = op.solve(g)
        return p, op.evaluate(state["pts"], p, g)
    if kind == "sampler":
        idx, x, n = nb.nat_bem_poisson_sample(state["V"], state["F"], state["u"], state["radius"])
        return _padded(idx, x, n, len(state["u"]))
    if kind == "fused":
        _, res = nb.nat_bem_run_batch_fused(state["jobs"], state["opts"])
        return [r[:2] for r in res]
    if kind == "requests":
        _, res = nb.nat_bem_run_batch(state["jobs"], state["opts"], concurrency=4)
        return [r[:2] for r in res]
    if kind == "training":
        op, p, g, rb = state["op"], state["p"], state["g"], state["rb"]
        coords, amp = op.sample_field(state["u"], state["center"], 1.5 * rb, 3.0 * rb, p, g)
        return coords, amp, op.far_field(state["dirs"], p, g)
    return state["field"].forward(state["x"])


# --------------------------------------------------------------------------------------- work
def _step_work(n, nrhs, points, pair_flops, el, iters=30):
    """Flops and bytes of one assemble, solve, evaluate step: `pair_flops` per operator entry
    pair, `iters` matvecs per right-hand side, 280 flops per (point, element) of the field."""
    flops = n * n * (pair_flops + 8.0 * nrhs * iters) + 280.0 * points * el * max(1, nrhs // 4)
    return 8.0 * nrhs * (el + n + points) + 24.0 * (el + points), flops


def work(case):
    kind = case["kind"]
    if kind == "sweep":
        b, f = _step_work(case["tri"], case["nrhs"], case["points"], 560, case["tri"])
    elif kind == "galerkin":
        b, f = _step_work(case["tri"] // 2 + 2, 1, case["points"], 4 * 4067, case["tri"])
    elif kind == "mc":
        b, f = _step_work(case["samples"], 1, case["points"], 40, case["samples"])
    elif kind in ("fused", "requests"):
        b = f = 0.0
        for i in range(case["jobs"]):
            n = case["lo"] * (case["hi"] / case["lo"]) ** ((i + 0.5) / case["jobs"])
            x, y = _step_work(n, 16 if kind == "requests" else 1, 1024, 560, n)
            b, f = b + x, f + y
    elif kind == "sampler":
        b, f = 24.0 * case["draws"] + 24.0 * case["tri"] + 56.0 * case["draws"] / 8, 1000.0 * case["draws"]
    elif kind == "training":
        b = 16.0 * case["tri"] + 24.0 * case["tri"] + 52.0 * case["samples"] + 32.0 * case["dirs"]
        f = 7.0 * case["tri"] * (40.0 * case["samples"] + 16.0 * case["dirs"])
    else:
        d = 4 + case["cond"]
        rows = sum(min((n + 1) ** 3, 1 << case["table"]) for n in LEVELS)
        b = 4.0 * case["n"] * (d + case["out"]) + 8.0 * rows + 2.0 * WIDTH * (4 * WIDTH + case["out"])
        f = 2.0 * case["n"] * WIDTH * (16 + 12 * (case["cond"] + 1) + 3 * WIDTH + case["out"])
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------------- 64-bit statements
# The discrete problems in torch float64 / complex128 on the GPU.
_S15 = math.sqrt(15.0)
_A, _B = (6 - _S15) / 21, (6 + _S15) / 21
BARY = np.array([[1 / 3] * 3, [_A, _A, 1 - 2 * _A], [_A, 1 - 2 * _A, _A], [1 - 2 * _A, _A, _A],
                 [_B, _B, 1 - 2 * _B], [_B, 1 - 2 * _B, _B], [1 - 2 * _B, _B, _B]])
WGT = np.array([9 / 40] + [(155 - _S15) / 1200] * 3 + [(155 + _S15) / 1200] * 3)


class _Geo:
    def __init__(self, V, F):
        self.V, self.F = V, F
        P, cen, nrm, area = _triangles(V, F)
        self.P, self.cen, self.nrm, self.area = _cuda(P), _cuda(cen), _cuda(nrm), _cuda(area)
        self.y = torch.einsum("qa,tad->tqd", _cuda(BARY), self.P)  # quadrature points
        self.w = _cuda(WGT) * self.area[:, None]                   # and weights

    @functools.cached_property
    def touching(self):
        """Ordered pairs of different triangles that share a vertex, with the number shared."""
        n, flat = len(self.F), self.F.reshape(-1)
        order = np.argsort(flat, kind="stable")
        at = np.split(order // 3, np.cumsum(np.bincount(flat, minlength=len(self.V)))[:-1])
        key = np.concatenate([(t[:, None] * n + t).ravel() for t in at]).astype(np.int64)
        key, cnt = np.unique(key, return_counts=True)
        i, j = key // n, key % n
        return i[i != j], j[i != j], cnt[i != j]


def _kernels(k, d, nx, ny):
    """G, dG/dn_y, dG/dn_x and d2G/dn_x dn_y for d = x - y (last axis)."""
    r = d.square().sum(-1).sqrt()
    G = torch.polar(1 / (4 * math.pi * r), k * r)
    f = G * torch.complex(-1 / r, torch.full_like(r, k))  # dG/dr
    rx, ry = (d * nx).sum(-1) / r, -(d * ny).sum(-1) / r
    h = G * torch.complex(2 / r ** 2 - k * k, -2 * k / r) * (rx * ry) - f * (((nx * ny).sum(-1) + rx * ry) / r)
    return G, f * ry, f * rx, h


def _collocation(V, F, k):
    """L and R of the Burton-Miller system by centroid collocation of piecewise constants."""
    g, n, beta = _Geo(V, F), len(F), 1j / k
    L = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    R = torch.empty_like(L)

    def entries(x, nx, y, ny, w):
        G, Gy, Gx, H = _kernels(k, x - y, nx, ny)
        return -((Gy + beta * H) * w).sum(-1), -((G + beta * Gx) * w).sum(-1)

    step = max(1, (1 << 22) // (7 * n))
    for a in range(0, n, step):
        s = slice(a, a + step)
        L[s], R[s] = entries(g.cen[s, None, None], g.nrm[s, None, None], g.y, g.nrm[:, None], g.w)
    tri = [np.eye(3)]  # vertex-sharing pairs: the rule on each of 16 congruent sub-triangles
    for _ in range(2):
        tri = [np.stack(c) for t in tri for m in [((t[0] + t[1]) / 2, (t[1] + t[2]) / 2, (t[2] + t[0]) / 2)]
               for c in ((t[0], m[0], m[2]), (m[0], t[1], m[1]), (m[2], m[1], t[2]), m)]
    bary, wgt = _cuda(np.concatenate([BARY @ t for t in tri])), _cuda(np.tile(WGT / 16, 16))
    i, j, _ = g.touching
    for a in range(0, len(i), 1 << 15):
        u, v = _cuda(i[a:a + (1 << 15)]), _cuda(j[a:a + (1 << 15)])
        y = torch.einsum("qa,tad->tqd", bary, g.P[v])
        L[u, v], R[u, v] = entries(g.cen[u, None], g.nrm[u, None], y, g.nrm[v, None], wgt * g.area[v, None])
    # the element itself: polar coordinates, exact in the radius, Hadamard finite part
    gx, gw = (_cuda(t) for t in np.polynomial.legendre.leggauss(32))
    S = torch.zeros(n, dtype=torch.complex128, device="cuda")
    FP = torch.zeros_like(S)
    for e in range(3):
        p, q = g.P[:, e] - g.cen, g.P[:, (e + 1) % 3] - g.cen
        t = (q - p) / (q - p).norm(dim=1, keepdim=True)
        foot = p - t * (p * t).sum(1, keepdim=True)
        dist = foot.norm(dim=1)
        lo, hi = torch.atan2((p * t).sum(1), dist), torch.atan2((q * t).sum(1), dist)
        psi = (lo + hi)[:, None] / 2 + (hi - lo)[:, None] / 2 * gx
        r, w = dist[:, None] / torch.cos(psi), (hi - lo)[:, None] / 2 * gw
        z = torch.polar(torch.ones_like(r), k * r)
        S += (w * (z - 1) / (1j * k)).sum(1) / (4 * math.pi)
        FP += (w * (1j * k - z / r)).sum(1) / (4 * math.pi)
    L.diagonal().copy_(0.5 - beta * FP)
    R.diagonal().copy_(-S - 0.5 * beta)
    return L, R


def _samples_system(Y, N, area, k):
    m = len(Y)
    w = area / m
    y, n = _cuda(Y), _cuda(N)
    L = torch.empty((m, m), dtype=torch.complex128, device="cuda")
    R = torch.empty_like(L)
    far = torch.eye(m, dtype=torch.float64, device="cuda") * 1e3  # keeps the diagonal finite
    for a in range(0, m, 512):
        d = y[a:a + 512, None] - y + far[a:a + 512, :, None]
        G, Gy, _, _ = _kernels(k, d, n[a:a + 512, None], n)
        L[a:a + 512], R[a:a + 512] = -w * Gy, -w * G
    L.diagonal().fill_(0.5)
    R.diagonal().fill_(-0.5 * math.sqrt(w / math.pi))
    return L, R


def _solve(L, b):
    """L x = b to 64 bits: a single-precision factorisation with refinement."""
    lu = torch.linalg.lu_factor(L.to(torch.complex64))
    x, scale = torch.zeros_like(b), b.abs().max()
    for _ in range(12):
        r = (b - L @ x) / scale
        dx = torch.linalg.lu_solve(*lu, r.to(torch.complex64)).to(torch.complex128) * scale
        x = x + dx
        if float(dx.norm() / x.norm()) < 1e-13:
            break
    return x


def _sources_field(k, pts, y, ny, qp, qg):
    """sum over sources of (qp dG/dn_y - qg G) at the points: sources (s, 3), charges (s, nrhs)."""
    out = []
    for x in _cuda(pts).split(max(1, (1 << 22) // len(y))):
        G, Gy, _, _ = _kernels(k, x[:, None] - y, ny, ny)
        out.append(Gy @ qp - G @ qg)
    return torch.cat(out)


def _field(V, F, k, pts, p, g):
    """Exterior representation with piecewise-constant data, p and g (nrhs, n): (nrhs, m)."""
    q = _Geo(V, F)
    w = q.w.reshape(-1, 1)
    rep = lambda a: a.T.repeat_interleave(7, 0) * w  # noqa: E731
    return _sources_field(k, pts, q.y.reshape(-1, 3), q.nrm.repeat_interleave(7, 0), rep(p), rep(g)).T


def _exact_problem(q):
    L, R = _collocation(q["V"], q["F"], q["k"])
    g = _cuda(q["g"]).to(torch.complex128)
    b = R @ g.T
    del R
    p = _solve(L, b).T
    del L
    return p, _field(q["V"], q["F"], q["k"], q["pts"], p, g)


# Galerkin pairs: barycentrics of x and y, x - y and weights, for a batch of pairs (m, 3, 3).
def _grid4():
    x, w = np.polynomial.legendre.leggauss(4)
    g = np.array(list(itertools.product((x + 1) / 2, repeat=4)))
    return _cuda(g), _cuda(np.array([np.prod(c) for c in itertools.product(w / 2, repeat=4)]))


def _combine(lam, E):
    return torch.einsum("pa,mad->mpd", lam, E)


def _vertex_pairs(Pt, Ps):
    """Pairs whose first vertices coincide: polar coordinates about it, the larger radius first."""
    (t, u, a, b), wg = _grid4()[0].T, _grid4()[1]
    for rt, rs in ((t, t * u), (t * u, t)):
        lam, mu = torch.stack([1 - rt, rt * (1 - a), rt * a], 1), torch.stack([1 - rs, rs * (1 - b), rs * b], 1)
        zero = torch.zeros_like(t)
        d = _combine(torch.stack([zero, rt * (1 - a), rt * a], 1), Pt - Pt[:, :1])
        d = d - _combine(torch.stack([zero, rs * (1 - b), rs * b], 1), Ps - Ps[:, :1])
        yield lam, mu, d, wg * t ** 3 * u * 4


def _edge_pairs(Pt, Ps):
    """Pairs whose first two vertices coincide: coordinates along and away from the edge."""
    (t, u, v, s), wg = _grid4()[0].T, _grid4()[1]
    A, B, Ct, Cs = (c[:, None] for c in (Pt[:, 0], Pt[:, 1], Pt[:, 2], Ps[:, 2]))
    for sign, (et, es, dd) in itertools.product((1.0, -1.0), ((t, t * u, t * v), (t * u, t, t * v), (t * u, t * v, t))):
        xi = (1 - dd) * s if sign > 0 else dd + (1 - dd) * s
        xs = xi + sign * dd
        col = lambda z: z[None, :, None]  # noqa: E731
        d = -col(sign * dd) * (B - A) + col(et) * (Ct - A - col(xi) * (B - A)) - col(es) * (Cs - A - col(xs) * (B - A))
        lam = torch.stack([(1 - et) * (1 - xi), (1 - et) * xi, et], 1)
        mu = torch.stack([(1 - es) * (1 - xs), (1 - es) * xs, es], 1)
        yield lam, mu, d, wg * t ** 2 * (1 - dd) * (1 - et) * (1 - es) * 4


def _same_pairs(P):
    """A triangle with itself: the offset z = y - x over a hexagon, x over a smaller copy."""
    (rho, w, a1, a2), wg = _grid4()[0].T, _grid4()[1]
    hexagon = [(1, 0), (1, 1), (0, 1), (-1, 0), (-1, -1), (0, -1)]
    for h, l in zip(hexagon, hexagon[1:] + hexagon[:1]):
        z0, z1 = rho * (h[0] + w * (l[0] - h[0])), rho * (h[1] + w * (l[1] - h[1]))
        s = (-z1).clamp(min=0) + (z1 - z0).clamp(min=0) + (1 - rho) * a1
        t = (-z1).clamp(min=0) + (1 - rho) * a1 * a2
        lam = torch.stack([1 - s, s - t, t], 1)
        mu = torch.stack([1 - s - z0, s + z0 - t - z1, t + z1], 1)
        d = -(z0[None, :, None] * (P[:, 1:2] - P[:, :1]) + z1[None, :, None] * (P[:, 2:] - P[:, 1:2]))
        yield lam, mu, d, wg * rho * (1 - rho) ** 2 * a1 * 4


def _galerkin(V, F, k):
    """L (nv x nv) and R (nv x nt) of the Galerkin form, hypersingular term by parts."""
    g, nt, nv, beta = _Geo(V, F), len(F), len(V), 1j / k
    idx = _cuda(F.astype(np.int64))
    curl = torch.stack([(g.P[:, (a + 1) % 3] - g.P[:, (a + 2) % 3]) / (2 * g.area[:, None]) for a in range(3)], 1)
    L = torch.zeros(nv * nv, dtype=torch.complex128, device="cuda")
    R = torch.zeros(nv * nt, dtype=torch.complex128, device="cuda")

    def add(i, j, li, lj, Kb, Gb, Vb, Kp):
        """The blocks of the pairs (i, j), li and lj the local vertices the rule's order stands for."""
        nn = (g.nrm[i] * g.nrm[j]).sum(-1)
        ci, cj = curl[i[..., None], li], curl[j[..., None], lj]
        H = k * k * nn[..., None, None] * Gb - (ci @ cj.transpose(-1, -2)) * Gb.sum((-1, -2))[..., None, None]
        rows, cols = idx[i[..., None], li], idx[j[..., None], lj]
        L.index_add_(0, (rows[..., :, None] * nv + cols[..., None, :]).reshape(-1), (-Kb - beta * H).reshape(-1))
        R.index_add_(0, (rows * nt + j[..., None]).reshape(-1), (-Vb - beta * Kp).reshape(-1))

    ti, tj, cnt = g.touching
    near = torch.zeros((nt, nt), dtype=torch.bool, device="cuda")
    near[_cuda(ti), _cuda(tj)] = True
    near.fill_diagonal_(True)
    bary, every, three = _cuda(BARY), torch.arange(nt, device="cuda"), torch.arange(3, device="cuda")
    step = max(1, (1 << 22) // (49 * nt))
    for a in range(0, nt, step):
        i = torch.arange(a, min(nt, a + step), device="cuda")
        d = g.y[i, None, :, None] - g.y[None, :, None]
        d = torch.where(near[i][:, :, None, None, None], torch.ones_like(d), d)
        G, Gy, Gx, _ = _kernels(k, d, g.nrm[i, None, None, None], g.nrm[None, :, None, None])
        w = (g.w[i, None, :, None] * g.w[None, :, None]) * ~near[i][:, :, None, None]
        both = lambda K: torch.einsum("pa,ijpq,qb->ijab", bary.to(K.dtype), K * w, bary.to(K.dtype))  # noqa: E731
        Gb = both(G)
        ii, jj = torch.broadcast_tensors(i[:, None], every)
        l3 = three.expand(*ii.shape, 3)
        add(ii, jj, l3, l3, both(Gy), Gb, Gb.sum(-1), both(Gx).sum(-1))

    def singular(i, j, li, lj, rule, chunk=2048):
        for a in range(0, len(i), chunk):
            s = slice(a, a + chunk)
            u, v, lu, lv = i[s], j[s], li[s], lj[s]
            Pt, Ps = g.P[u[:, None], lu], g.P[v[:, None], lv]
            for lam, mu, d, w in rule(Pt, Ps):
                G, Gy, Gx, _ = _kernels(k, d, g.nrm[u, None], g.nrm[v, None])
                ww = w * (g.area[u] * g.area[v])[:, None]
                both = lambda K: torch.einsum("pa,mp,pb->mab", lam.to(K.dtype), K * ww, mu.to(K.dtype))  # noqa: E731
                Gb = both(G)
                add(u, v, lu, lv, both(Gy), Gb, Gb.sum(-1), both(Gx).sum(-1))

    eq = F[ti][:, :, None] == F[tj][:, None, :]
    for shared, rule in ((1, _vertex_pairs), (2, _edge_pairs)):
        at = np.nonzero(cnt == shared)[0]
        first = eq[at].reshape(-1, 9).argmax(1)
        if shared == 1:
            li = (first // 3)[:, None] + np.arange(3)
            lj = (first % 3)[:, None] + np.arange(3)
        else:
            last = 8 - eq[at].reshape(-1, 9)[:, ::-1].argmax(1)
            li = np.stack([first // 3, last // 3, 3 - first // 3 - last // 3], 1)
            lj = np.stack([first % 3, last % 3, 3 - first % 3 - last % 3], 1)
        singular(_cuda(ti[at]), _cuda(tj[at]), _cuda(li % 3), _cuda(lj % 3), rule)
    l3 = three.expand(nt, 3)
    singular(every, every, l3, l3, lambda Pt, Ps: _same_pairs(Pt))
    mass = g.area[:, None, None] / 24 * (1 + torch.eye(3, device="cuda", dtype=torch.float64))
    L.index_add_(0, (idx[:, :, None] * nv + idx[:, None]).reshape(-1), mass.reshape(-1).to(L.dtype))
    R.index_add_(0, (idx * nt + every[:, None]).reshape(-1),
                 (-0.5 * beta / 3 * g.area[:, None].to(R.dtype)).expand(nt, 3).reshape(-1))
    return L.reshape(nv, nv), R.reshape(nv, nt)


def _exact_galerkin(case, q):
    V, F, k = q["V"], q["F"], case["ka"]
    L, R = _galerkin(V, F, k)
    g = _cuda(q["g"][0]).to(torch.complex128)
    p = _solve(L, (R @ g)[:, None])[:, 0]
    geo = _Geo(V, F)
    at = torch.einsum("qa,ta->tq", _cuda(BARY).to(p.dtype), p[_cuda(F.astype(np.int64))])
    f = _sources_field(k, q["pts"], geo.y.reshape(-1, 3), geo.nrm.repeat_interleave(7, 0),
                       (at * geo.w).reshape(-1, 1), (g[:, None] * geo.w).reshape(-1, 1))
    return p, f[:, 0]


def _padded(idx, x, n, draws):
    """Samples, as many as there are, in buffers of a fixed size."""
    rest = draws // 2 + 64 - len(idx)
    return np.pad(idx, (0, rest), constant_values=-1), *(torch.nn.functional.pad(a, (0, 0, 0, rest)) for a in (x, n))


def _exact_sampler(case, rng):
    """Grid dart throwing in 27 phases, as the sampler defines it, one cell after another."""
    V, F, u, radius = _draws(case["tri"], case["draws"], rng)
    x, n = _candidates(V, F, u)
    lo, h = V.min(0), radius / math.sqrt(3.0)
    dims = np.floor((V.max(0) - lo) / h).astype(int) + 1
    cells = np.clip(np.floor((x - lo) / h).astype(int), 0, dims - 1)
    phase = (cells % 3) @ np.array([9, 3, 1])
    order = np.lexsort((np.arange(len(x)), cells[:, 2], cells[:, 1], cells[:, 0], phase))
    around = list(itertools.product(range(-2, 3), repeat=3))
    taken = {}
    for i in order:
        c = tuple(cells[i])
        if c in taken:
            continue
        near = [taken[q] for q in ((c[0] + a, c[1] + b, c[2] + d) for a, b, d in around) if q in taken]
        if not near or ((x[near] - x[i]) ** 2).sum(1).min() >= radius * radius:
            taken[c] = i
    keep = np.sort(np.array(list(taken.values())))
    return _padded(keep, torch.from_numpy(x[keep]), torch.from_numpy(n[keep]), len(x))


def _exact_training(case, q):
    k, u = case["ka"], q["u"]
    th, ph = np.pi * u[:, 0], 2 * np.pi * u[:, 1]
    r = 1.5 * q["rb"] + 1.5 * q["rb"] * u[:, 2]
    x = q["center"] + r[:, None] * np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)
    p, g = (_cuda(q[c]).to(torch.complex128) for c in "pg")
    amp = _field(q["V"], q["F"], k, x, p, g)[0].abs()
    geo, far = _Geo(q["V"], q["F"]), []
    for d in _cuda(q["dirs"]).split(64):
        phase = torch.polar(geo.w / (4 * math.pi), torch.zeros_like(geo.w)) * torch.exp(-1j * k * (geo.y @ d.T).permute(2, 0, 1))
        far.append((phase.sum(-1) * (-1j * k * (d @ geo.nrm.T) * p - g)).sum(1))
    return np.stack([th, ph, r], 1), amp, torch.cat(far)


def _exact_field(case, seed):
    prm, x = _field_inputs(case, seed)
    T = 1 << case["table"]
    tables, W, b = ([_cuda(a).double() for a in prm[c]] for c in ("tables", "weights", "biases"))
    out = []
    for xs in x.split(1 << 18):
        xs, enc = xs.double(), []
        for t, n in zip(tables, LEVELS):
            p = xs[:, :3].clamp(0, 1) * n
            i0 = p.floor().clamp(max=n - 1)
            w, i0, f = p - i0, i0.long(), 0
            for c in itertools.product((0, 1), repeat=3):
                i, j, l = (i0[:, a] + c[a] for a in range(3))
                at = i + (n + 1) * (j + (n + 1) * l) if (n + 1) ** 3 <= T else (i ^ (j * 2654435761) ^ (l * 805459861)) % T
                f = f + t[at] * torch.stack([w[:, a] if c[a] else 1 - w[:, a] for a in range(3)]).prod(0)[:, None]
            enc.append(f)
        for a in range(3, xs.shape[1]):
            for l in range(6):
                enc += [torch.sin(2.0 ** l * math.pi * xs[:, a:a + 1]), torch.cos(2.0 ** l * math.pi * xs[:, a:a + 1])]
        h = torch.cat(enc, 1)
        h = torch.nn.functional.pad(h, (0, WIDTH - h.shape[1]))
        for l in range(4):
            h = (h @ W[l].T + b[l]).clamp(min=0)
        out.append(h @ W[4].T + b[4])
    return torch.cat(out)


def exact(case, seed):
    rng, kind = np.random.default_rng(seed), case["kind"]
    if kind in ("sweep", "galerkin"):
        q = _problem(case["tri"], case["ka"], case.get("nrhs", 1), case["points"], rng)
        if kind == "galerkin":
            return _exact_galerkin(case, q)
        p, f = _exact_problem(q)
        return (p, f) if case["nrhs"] > 1 else (p[0], f[0])
    if kind == "mc":
        q = _mc_inputs(case, rng)
        L, R = _samples_system(q["Y"], q["N"], q["area"], case["ka"])
        g = _cuda(q["g"]).to(torch.complex128)[:, None]
        p, w = _solve(L, R @ g), q["area"] / len(q["Y"])
        return p[:, 0], _sources_field(case["ka"], q["pts"], _cuda(q["Y"]), _cuda(q["N"]), w * p, w * g)[:, 0]
    if kind == "sampler":
        return _exact_sampler(case, rng)
    if kind in ("fused", "requests"):
        return [_exact_problem(q) for q in _jobs(case, rng)]
    if kind == "training":
        return _exact_training(case, _training_inputs(case, rng))
    return _exact_field(case, seed)
