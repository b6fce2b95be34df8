"""What this library is measured on: passes through its public entry points
(``hz.Solver``), from one operator product on the tiny configuration to one right-hand
side of the 5 Hz workload.

A case names a model (the synthetic media of ``synth``), the solver options and the call.
A program builds one context per model and frequency and then runs many vectors or sources
through it, so the context belongs to the model and the seed draws the vectors, the source
positions and, where a pass factorises, the frequency.
"""
import functools
import gc
import itertools
import math

import numpy as np
import torch

import synth
from paper_2004_06309_gb300 import hz

# Defaults of a case's fields: one right-hand side at a time, direct coarse solve, the
# operator in FP64, device buffers, a stream of the program's own (iterations replayed as
# CUDA graphs).
_DEFAULTS = dict(model="overthrust", medium=0, hertz=1.25, cells=0, order=2, nsub=8, overlap=2, levels=2,
                 restart=50, mixed=False, slots=0, rhs=1, columns=0, iterative_coarse=False, host=False,
                 default_stream=False, tol=1e-6, iterations=1)


def _case(name, call, **kw):
    c = dict(_DEFAULTS, call=call, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    tiny = dict(model="cube", cells=12, hertz=1.2, order=1, levels=1, overlap=1, restart=30)   # 2,197 P1 dofs
    sample = dict(hertz=0.625)                     # 9,801 P2 dofs
    small = dict(hertz=1.25, nsub=7)               # 54,925 P2 dofs, ragged parts
    survey = dict(hertz=2.5, nsub=16)              # 349,461 P2 dofs
    return [
        # an outer program's residual check on the smallest model: one short launch
        _case("apply_a_tiny", "apply_a", **tiny),
        # the operator inside another Krylov method, at a survey's size
        _case("apply_a_survey", "apply_a", **survey),
        # one Arnoldi orthogonalisation halfway through a cycle
        _case("cgs2_survey", "cgs2", columns=25, **survey),
        # the preconditioner alone, in both precisions: every local and coarse sweep once
        _case("precond_survey_mixed", "precond", mixed=True, **survey),
        _case("precond_survey_fp64", "precond", **survey),
        # an interactive solve with host buffers on the default stream, one level
        _case("solve_tiny_host", "solve", host=True, default_stream=True, iterations=12, **tiny),
        # a small request of a serving stream: six sources through four slots, FP64
        _case("solve_sample_fp64_slots", "solve", slots=4, rhs=6, iterations=8, **sample),
        # the iterative coarse solve that the large models use, overlap 1
        _case("solve_small_mixed_oras", "solve", mixed=True, iterative_coarse=True, hertz=1.25, overlap=1,
              iterations=12),
        # a batch of a survey's sources: sixteen right-hand sides share every panel read
        _case("solve_survey_mixed_16", "solve", mixed=True, slots=16, rhs=16, iterations=30, **survey),
        # the next frequency of a sweep: factorise, then one source
        _case("frequency_small_fp64", "frequency", iterations=11, **small),
        _case("frequency_survey_mixed", "frequency", mixed=True, iterations=32, **survey),
        # the benchmark's workload: one source on the 5 Hz model (2,368,333 P2 dofs)
        _case("solve_5hz_mixed", "solve", mixed=True, hertz=5.0, nsub=64, iterations=74),
    ]


def draw(rng):
    call = rng.choice(["apply_a", "cgs2", "precond", "precond", "solve", "solve", "solve", "frequency"])
    mixed = rng.random() < 0.6
    levels = rng.choice([1, 2, 2])
    kw = dict(medium=rng.randrange(1000), levels=levels, overlap=rng.choice([1, 2]), mixed=mixed)
    if rng.random() < 0.25:
        order = rng.choice([1, 2])
        cells = 2 * rng.randint(4, 14 if order == 1 else 9)
        kw.update(model="cube", order=order, cells=cells, hertz=round(cells * order / rng.uniform(9.0, 14.0), 3),
                  nsub=rng.randint(2, 9), restart=30)
    else:
        # dofs grow with the cube of the frequency; FP64 factorisations and batches, and the
        # iterative coarse solve, stay below the cost of the largest listed case
        heavy = call == "frequency" or call == "solve"
        top = 1.6 if heavy and not mixed else 2.4
        kw.update(hertz=round(0.5 * (top / 0.5) ** rng.random(), 3))
        n = _ndofs(dict(_DEFAULTS, **kw))
        kw.update(nsub=max(3, min(24, int(n / rng.uniform(3000.0, 22000.0)))))
    if call == "cgs2":
        kw.update(columns=rng.randint(1, 50))
    if call == "solve":
        how = rng.random()
        if how < 0.35:
            s = rng.choice([4, 8, 16])
            kw.update(slots=s, rhs=rng.randint(2, s + s // 2 if s < 16 else 16))
        elif how < 0.5 and levels == 2:
            kw.update(iterative_coarse=True)
            if kw.get("hertz", 0.0) > 1.6 and kw.get("model") != "cube":
                kw.update(hertz=1.6)
        kw.update(host=rng.random() < 0.3, default_stream=rng.random() < 0.2)
    c = _case(None, call, **kw)
    f = max(c["hertz"], 0.3)
    c["iterations"] = int(12 * (f / 1.25) ** 1.35 + 1) if levels == 2 else int(16 * (f / 0.625) ** 0.43)
    return c


def _cells(c):
    return synth.overthrust_cells(c["hertz"])


def _ndofs(c):
    if c["model"] == "cube":
        return (c["cells"] * c["order"] + 1) ** 3
    nx, ny, nz = _cells(c)
    p = 2 * c["order"]
    return (p * nx + 1) * (p * ny + 1) * (p * nz + 1)


# --- the model and the context a program keeps ------------------------------------------

def _model_key(c):
    return tuple(c[k] for k in ("model", "medium", "hertz", "cells", "order", "nsub", "overlap", "levels", "restart"))


@functools.lru_cache(maxsize=2)
def _problem(key):
    model, medium, hertz, cells, order, nsub, overlap, levels, restart = key
    if model == "cube":
        return synth.unit_cube_problem(n=cells, freq=hertz, order=order, nsub=nsub, overlap=overlap, levels=levels,
                                       restart=restart)
    return synth.overthrust_problem(seed=medium, freq=hertz, order=order, nsub=nsub, overlap=overlap, levels=levels,
                                    restart=restart)


_kept = {}


def _solver(c):
    """The factorised context of the case's model: one is kept, as a program works through one
    model's sources before it turns to the next."""
    key = (_model_key(c), c["mixed"], c["slots"], c["iterative_coarse"], c["default_stream"])
    if key not in _kept:
        _kept.clear()
        gc.collect()
        stream = torch.cuda.default_stream() if c["default_stream"] else torch.cuda.Stream()
        G = hz.Solver(_problem(_model_key(c)), precision=hz.HZ_MIXED if c["mixed"] else hz.HZ_FP64, stream=stream,
                      block_size=c["slots"],
                      coarse_solver=hz.HZ_COARSE_ORAS if c["iterative_coarse"] else hz.HZ_COARSE_DIRECT,
                      coarse_tol=0.1 if c["iterative_coarse"] else 0.0)
        G.factor()
        _kept[key] = G
    return _kept[key]


def _sources(c, rng):
    """Source positions: anywhere along the model's top, within the upper fifth of its depth."""
    top = _problem(_model_key(c)).mesh.xyz.max(axis=0)
    return top * np.stack([rng.uniform(0.05, 0.95, c["rhs"]), rng.uniform(0.05, 0.95, c["rhs"]),
                           rng.uniform(0.02, 0.2, c["rhs"])], axis=1)


def _frequency(c, rng):
    return c["hertz"] * rng.uniform(0.96, 1.04) if c["call"] == "frequency" else c["hertz"]


def _vectors(c, rng, n):
    """A Krylov-like vector, and for the orthogonalisation a basis of unit columns (column-major)."""
    g = torch.Generator("cuda").manual_seed(int(rng.integers(1 << 40)))
    v = torch.randn(n, dtype=torch.complex128, device="cuda", generator=g)
    if c["call"] != "cgs2":
        return v, None
    V = torch.randn((c["columns"], n), dtype=torch.complex128, device="cuda", generator=g)
    return v, V / torch.linalg.vector_norm(V, dim=1, keepdim=True)


def prepare(case, seed):
    c = case
    G = _solver(c)
    rng = np.random.default_rng(seed)
    with torch.cuda.stream(G.stream):
        if c["call"] in ("solve", "frequency"):
            f = _frequency(c, rng)
            B = G.point_sources(_sources(c, rng), device=not c["host"])
            return dict(case=c, solver=G, rhs=B[:, 0] if c["rhs"] == 1 else B, hertz=f)
        v, V = _vectors(c, rng, G.n)
        return dict(case=c, solver=G, v=v, V=None if V is None else V.T)


def run(state):
    c, G = state["case"], state["solver"]
    with torch.cuda.stream(G.stream):
        if c["call"] == "apply_a":
            return G.apply_A(state["v"])
        if c["call"] == "cgs2":
            w = state["v"].clone()                  # orthogonalised in place
            h, norm = G.cgs2(state["V"], w)
            return dict(w=w, h=h, norm=norm)
        if c["call"] == "precond":
            z = G.apply_M(state["v"])
            # complex64 subdomain solves: the program keeps its preconditioned basis in complex64
            return z.to(torch.complex64) if c["mixed"] else z
        if c["call"] == "frequency":
            G.factor(state["hertz"])
        X, info = G.solve(state["rhs"], tol=c["tol"])
        return dict(x=X, status=np.array([i[1] for i in info], np.int32))


# --- the work a pass cannot do without ---------------------------------------------------

@functools.lru_cache(maxsize=4)
def _plan(key, mixed, iterative):
    return hz.plan(_problem(key), precision=hz.HZ_MIXED if mixed else hz.HZ_FP64,
                   coarse_solver=hz.HZ_COARSE_ORAS if iterative else hz.HZ_COARSE_DIRECT)


def work(case):
    """One pass's bytes and flops: matrix and factor entries read once per operator product or
    sweep direction whatever the number of right-hand sides, vectors once each; the iteration
    count is the case's typical one."""
    c = case
    s = _plan(_model_key(c), c["mixed"], c["iterative_coarse"])
    n, nnz, r = s["n"], s["nnz"], c["rhs"]
    mat = dict(bytes=20.0 * nnz + 8.0 * n, flops=8.0 * nnz)
    vs = 8 if c["mixed"] else 16
    # a forward and a backward sweep over every factor entry, the vectors of all subdomains
    pre = dict(bytes=2.0 * vs * s["nnz_factor"] + 2.0 * 16 * s["nnz_factor_coarse"],
               flops=16.0 * (s["nnz_factor"] + s["nnz_factor_coarse"]))
    pvec = 2.0 * vs * s["sum_ni"] + 48.0 * n
    if c["levels"] == 2:
        pre = dict(bytes=pre["bytes"] + mat["bytes"], flops=pre["flops"] + mat["flops"])
    if c["call"] == "apply_a":
        return dict(bytes=mat["bytes"] + 32.0 * n, flops=mat["flops"])
    if c["call"] == "cgs2":
        k = c["columns"]
        return dict(bytes=16.0 * n * (k + 2), flops=32.0 * n * k)
    if c["call"] == "precond":
        return dict(bytes=pre["bytes"] + pvec, flops=pre["flops"])
    it = c["iterations"]
    batches = math.ceil(r / max(c["slots"], 1))
    depth = min(it, c["restart"]) / 2.0 + 1.0          # mean columns of the basis
    b = it * (batches * (pre["bytes"] + mat["bytes"]) + r * (pvec + 32.0 * n + 16.0 * n * (depth + 2)))
    f = it * r * (pre["flops"] + mat["flops"] + 32.0 * n * depth)
    if c["call"] == "frequency":
        f += s["factor_flops"]
        b += 40.0 * nnz + 40.0 * s["nnz_local"] + float(vs) * s["nnz_factor"] + 16.0 * s["nnz_factor_coarse"]
    return dict(bytes=b, flops=f)


# --- the same results in 64 bits, from plain numpy and torch -------------------------------

_EDGES = list(itertools.combinations(range(4), 2))


def _reference(order, d):
    """Basis at the points of a product Gauss rule on the d-simplex (exact to degree 4 and
    more), its derivatives by barycentric coordinate, and the rule's weights (sum 1)."""
    x, w = np.polynomial.legendre.leggauss(5)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    grids = np.meshgrid(*([np.arange(5)] * d), indexing="ij")
    idx = [g.ravel() for g in grids]
    lam, rest, wt = [], np.ones(idx[0].size), np.ones(idx[0].size)
    for a in range(d):                                # collapsed coordinates
        t = x[idx[a]]
        lam.append(rest * t)
        rest = rest * (1.0 - t)
        wt = wt * w[idx[a]] * (1.0 - t) ** (d - 1 - a)
    lam = np.stack([rest] + lam, axis=1)
    wt = wt / wt.sum()
    if order == 1:
        return lam, np.broadcast_to(np.eye(d + 1), (len(wt), d + 1, d + 1)), wt
    edges = list(itertools.combinations(range(d + 1), 2))
    phi = [lam[:, i] * (2.0 * lam[:, i] - 1.0) for i in range(d + 1)] + [4.0 * lam[:, i] * lam[:, j] for i, j in edges]
    dphi = np.zeros((len(wt), len(phi), d + 1))
    for i in range(d + 1):
        dphi[:, i, i] = 4.0 * lam[:, i] - 1.0
    for q, (i, j) in enumerate(edges):
        dphi[:, d + 1 + q, i] = 4.0 * lam[:, j]
        dphi[:, d + 1 + q, j] = 4.0 * lam[:, i]
    return np.stack(phi, axis=1), dphi, wt


def _numbering(mesh, order):
    """Dofs of every tet and of every boundary face: vertices, then edges by (min, max) vertex."""
    t, f, nv = mesh.tets.astype(np.int64), mesh.faces.astype(np.int64), len(mesh.xyz)
    if order == 1:
        return t, f, nv
    key = lambda a, i, j: np.minimum(a[:, i], a[:, j]) * nv + np.maximum(a[:, i], a[:, j])  # noqa: E731
    te = np.stack([key(t, i, j) for i, j in _EDGES], axis=1)
    fe = np.stack([key(f, i, j) for i, j in itertools.combinations(range(3), 2)], axis=1)
    u, inv = np.unique(te.ravel(), return_inverse=True)
    return (np.concatenate([t, nv + inv.reshape(te.shape)], axis=1),
            np.concatenate([f, nv + np.searchsorted(u, fe)], axis=1), nv + len(u))


def _operator(p, hertz):
    """A = K - w^2 M - i w B as (rows, columns, values) with identity Dirichlet rows; the mask
    of Dirichlet dofs; the dofs of every tet."""
    w = 2.0 * np.pi * hertz
    td, fd, n = _numbering(p.mesh, p.order)
    X = p.mesh.xyz[p.mesh.tets]
    J = (X[:, 1:] - X[:, :1]).transpose(0, 2, 1)
    vol = np.abs(np.linalg.det(J)) / 6.0
    g = np.linalg.inv(J)                              # gradients of lambda_1..3
    g = np.concatenate([-g.sum(axis=1, keepdims=True), g], axis=1)
    phi, dphi, wt = _reference(p.order, 3)
    mass = np.einsum("q,qa,qb->ab", wt, phi, phi)
    stiff = np.einsum("q,qai,qbj->ijab", wt, dphi, dphi)
    G = np.einsum("eid,ejd->eij", g, g) * vol[:, None, None]
    val = (np.tensordot(G, stiff, axes=([1, 2], [0, 1]))
           - (w * w * vol / p.c ** 2)[:, None, None] * mass)
    # absorbing faces: the speed of the one tet that owns the face
    ab = p.mesh.face_tag == synth.TAG_ABC
    nv = len(p.mesh.xyz)
    fkey = lambda a: (a[:, 0] * nv + a[:, 1]) * nv + a[:, 2]  # noqa: E731
    tf = np.sort(p.mesh.tets.astype(np.int64)[:, [[1, 2, 3], [0, 2, 3], [0, 1, 3], [0, 1, 2]]].reshape(-1, 3), axis=1)
    tk = fkey(tf)
    o = np.argsort(tk)
    face = p.mesh.faces[ab].astype(np.int64)
    own = o[np.searchsorted(tk[o], fkey(np.sort(face, axis=1)))] // 4
    Y = p.mesh.xyz[face]
    area = 0.5 * np.linalg.norm(np.cross(Y[:, 1] - Y[:, 0], Y[:, 2] - Y[:, 0]), axis=1)
    phi2, _, wt2 = _reference(p.order, 2)
    fval = (-1j * w * area / p.c[own])[:, None, None] * np.einsum("q,qa,qb->ab", wt2, phi2, phi2)
    fixed = np.zeros(n, bool)
    fixed[fd[~ab].ravel()] = True
    fa = fd[ab]
    r = np.concatenate([np.repeat(td, td.shape[1], axis=1).ravel(), np.repeat(fa, fa.shape[1], axis=1).ravel()])
    k = np.concatenate([np.tile(td, (1, td.shape[1])).ravel(), np.tile(fa, (1, fa.shape[1])).ravel()])
    v = np.concatenate([val.ravel(), fval.ravel()])
    keep = ~(fixed[r] | fixed[k])
    d = np.nonzero(fixed)[0]
    return (np.concatenate([r[keep], d]), np.concatenate([k[keep], d]),
            np.concatenate([v[keep], np.ones(len(d), complex)])), fixed, td


def _loads(p, pts, fixed, td):
    B = np.zeros((len(fixed), len(pts)), np.complex128)
    X = p.mesh.xyz[p.mesh.tets]
    J = (X[:, 1:] - X[:, :1]).transpose(0, 2, 1)
    for j, x in enumerate(pts):
        lam = np.linalg.solve(J, (x - X[:, 0])[..., None])[..., 0]
        lam = np.concatenate([1.0 - lam.sum(axis=1, keepdims=True), lam], axis=1)
        e = int(np.argmax(lam.min(axis=1)))
        m = lam[e]
        phi = m if p.order == 1 else np.concatenate([m * (2 * m - 1), [4 * m[a] * m[b] for a, b in _EDGES]])
        B[td[e], j] -= phi
    B[fixed] = 0.0
    return B


def exact(case, seed):
    c = case
    n = _ndofs(c)
    solves = c["call"] in ("solve", "frequency")
    if c["call"] == "precond" or (solves and n > 11000):
        return None          # no plain counterpart; a dense solve beyond some 10^4 dofs takes too long
    rng = np.random.default_rng(seed)
    if c["call"] == "cgs2":
        v, V = _vectors(c, rng, n)
        h1 = V.conj() @ v
        w = v - h1 @ V
        h2 = V.conj() @ w
        w = w - h2 @ V
        return dict(w=w, h=h1 + h2, norm=float(torch.linalg.vector_norm(w)))
    p = _problem(_model_key(c))
    (r, k, a), fixed, td = _operator(p, _frequency(c, rng))
    if c["call"] == "apply_a":
        v = _vectors(c, rng, n)[0].cpu().numpy()
        y = a * v[k]
        return torch.from_numpy(np.bincount(r, y.real, n) + 1j * np.bincount(r, y.imag, n))
    A = torch.zeros((n, n), dtype=torch.complex128, device="cuda")
    at = [torch.from_numpy(i).cuda() for i in (r, k)]
    A.index_put_(tuple(at), torch.from_numpy(a).cuda(), accumulate=True)
    B = torch.from_numpy(_loads(p, _sources(c, rng), fixed, td)).cuda()
    X = torch.linalg.solve(A, B)
    return dict(x=X[:, 0] if c["rhs"] == 1 else X, status=None)
