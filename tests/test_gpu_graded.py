"""Complex128 sweeps (csrc/sweeps64.cu) on right-hand sides whose entries differ by up to 2^40 within a
supernode.  The digits of a task's right-hand side reach 62 bits below its largest entry, which is
less than a double holds of an entry 2^40 below it.

- Dirichlet dofs are decoupled (identity rows and columns), so 2^40 on them must not change the rest
  of M^{-1} v.  Tolerance 1e-10 relative L2, as for two direct solvers in test_gpu_parity; the sums
  that carry the rest are done on the FP64 units then, whose error does not depend on the decoupled
  entries at all.  Left to the digits, the rest was off by 1e-6.
- One subdomain is A^{-1}: the residual |A z - v| of every row within 1e-12 of (|A| |z| + |v|) of that row
  for entries spread over 2^40, at random and along an axis.  A sum that is left to the digits, or what it
  is added to, is at least 2^-14 of its bound, and the digits miss 2^-59 (rms) of this bound per
  column: 2^-45 sqrt(448) = 6e-13 of it for the widest supernode.
- The same bound for random vectors on matrices whose rows differ: wave speeds 10^12 apart from element to
  element, and element layers 10^6 thinner than their neighbours, with the library's own A (its product
  adds 30 entries x 2^-53 per row).  The factorisation scales rows and columns by powers of two for
  this; unscaled, the rows were off by up to 3e-9 of their terms.  Vectors whose solution decays by more
  than about 2^40 within a supernode are outside the bound in such media: the panels hold 62 bits below
  their rows' largest entries.  The smallest pivot stays that of the unscaled matrix."""
import numpy as np
import pytest

import synth
from oracle.solver import OracleSolver

pytestmark = pytest.mark.gpu

SCHEDULES = [dict(), dict(sweep_tasks=1), dict(sweep_tasks=2), dict(sweep_tasks=1, bwd_chunk=34),
             dict(max_snode=17, leaf_size=8)]


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


def _case(levels):
    p = synth.small_overthrust(levels=levels, cells=(7, 6, 3), freq=0.7, nsub=5)
    S = OracleSolver(p)
    fixed = np.zeros(S.n, bool)
    fixed[S.ddofs] = True
    rng = np.random.default_rng(4)
    v = rng.standard_normal((S.n, 17)) + 1j * rng.standard_normal((S.n, 17))
    g = np.where(fixed[:, None], v * 2.0 ** 40, 0.0)
    v[fixed] = 0.0
    return p, fixed, v, v + g


@pytest.fixture(scope="module")
def one_level():
    return _case(1)


@pytest.fixture(scope="module")
def two_level():
    return _case(2)


def _rest_unchanged(z0, z1, fixed):
    assert fixed.any() and not fixed.all()
    assert np.linalg.norm((z1 - z0)[~fixed]) <= 1e-10 * np.linalg.norm(z0[~fixed])


@pytest.mark.parametrize("levels", [1, 2])
@pytest.mark.parametrize("kw", SCHEDULES)
def test_decoupled_entries_leave_the_rest_alone(hzmod, one_level, two_level, levels, kw):
    import torch
    p, fixed, v, g = one_level if levels == 1 else two_level
    G = hzmod.Solver(p, **kw)
    G.factor()
    z0, z1 = (G.apply_M(torch.from_numpy(x[:, 0].copy()).cuda()).cpu().numpy() for x in (v, g))
    G.close()
    _rest_unchanged(z0, z1, fixed)


@pytest.mark.parametrize("slots", [4, 8, 16])
@pytest.mark.parametrize("kw", [dict(), dict(max_snode=17, leaf_size=8)])
def test_decoupled_entries_in_a_batch(hzmod, one_level, slots, kw):
    """One iteration of the batched solve: x = c M^{-1} b with c = 1 to about 2^-80, since M^{-1} is
    the identity on the decoupled dofs, which hold all but 2^-40 of b."""
    import torch
    p, fixed, v, g = one_level
    G = hzmod.Solver(p, **kw)
    G.factor()
    ref = [G.apply_M(torch.from_numpy(v[:, j].copy()).cuda()).cpu().numpy() for j in range(slots)]
    G.close()
    G = hzmod.Solver(p, block_size=slots, **kw)
    G.factor()
    X, info = G.solve(torch.from_numpy(g[:, :slots].copy()).cuda(), tol=1e-6)
    X = X.cpu().numpy()
    G.close()
    assert all(i[0] == 1 and i[1] == 0 for i in info)
    for j in range(slots):
        _rest_unchanged(ref[j], X[:, j], fixed)


@pytest.mark.parametrize("kw", SCHEDULES)
def test_graded_vectors_row_by_row(hzmod, kw):
    import torch
    p = synth.unit_cube_problem(n=9, order=2, nsub=1, overlap=0, freq=1.2, c=1.0 * (1 - 0.5j))
    S = OracleSolver(p)
    rng = np.random.default_rng(5)
    v = rng.standard_normal(S.n) + 1j * rng.standard_normal(S.n)
    X = S.dm.coords()
    G = hzmod.Solver(p, **kw)
    G.factor()
    for e in (rng.uniform(0, 40, S.n), 40 * X[:, 0], 40 * X[:, 2], 40 * (1 - X[:, 2])):
        b = v * 2.0 ** -e
        z = G.apply_M(torch.from_numpy(b).cuda()).cpu().numpy()
        assert np.all(np.abs(S.A @ z - b) <= 1e-12 * (abs(S.A) @ np.abs(z) + np.abs(b)))
    G.close()


def _contrast():
    p = synth.unit_cube_problem(n=8, order=2, nsub=1, overlap=0, freq=1.2)
    p.c = p.c * 10.0 ** np.random.default_rng(1).uniform(-6, 6, len(p.c))
    return p


def _layers():
    p = synth.unit_cube_problem(n=8, order=2, nsub=1, overlap=0, freq=0.3)
    z = np.concatenate([[0.0], np.cumsum([1, 1, 1, 1e-6, 1e-6, 1e-6, 1e-6, 1])])
    a = np.linspace(0.0, 1.0, 9)
    p.mesh = synth.kuhn_box_mesh(a, a, z / z[-1])
    return p


@pytest.mark.parametrize("make", [_contrast, _layers])
@pytest.mark.parametrize("kw", [dict(), dict(max_snode=17, leaf_size=8)])
def test_rows_of_very_different_size(hzmod, make, kw):
    import torch
    p = make()
    S = OracleSolver(p)
    rng = np.random.default_rng(5)
    v = rng.standard_normal(S.n) + 1j * rng.standard_normal(S.n)
    G = hzmod.Solver(p, **kw)
    G.factor()
    z = G.apply_M(torch.from_numpy(v).cuda())
    r = v - G.apply_A(z).cpu().numpy()
    G.close()
    assert np.all(np.abs(r) <= 1e-12 * (abs(S.A) @ np.abs(z.cpu().numpy()) + np.abs(v)))


def test_smallest_pivot_is_the_unscaled_one(hzmod):
    """Of a diagonal-dominated matrix (wave speed 10^-3: -w^2 M) in both precisions, to complex64 rounding."""
    p = synth.unit_cube_problem(n=6, order=1, nsub=3, overlap=1, freq=1.2, c=1e-3 * (1 - 0.01j))
    out = []
    for precision in (hzmod.HZ_FP64, hzmod.HZ_MIXED):
        G = hzmod.Solver(p, precision=precision)
        G.factor()
        out.append(G.stats()["min_pivot"])
        G.close()
    assert abs(out[0] - out[1]) <= 1e-4 * out[1]
