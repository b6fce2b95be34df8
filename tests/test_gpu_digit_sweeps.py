"""Complex128 triangular sweeps in digits (csrc/sweeps64.cu) at the sizes where they can go
wrong: supernodes narrower than one 16-column step, one column past a step, merged ones
wider than one accumulator takes; backward chunks that are no multiple of 16 rows; one, and
4, 8 and 16 right-hand sides.

Tolerances: M^{-1} v to 1e-10 of the oracle's (two direct solvers, as in test_gpu_parity) and
solutions to 1e-9.  A power of two times v only shifts the exponents of the digits, so the
result is that power times M^{-1} v, bit for bit.  An infinity or NaN spoils the subdomains that
hold it and nothing else."""
import numpy as np
import pytest

import synth
from oracle.solver import OracleSolver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


@pytest.fixture(scope="module")
def two_level():
    p = synth.small_overthrust(levels=2, cells=(7, 6, 3), freq=0.7, nsub=5)
    S = OracleSolver(p)
    S.factor()
    rng = np.random.default_rng(3)
    v = rng.standard_normal(S.n) + 1j * rng.standard_normal(S.n)
    return p, S, v, S.apply_M(v)


@pytest.mark.parametrize("kw", [dict(max_snode=5, leaf_size=8), dict(max_snode=16), dict(max_snode=17, bwd_chunk=34),
                                dict(max_snode=33, sweep_tasks=1, bwd_chunk=46), dict(sweep_tasks=2),
                                dict(sweep_tasks=1), dict(sweep_tasks=1, bwd_chunk=512)])
def test_apply_M(hzmod, two_level, kw):
    import torch
    p, S, v, ref = two_level
    G = hzmod.Solver(p, **kw)
    G.factor()
    vd = torch.from_numpy(v).cuda()
    z = G.apply_M(vd)
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
    for e in (-600, 3, 500):
        zs = G.apply_M(vd * 2.0 ** e)
        assert torch.equal(zs, z * 2.0 ** e), e
    assert not torch.any(G.apply_M(torch.zeros_like(vd)))
    G.close()


@pytest.mark.parametrize("slots", [3, 8, 16])
@pytest.mark.parametrize("kw", [dict(), dict(max_snode=17, leaf_size=8)])
def test_slot_solves(hzmod, two_level, slots, kw):
    import torch
    p, S, _, _ = two_level
    top = p.mesh.xyz.max(axis=0)
    rng = np.random.default_rng(slots)
    pts = top * np.stack([rng.uniform(0.1, 0.9, slots + 1) for _ in range(3)], axis=1)
    B = S.rhs(pts)
    G = hzmod.Solver(p, block_size=slots, **kw)
    G.factor()
    X, info = G.solve(torch.from_numpy(B).cuda())
    X = X.cpu().numpy()
    for j in range(slots + 1):
        xo, ito, _, ok = S.solve(B[:, j])
        assert ok and info[j][1] == 0 and abs(info[j][0] - ito) <= 1
        assert np.linalg.norm(X[:, j] - xo) <= 1e-9 * np.linalg.norm(xo)
    G.close()


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_non_finite_right_hand_side_stays_in_its_subdomains(hzmod, bad):
    import torch
    p = synth.unit_cube_problem(n=10, order=2, nsub=6, overlap=1, freq=1.5)
    S = OracleSolver(p)
    S.factor()
    rng = np.random.default_rng(8)
    v = rng.standard_normal(S.n) + 1j * rng.standard_normal(S.n)
    dof = int(S.subs[2].dofs[len(S.subs[2].dofs) // 2])
    G = hzmod.Solver(p)
    G.factor()
    clean = G.apply_M(torch.from_numpy(v).cuda()).cpu().numpy()
    v[dof] = bad
    z = G.apply_M(torch.from_numpy(v).cuda()).cpu().numpy()
    G.close()
    hit = np.zeros(S.n, bool)
    for s in S.subs:
        if dof in s.dofs:
            hit[s.dofs[s.D != 0]] = True
    assert hit.any() and not hit.all()
    assert np.array_equal(z[~hit], clean[~hit])
    assert not np.isfinite(z[hit]).any()
