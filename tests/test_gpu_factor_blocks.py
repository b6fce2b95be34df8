"""Blocked pivot-block factorisation (csrc/diag.cu) around its 16-column blocks: supernodes of one
column, below, at and above one and several blocks, in both precisions.

Tolerances: complex128 M^{-1} v to 1e-10 of the oracle's (as in test_gpu_parity); complex64
subdomain factors through a solve to 1e-9, which the FP64 outer iteration verifies, within 1e-6
of the oracle's solution and one iteration of its count (as in test_gpu_variants); the smallest
pivot, which is the same number however the block is cut, to 1e-9 (complex128) across widths."""
import numpy as np
import pytest

import synth
from oracle.solver import OracleSolver

pytestmark = pytest.mark.gpu

WIDTHS = [1, 15, 16, 17, 31, 48, 49, 0]


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


@pytest.fixture(scope="module")
def case():
    p = synth.small_overthrust(levels=2, cells=(6, 6, 3), freq=0.6, nsub=3)
    S = OracleSolver(p)
    S.factor()
    rng = np.random.default_rng(6)
    v = rng.standard_normal(S.n) + 1j * rng.standard_normal(S.n)
    return p, S, v, S.apply_M(v)


@pytest.mark.parametrize("width", WIDTHS)
def test_fp64(hzmod, case, width):
    import torch
    p, S, v, ref = case
    G = hzmod.Solver(p, max_snode=width)
    G.factor()
    z = G.apply_M(torch.from_numpy(v).cuda()).cpu().numpy()
    pivot = G.stats()["min_pivot"]
    G.close()
    assert np.linalg.norm(z - ref) <= 1e-10 * np.linalg.norm(ref)
    G = hzmod.Solver(p, max_snode=7)
    G.factor()
    assert abs(G.stats()["min_pivot"] - pivot) <= 1e-9 * pivot
    G.close()


@pytest.mark.parametrize("width", WIDTHS)
def test_mixed(hzmod, case, width):
    p, S, _, _ = case
    b = S.rhs()[:, 0]
    xo, ito, _, ok = S.solve(b, tol=1e-9)
    G = hzmod.Solver(p, precision=hzmod.HZ_MIXED, max_snode=width)
    G.factor()
    x, info = G.solve(b, tol=1e-9)
    G.close()
    assert ok and info[0][1] == 0 and abs(info[0][0] - ito) <= 1
    assert np.linalg.norm(x - xo) <= 1e-6 * np.linalg.norm(xo)
