"""The operator product around the line between natural and sorted rows (csrc/capi.cu, spmv_rows): P2 matrices
below and above three windows of 4,096 rows (a last window of 33 rows among them), and a P1 matrix above
it whose rows are alike and stay in order; every number of lanes per row, with and without the residual
form (through a solve's true residual).

Tolerance: rows of at most 65 entries, so 65 x 4 x 2^-53 = 3e-14 of |A| |x|, against the oracle's A."""
import numpy as np
import pytest

import synth
from oracle.solver import OracleSolver

pytestmark = pytest.mark.gpu

MODELS = [lambda: synth.overthrust_problem(seed=0, freq=0.625, nsub=3, overlap=1, restart=30, levels=1),
          lambda: synth.overthrust_problem(seed=0, freq=0.7, nsub=3, overlap=1, restart=30, levels=1),
          lambda: synth.unit_cube_problem(n=26, nsub=8)]


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


@pytest.mark.parametrize("make,n", list(zip(MODELS, [9801, 12321, 19683])))
def test_every_lane_count(hzmod, make, n):
    import torch
    p = make()
    S = OracleSolver(p)
    assert S.n == n
    rng = np.random.default_rng(2)
    x = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    ref, bound = S.A @ x, 3e-14 * (abs(S.A) @ np.abs(x))
    b = S.rhs()[:, 0]
    for lanes in (2, 4, 8, 16):
        G = hzmod.Solver(p, spmv_lanes=lanes)
        G.factor()
        y = G.apply_A(torch.from_numpy(x).cuda()).cpu().numpy()
        xs, info = G.solve(b)
        G.close()
        assert np.all(np.abs(y - ref) <= bound)
        assert info[0][1] == 0
        assert abs(np.linalg.norm(b - S.A @ xs) / np.linalg.norm(b) - info[0][2]) <= 1e-10
