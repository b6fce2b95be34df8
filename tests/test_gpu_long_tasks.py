"""Complex128 sweep tasks of 128 and 256 rows and of two and four column blocks (csrc/sweeps64.cu: npass,
ncol; k_to_digits with several row blocks per task), which a level takes once it has enough tasks for
three waves: 117,649 dofs in 32 subdomains, with supernodes up to 33, 65, 100 and 112 wide (a last
block of one column, of four, full ones; last row blocks of any size).

Against sweep_tasks=1, 64 rows and one column block on every level, which test_gpu_variants compares
with the oracle: a row's sum and, for the same chunk, a column's are the same exact sums, so with
backward chunks of at most 64 rows (all levels the same) M^{-1} v is the same bit for bit.  With longer
ones the sparse levels' chunks differ from the forced ones and with them the rounding: 1e-12, some
10^3 (the condition) times 2^-53.  The shapes a level takes are read from hz_plan's log."""
import os
import re
import subprocess
import sys

import pytest

import synth

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CONFIGS = [dict(max_snode=33, leaf_size=33, bwd_chunk=34), dict(max_snode=65, leaf_size=65, bwd_chunk=64),
           dict(max_snode=100, leaf_size=100, bwd_chunk=512), dict(bwd_chunk=64), dict()]
MODEL = "synth.unit_cube_problem(n=24, order=2, nsub=32, overlap=1, freq=1.5)"


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


@pytest.fixture(scope="module")
def problem():
    return eval(MODEL)


@pytest.fixture(scope="module")
def shapes(hzmod):
    """Per configuration: levels of 128- and 256-row tasks and of two and four column blocks."""
    code = (f"import sys, synth\nfrom paper_2004_06309_gb300 import hz\np = {MODEL}\n"
            f"for kw in {CONFIGS!r}:\n    print('config', file=sys.stderr, flush=True)\n    hz.plan(p, **kw)\n")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, HZ_VERBOSE="1", PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stderr
    out = []
    for part in r.stderr.split("config\n")[1:]:
        a, b, c, d, e, f, g = map(int, re.search(r"sweep tasks: .* rows (\d+)/(\d+)/(\d+)/(\d+), .* blocks "
                                                 r"(\d+)/(\d+)/(\d+)", part).groups())   # the solve tree's come first
        out.append((c, d, f, g))
    return out


def test_every_shape_is_taken(shapes):
    assert all(max(s) > 0 for s in shapes)
    assert all(any(s[q] > 0 for s in shapes) for q in range(4)), shapes


@pytest.mark.parametrize("i", range(len(CONFIGS)))
def test_same_as_short_tasks(hzmod, problem, shapes, i):
    import torch
    kw = CONFIGS[i]
    assert shapes[i][0] + shapes[i][1] > 0 and shapes[i][2] + shapes[i][3] > 0
    z = []
    for sweep in (0, 1):
        G = hzmod.Solver(problem, sweep_tasks=sweep, spmv_lanes=8, **kw)
        G.factor()
        v = torch.randn(G.n, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(9))
        z.append(G.apply_M(v).clone())
        G.close()
    if 0 < kw.get("bwd_chunk", 0) <= 64:
        assert torch.equal(z[0], z[1])
    else:
        assert torch.linalg.vector_norm(z[0] - z[1]) <= 1e-12 * torch.linalg.vector_norm(z[1])
