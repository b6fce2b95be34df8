"""hz_factor gives its workspaces back however it ends, and a context goes on afterwards.

- A CUDA call that fails on the host: the context's stream is being captured (relaxed mode), where waiting
  for the stream is refused.  Nothing of the factorisation runs on the GPU.
- A subdomain without usable pivots beside a good coarse matrix: with a wave speed of 1e30 A is K to
  rounding, and a subdomain that does not touch the Dirichlet top is a Neumann problem, singular
  by the constants; E keeps the Dirichlet condition.
- The reverse: one free coarse dof, so E = a - w^2 b is one number, zero to rounding at its own resonance
  (real wave speed, Dirichlet all around), where the subdomains' matrices with their impedance
  conditions are not singular.
- Which of the two orders hz_factor takes is read from its log (HZ_VERBOSE): both workspaces before
  the first factor's levels, or one after the other."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from oracle.solver import OracleSolver

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


def _apply(G, seed=2):
    import torch
    v = torch.randn(G.n, dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
    return G.apply_M(v).clone()


def _goes_on(hzmod, G, p, freq, held):
    """The failed hz_factor left nothing behind: same bytes, and the factors of a context of its own."""
    import torch
    G.factor(freq)
    assert G.stats()["device_bytes"] == held
    z = _apply(G)
    H = hzmod.Solver(p, spmv_lanes=8, stream=G.stream)
    H.factor(freq)
    assert torch.equal(_apply(H), z)
    H.close()


@pytest.mark.parametrize("levels", [1, 2])
@pytest.mark.parametrize("precision", ["HZ_FP64", "HZ_MIXED"])
def test_failed_cuda_call(hzmod, levels, precision):
    import torch
    cu = C.CDLL("libcuda.so.1")
    p = synth.small_overthrust(levels=levels, cells=(5, 5, 3), freq=0.6, nsub=4)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        G = hzmod.Solver(p, precision=getattr(hzmod, precision), spmv_lanes=8, stream=stream)
        G.factor()
        held, z = G.stats()["device_bytes"], _apply(G)
        torch.cuda.synchronize()
        for _ in range(2):
            assert cu.cuStreamBeginCapture_v2(C.c_void_p(stream.cuda_stream), 2) == 0
            try:
                with pytest.raises(hzmod.HzError) as e:
                    G.factor()
            finally:
                graph = C.c_void_p()
                cu.cuStreamEndCapture(C.c_void_p(stream.cuda_stream), C.byref(graph))
            assert e.value.status == hzmod.HZ_ERR_CUDA
            assert G.stats()["device_bytes"] == held
        G.factor()
        assert G.stats()["device_bytes"] == held and torch.equal(_apply(G), z)
        G.close()


def test_subdomain_without_pivots_beside_a_good_coarse_matrix(hzmod):
    p = synth.unit_cube_problem(n=8, levels=2, nsub=8, overlap=1)
    good = p.c.copy()
    p.c = np.full(len(p.c), 1e30 + 0j)
    S = OracleSolver(p)
    S.factor()
    assert np.linalg.cond(S.E.toarray()) < 1e8 and np.linalg.cond(S.A.toarray()) < 1e8
    assert max(np.linalg.cond(s.A.toarray()) for s in S.subs) > 1e14
    G = hzmod.Solver(p, spmv_lanes=8)
    held = G.stats()["device_bytes"]
    for _ in range(2):
        with pytest.raises(hzmod.HzError) as e:
            G.factor()
        assert e.value.status == hzmod.HZ_ERR_ZERO_PIVOT
        assert G.stats()["device_bytes"] == held
    G.close()
    p.c = good
    G = hzmod.Solver(p, spmv_lanes=8)
    G.factor()
    assert np.isfinite(_apply(G).cpu().numpy()).all()
    G.close()


def test_coarse_matrix_without_pivot_beside_good_subdomains(hzmod):
    p = synth.unit_cube_problem(n=4, levels=2, nsub=2, overlap=0, c=1.0 + 0j)
    for mesh in (p.mesh, p.coarse):
        mesh.face_tag = np.full(len(mesh.face_tag), synth.TAG_DIRICHLET, np.int8)
    S = OracleSolver(p)
    f0, f1, e = 0.5, 1.0, []
    for f in (f0, f1):
        S.factor(f)
        assert S.E.shape == (1, 1)
        e.append(complex(S.E.toarray()[0, 0]).real)
    b = (e[0] - e[1]) / (f1 ** 2 - f0 ** 2)
    res = float(np.sqrt((e[0] + b * f0 ** 2) / b))
    S.factor(1.01 * res)
    assert max(np.linalg.cond(s.A.toarray()) for s in S.subs) < 1e8
    G = hzmod.Solver(p, spmv_lanes=8)
    held = G.stats()["device_bytes"]
    for _ in range(2):
        with pytest.raises(hzmod.HzError) as err:
            G.factor(res)
        assert err.value.status == hzmod.HZ_ERR_ZERO_PIVOT
        assert G.stats()["device_bytes"] == held
    _goes_on(hzmod, G, p, 0.75 * res, held)
    G.close()


ORDER = """
import sys
import synth
from paper_2004_06309_gb300 import hz
p = synth.small_overthrust(levels=2, cells=(7, 6, 3), freq=0.7, nsub=5)
G = hz.Solver(p, hbm_budget=int(sys.argv[1]), spmv_lanes=8)
G.factor()
st = G.stats()
print(st["device_bytes"], st["front_bytes"])
"""


def _order(limit):
    r = subprocess.run([sys.executable, "-c", ORDER, str(limit)], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, HZ_VERBOSE="1", PYTHONPATH=ROOT))
    assert r.returncode == 0, r.stderr
    steps = ["alloc" if "allocated" in q else "levels" for q in r.stderr.splitlines()
             if "[hz] factor: workspace" in q or ("[hz] factor:" in q and "levels in" in q)]
    return steps, [int(x) for x in r.stdout.split()]


def test_both_orders_run_and_the_limit_decides(hzmod):
    """The smallest limit that is accepted has room for the subdomains' workspace alone."""
    import torch
    p = synth.small_overthrust(levels=2, cells=(7, 6, 3), freq=0.7, nsub=5)

    def run(limit):
        G = hzmod.Solver(p, hbm_budget=limit, spmv_lanes=8)
        try:
            G.factor()
            return _apply(G)
        except hzmod.HzError as e:
            assert e.status == hzmod.HZ_ERR_OOM
            return None
        finally:
            G.close()

    steps, (held, front) = _order(0)
    assert steps == ["alloc", "alloc", "levels", "levels"]            # beside each other
    z = run(0)
    low, high = held, held + 4 * front                                 # refused, accepted
    steps, _ = _order(high)
    assert steps == ["alloc", "alloc", "levels", "levels"]
    assert run(low) is None
    while high - low > 4096:
        mid = (low + high) // 2
        zl = run(mid)
        if zl is None:
            low = mid
        else:
            assert torch.equal(zl, z)
            high = mid
    steps, (h, _) = _order(high)
    assert steps == ["alloc", "levels", "alloc", "levels"] and h == held
