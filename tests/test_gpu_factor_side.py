"""The coarse factorisation on its side stream beside the subdomains' (csrc/capi.cu, factor_both)
against one after the other, which is what runs when the context's limit has no room for both
workspaces.  The kernels and their inputs are the same (spmv_lanes is fixed: left to itself each context
times its own, and the sums' order with it), so M^{-1} v is the same bit for bit; a limit
below the larger workspace is refused as before, and a limit in between is never exceeded."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


@pytest.mark.parametrize("precision", ["HZ_FP64", "HZ_MIXED"])
@pytest.mark.parametrize("default_stream", [False, True])
def test_same_result_within_a_limit(hzmod, precision, default_stream):
    import torch
    p = synth.small_overthrust(levels=2, cells=(7, 6, 3), freq=0.7, nsub=5)
    prec = getattr(hzmod, precision)
    stream = torch.cuda.default_stream() if default_stream else torch.cuda.Stream()
    with torch.cuda.stream(stream):
        def run(limit):
            G = hzmod.Solver(p, precision=prec, hbm_budget=limit, stream=stream, spmv_lanes=8)
            try:
                G.factor()
                v = torch.randn(G.n, dtype=torch.complex128, device="cuda",
                                generator=torch.Generator("cuda").manual_seed(1))
                z = G.apply_M(v).clone()
                st = G.stats()
                G.factor(0.71)                     # another frequency and back, on the same context
                G.factor(0.7)
                assert torch.equal(G.apply_M(v), z)
                return z, st["device_bytes"], st["front_bytes"]
            finally:
                G.close()

        z, held, front = run(0)
        # from no room for a workspace to room for both, in quarters of the larger one's fronts
        outcomes = []
        for k in range(13):
            try:
                zl, h, _ = run(held + k * front // 4)
            except hzmod.HzError as e:
                assert "hbm_budget" in str(e)
                outcomes.append(False)
                continue
            assert h == held and torch.equal(zl, z)
            outcomes.append(True)
        assert not outcomes[0] and outcomes == sorted(outcomes)
    torch.cuda.synchronize()
