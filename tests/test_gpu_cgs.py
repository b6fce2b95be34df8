"""The orthogonalisation kernels (csrc/cgs.cu) at the edges of their dispatch, against numpy: one to
eight columns per warp (8/9, 16/17, .. columns), warps that share a column's rows (1 to 4 columns),
vectors shorter than a warp, one chunk of rows and one row more, the longest vector whose last block adds
the sums (160 chunks of 64 rows) and one row more, several sub-chunks per block (from 155,649 rows)
and a ragged last one.

Tolerance: a dot is summed by at most 32 lanes x 608 blocks, fewer than 128 additions one after the other
for up to 200,003 rows, so its error is below 128 u |v| |w| < 1.5e-14 |w| for unit v; 64 such
columns come to less than 1e-12 |w|, in h, in the orthogonalised w and in its norm."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

COLUMNS = [1, 2, 3, 4, 5, 8, 9, 16, 17, 24, 25, 32, 33, 40, 41, 48, 49, 56, 57, 64]


@pytest.fixture(scope="module")
def hzmod():
    from paper_2004_06309_gb300 import build, hz
    build.build()
    return hz


def _case(n, seed):
    import torch
    g = torch.Generator("cuda").manual_seed(seed)
    V = torch.randn((64, n), dtype=torch.complex128, device="cuda", generator=g)
    V /= torch.linalg.vector_norm(V, dim=1, keepdim=True)
    return V, torch.randn(n, dtype=torch.complex128, device="cuda", generator=g)


def _expected(V, w):
    h1 = V.conj() @ w
    w = w - h1 @ V
    h2 = V.conj() @ w
    w = w - h2 @ V
    return w, h1 + h2, np.linalg.norm(w)


def _check(V, w0, nc, w, h, norm):
    we, he, ne = _expected(V[:nc].cpu().numpy(), w0.cpu().numpy())
    tol = 1e-12 * float(np.linalg.norm(w0.cpu().numpy()))
    assert np.abs(h.cpu().numpy() - he).max() <= tol
    assert np.linalg.norm(w.cpu().numpy() - we) <= tol
    assert abs(norm - ne) <= tol


@pytest.mark.parametrize("n", [1, 31, 64, 65, 10240, 10241, 38913, 155649, 200003])
def test_without_a_context(hzmod, n):
    import torch
    lib = hzmod.lib()
    V, w0 = _case(n, n)
    p = lambda t: C.c_void_p(t.data_ptr())  # noqa: E731
    for nc in COLUMNS:
        w = w0.clone()
        h = torch.empty(nc, dtype=torch.complex128, device="cuda")
        norm = torch.empty(1, dtype=torch.float64, device="cuda")
        assert lib.hz_cgs2_noalloc(p(V), n, n, nc, p(w), p(h), p(norm),
                                   C.c_void_p(torch.cuda.current_stream().cuda_stream or None)) == hzmod.HZ_OK
        _check(V, w0, nc, w, h, float(norm[0]))


@pytest.mark.parametrize("cells", [(4, 4, 4), (8, 4, 4), (9, 4, 4)])
def test_of_a_context(hzmod, cells):
    """Below and above the vectors whose sums the last block of a pass adds (10,240 rows)."""
    p = synth.small_overthrust(levels=1, cells=cells, freq=0.6, nsub=2)
    G = hzmod.Solver(p)
    V, w0 = _case(G.n, 7)
    for nc in COLUMNS:
        w = w0.clone()
        h, norm = G.cgs2(V[:nc].T, w)
        _check(V, w0, nc, w, h, norm)
    G.close()
