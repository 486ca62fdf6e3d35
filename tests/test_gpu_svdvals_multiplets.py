"""ctm_svdvals_noalloc on spectra with close singular values: all within s of
one value (columns whose overlaps are tiny from the start and whose rotations
are by any angle), and multiplets of 3 to 8 values split by s, dense and as the
blocks of a permuted block-diagonal matrix (the corners of states with a
symmetry). Reference: torch.linalg.svdvals in 64 bits.

Tolerance as in test_gpu_svdvals.py: 50 k eps of the largest singular value.
"""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(8, False), (8, True), (37, False), (37, True), (64, False), (64, True), (96, True),
         (128, False)]


def _unitary(g, k, cplx):
    M = torch.randn(k, k, dtype=torch.complex128 if cplx else torch.float64, generator=g)
    return torch.linalg.qr(M)[0]


def _check(M):
    k, cplx = M.shape[0], M.is_complex()
    a = M.cuda().contiguous()
    s = torch.empty(k, dtype=torch.float64, device="cuda")
    pkg.ctm_svdvals_noalloc(a.data_ptr(), k, pkg.CTM_C128 if cplx else pkg.CTM_F64, s.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    ref = torch.linalg.svdvals(M)
    tol = 50 * k * np.finfo(float).eps * float(ref[0])
    assert float((s.cpu() - ref).abs().max()) <= tol


@pytest.mark.parametrize("k,cplx", SIZES)
@pytest.mark.parametrize("split", [1e-11, 1e-10, 1e-9, 3e-9, 1e-8])
def test_one_cluster(k, cplx, split):
    g = torch.Generator().manual_seed(k)
    s = 1.0 + split * torch.rand(k, dtype=torch.float64, generator=g)
    U, V = _unitary(g, k, cplx), _unitary(g, k, cplx)
    _check((U * s) @ V.conj().T)


@pytest.mark.parametrize("k,cplx", SIZES)
@pytest.mark.parametrize("size", [3, 4, 8])
@pytest.mark.parametrize("split", [1e-11, 1e-9])
@pytest.mark.parametrize("blocks", [False, True])
def test_multiplets(k, cplx, size, split, blocks):
    g = torch.Generator().manual_seed(1000 * size + k)
    level = torch.arange(k) // size
    s = torch.exp(-4.0 * size * level / k) * (1.0 + split * torch.rand(k, dtype=torch.float64,
                                                                       generator=g))
    if not blocks:
        _check((_unitary(g, k, cplx) * s) @ _unitary(g, k, cplx).conj().T)
        return
    M = torch.zeros(k, k, dtype=torch.complex128 if cplx else torch.float64)
    for i in range(0, k, size):
        m = min(size, k - i)
        M[i:i + m, i:i + m] = (_unitary(g, m, cplx) * s[i:i + m]) @ _unitary(g, m, cplx).conj().T
    p = torch.randperm(k, generator=g)
    _check(M[p][:, p])
