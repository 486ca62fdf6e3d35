"""ctm_svdvals_noalloc on matrices whose rows differ so much in scale that every
CTA of a cluster needs the largest exponent of all the others before it starts:
one group of rows of order 2^400, the rest of order 2^-400 (their squares leave
the fp64 range at any scale that a CTA would take from its own rows alone). Two
CTAs to eight, several calls in a row, which must return the same bits.

Tolerance as in test_gpu_svdvals.py: 50 k eps of the largest singular value.
"""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _svdvals(a, cplx):
    k = a.shape[0]
    s = torch.empty(k, dtype=torch.float64, device="cuda")
    pkg.ctm_svdvals_noalloc(a.data_ptr(), k, pkg.CTM_C128 if cplx else pkg.CTM_F64, s.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    return s.cpu()


@pytest.mark.parametrize("k,cplx", [(9, False), (16, True), (17, False), (33, True), (64, False),
                                    (96, True), (128, False)])
def test_scale_of_one_cta_reaches_all(k, cplx):
    g = torch.Generator().manual_seed(k)
    M = torch.randn(k, k, dtype=torch.complex128 if cplx else torch.float64, generator=g)
    for first in (0, k // 2, k - 2):
        A = M * 2.0**-400
        A[first:first + 2] = M[first:first + 2] * 2.0**400
        a = A.cuda().contiguous()
        runs = [_svdvals(a, cplx) for _ in range(20)]
        assert all(torch.equal(runs[0], r) for r in runs[1:])
        ref = torch.linalg.svdvals(A * 2.0**-400) * 2.0**400
        tol = 50 * k * np.finfo(float).eps * float(ref[0])
        assert float((runs[0] - ref).abs().max()) <= tol
