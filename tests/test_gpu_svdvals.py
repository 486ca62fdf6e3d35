"""ctm_svdvals_noalloc against torch.linalg.svdvals in 64 bits at the sizes
where the values-only Jacobi kernel changes (CTAs per matrix, columns per
lane, odd k, the last size before the cooperative kernel and the first after
it) and on the matrices that can trip it: graded, with zero and equal
columns, far from 1 in scale, with entries whose squares leave the range.

A column takes part in k - 1 rotations per sweep and at most a dozen sweeps;
each rotation is orthogonal to a few eps, so the tolerance is 50 k eps of the
largest singular value.
"""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _svdvals(M):
    k, cplx = M.shape[0], M.is_complex()
    a = M.cuda().contiguous()
    s = torch.empty(k, dtype=torch.float64, device="cuda")
    pkg.ctm_svdvals_noalloc(a.data_ptr(), k, pkg.CTM_C128 if cplx else pkg.CTM_F64, s.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    return s.cpu()


def _check(M):
    s, ref = _svdvals(M), torch.linalg.svdvals(M)
    tol = 50 * M.shape[0] * np.finfo(float).eps * float(ref[0])
    assert float((s - ref).abs().max()) <= tol
    assert bool((s[:-1] >= s[1:]).all())


@pytest.mark.parametrize("k,cplx", [(1, False), (2, False), (3, True), (4, False), (5, True),
                                    (8, True), (9, False), (13, False), (17, True), (32, False),
                                    (33, True), (64, False), (65, True), (96, True), (97, True),
                                    (97, False), (128, False), (129, False), (144, False),
                                    (145, False)])
def test_random(k, cplx):
    g = torch.Generator().manual_seed(k)
    _check(torch.randn(k, k, dtype=torch.complex128 if cplx else torch.float64, generator=g))


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("kind", ["graded", "rank1", "zero", "equal", "identity", "big", "small",
                                  "wide"])
def test_special(kind, cplx):
    k = 37
    g = torch.Generator().manual_seed(5)
    M = torch.randn(k, k, dtype=torch.complex128 if cplx else torch.float64, generator=g)
    w = torch.arange(k, dtype=torch.float64)
    if kind == "graded":
        M = M * torch.exp(-w)[:, None] * torch.exp(-w)[None, :]
    elif kind == "rank1":
        M = M[:, :1] @ M[:1, :]
    elif kind == "zero":
        M = torch.zeros_like(M)
    elif kind == "equal":
        M[:, 1::2] = M[:, 0:1]
    elif kind == "identity":
        M = torch.eye(k, dtype=M.dtype)
    elif kind == "big":
        M = M * 2.0**300
    elif kind == "small":
        M = M * 2.0**-300
    else:
        M = M * (10.0 ** (-8 * w))[None, :]   # column norms from 1 to 1e-288
    _check(M)


def test_nan_is_reported():
    M = torch.randn(20, 20, dtype=torch.float64)
    M[3, 4] = float("nan")
    with pytest.raises(pkg.CTMError) as e:
        _svdvals(M)
    assert e.value.status == pkg.CTM_ENUMERIC
