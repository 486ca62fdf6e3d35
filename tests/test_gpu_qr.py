"""CholeskyQR of the rangefinders at the block sizes k where its kernels
change: the factor on one CTA up to k = 97 real / 48 complex, on a cluster of
eight above; with the explicit inverse (split contexts) on one CTA up to
k = 45 / 22; the row solve with one to four columns per lane; and the SVD of rho on
a cluster of one, two, four and eight CTAs up to k = 8, 16, 32 and 64. One move against
the oracle (spectra 1e-9, as for the other single moves), and P_r P_l = I,
which fails at once if a block is not orthonormal.
"""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg
from pairs import make_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,cplx,exact", [
    (6, False, False), (8, False, False), (9, False, False), (16, False, False),
    (17, True, False), (64, True, False), (32, False, False), (33, False, False), (64, False, False),
    (65, False, False), (97, False, False), (98, False, False), (129, False, False),
    (31, True, False), (48, True, False), (49, True, False), (97, True, False),
    (45, False, True), (46, False, True), (22, True, True), (23, True, True), (97, True, True),
])
def test_one_move_at_block_size(k, cplx, exact):
    kw = dict(prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=float("inf")) if exact else {}
    ctx, ref = make_pair(1, 1, 2, 2, k - 5, 5, cplx, 1, warmup_iters=0, **kw)
    assert ctx.k == min(k, ctx.N)
    ctx.ctm_move(0)
    ref.left_move(0)
    spec = ref.spectra()
    for lab in range(4):
        assert np.abs(ctx.ctm_spectrum(0, 0, lab + 1) - spec[lab][0]).max() < 1e-9, lab
    Pl, PrH = ctx.ctm_get_projectors(0, 0, 0)
    assert np.abs(PrH.conj().T @ Pl - np.eye(Pl.shape[1])).max() < 1e-9
    ctx.ctm_free()
