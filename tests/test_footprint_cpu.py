"""ctm_footprint counts the arrays that a context cannot run without, and not the
helpers on which it runs halves of cuts side by side (they live in the rounding):
the values, in bytes, by which requests have been admitted since before there were
helpers."""
import os

import pytest

import paper_2607_15158_gb300 as pkg
from paper_2607_15158_gb300 import build as B

INF = float("inf")


@pytest.mark.parametrize("cell,cplx,kw,want", [
    ((1, 1, 2, 3, 27), False, {}, 152390733),
    ((2, 2, 2, 3, 33), True, {}, 356778475),
    ((3, 3, 2, 4, 64), False, {}, 878471689),
    ((1, 2, 2, 4, 33), False, dict(prec=pkg.CTM_PREC_SPLIT_TF32), 501986435),
    ((2, 2, 2, 4, 64), True, dict(prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=INF), 3442747988),
    ((3, 3, 2, 6, 144), True, dict(prec=pkg.CTM_PREC_SPLIT_BF16), 39059364111),
    ((1, 1, 2, 8, 256), True, dict(prec=pkg.CTM_PREC_SPLIT_BF16), 147025453805),
    ((2, 2, 2, 3, 18), False, dict(si_coupled=1), 291312285),
    ((2, 2, 2, 3, 18), False, dict(method=pkg.CTM_PROJ_SVD), 147239987),
])
def test_footprint_has_no_helpers(cell, cplx, kw, want):
    if not os.path.exists(pkg.LIB_PATH):
        B.build()
    assert pkg.ctm_footprint(*cell, cplx, pkg.ctm_default_opts(**kw)) == want
