"""Corner x block products (ctm_corner_apply: the contractions of an enlarged
corner, its absorption of A and conj(A), and the product with an N x k block)
against a NumPy contraction of the same seeded tensors, at the sizes where the
fp64 kernels can go wrong: one tile and less, ragged rows and columns, K
splits that do not divide evenly among the CTAs of a cluster, and every
geometry of the fused absorption.

Every value is a chain of four fp64 sums of lengths chi, chi, D^2 and d D^2,
then one of length N, so its error is at most (sum of the lengths + 5) eps
times the same contraction of absolute values (each complex multiply-add
counts as two real ones, hence the factor 2); the tolerance is that bound.
"""
import numpy as np
import pytest

import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu


def _normal(rng, shape, cplx):
    x = rng.standard_normal(shape)
    return x + 1j * rng.standard_normal(shape) if cplx else x


def _corner(A, B, C, Ta, Tb):
    x = np.einsum("pm,mnuv->pnuv", C, Ta)
    x = np.einsum("tplw,pnuv->tlwnuv", Tb, x, optimize=True)
    x = np.einsum("tlwnuv,sulde->twnvsde", x, A, optimize=True)
    x = np.einsum("twnvsde,svwDE->tdDneE", x, B, optimize=True)
    n = x.shape[0] * x.shape[1] * x.shape[2]
    return x.reshape(n, n)


@pytest.mark.parametrize("d,D,chi,p,cplx", [
    (2, 2, 1, 5, False),     # N = k = 4: less than one tile
    (2, 2, 8, 5, False),     # N = 32, k = 13
    (2, 2, 9, 5, True),      # N = 36, k = 14
    (1, 3, 10, 5, True),     # N = 90, d = 1
    (2, 3, 27, 5, False),    # N = 243: four K splits
    (2, 3, 33, 5, True),     # N = 297: five K splits on three CTAs
    (3, 4, 17, 4, False),    # N = 272, d = 3, D = 4
    (2, 4, 9, 2, True),      # D = 4 complex
    (2, 5, 11, 5, False),    # N = 275, D = 5
    (2, 5, 5, 5, True),
    (2, 6, 7, 5, False),     # D = 6
    (2, 6, 5, 1, True),
    (2, 7, 4, 3, False),     # D = 7, 8: one pair per block
    (2, 8, 3, 3, False),
])
@pytest.mark.parametrize("herm", [False, True])
def test_corner_apply_fp64(d, D, chi, p, cplx, herm):
    rng = np.random.default_rng(100 * D + chi)
    A = _normal(rng, (d, D, D, D, D), cplx)
    C = _normal(rng, (4, 1, chi, chi), cplx)
    T = _normal(rng, (4, 1, chi, chi, D, D), cplx)
    ctx = pkg.ctm_init(1, 1, [A], d, D, chi, cplx=cplx, opts=pkg.ctm_default_opts(p=p))
    ctx.ctm_set_env(C, T)
    Z = _normal(rng, (ctx.N, ctx.k), cplx)
    out = ctx.ctm_corner_apply(0, 0, 0, 1, Z, herm=herm)
    ctx.ctm_free()
    Q = _corner(A, A.conj(), C[0, 0], T[0, 0], T[3, 0])
    Qa = _corner(abs(A), abs(A), abs(C[0, 0]), abs(T[0, 0]), abs(T[3, 0]))
    ref = (Q.conj().T if herm else Q) @ Z
    bound = (Qa.T if herm else Qa) @ abs(Z)
    n = 2 * chi + D * D + d * D * D + chi * D * D + 5
    tol = (2 if cplx else 1) * n * np.finfo(float).eps
    assert (np.abs(out - ref) <= tol * bound).all(), float((np.abs(out - ref) / bound).max())


# The split-precision corner product over more than 608 (t, n) pairs, at square
# bonds D = 4, 5, 6: the fp32 absorption whose warps copy and multiply side by
# side, with a last group of pairs that is not full and blocks that run one and
# several steps. Each of the three slice products sums at most 8 K blocks of four
# matrix instructions in fp32 and keeps values to a few units of 2^-24 (38 in
# all; tf32: 64 instructions and 12 units, 80 in all); the absorption is two fp32
# sums of D^2 and d D^2 complex terms between three roundings. The tolerance is
# the sum of these times 2^-24 times the contraction of absolute values.
@pytest.mark.parametrize("d,D,chi,p,prec,cplx", [
    (2, 4, 25, 5, "BF16", True),     # 24 pairs a block: fewer blocks than SMs, the last with one pair
    (3, 4, 62, 5, "BF16", False),    # a second step for some blocks
    (2, 5, 25, 5, "BF16", True),     # 12 pairs a block
    (1, 5, 45, 5, "BF16", False),
    (2, 6, 25, 5, "BF16", True),     # 4 pairs a block, two steps
    (2, 6, 37, 5, "BF16", False),    # 1369 pairs: three steps, both X buffers filled again
    (1, 6, 25, 600, "BF16", True),    # 625 columns: more slice products than CTAs
    (1, 6, 26, 600, "TF32", False),
    (1, 5, 25, 3, "TF32", True),      # N = 625: odd, the slices' second half misaligned
])
@pytest.mark.parametrize("herm", [False, True])
def test_corner_apply_split(d, D, chi, p, prec, cplx, herm):
    rng = np.random.default_rng(10 * D + chi)
    A = _normal(rng, (d, D, D, D, D), cplx)
    C = _normal(rng, (4, 1, chi, chi), cplx)
    T = _normal(rng, (4, 1, chi, chi, D, D), cplx)
    opts = pkg.ctm_default_opts(p=p, prec=getattr(pkg, "CTM_PREC_SPLIT_" + prec))
    ctx = pkg.ctm_init(1, 1, [A], d, D, chi, cplx=cplx, opts=opts)
    ctx.ctm_set_env(C, T)
    Z = _normal(rng, (ctx.N, ctx.k), cplx)
    out = ctx.ctm_corner_apply(0, 0, 0, 1, Z, herm=herm)
    ctx.ctm_free()
    a = (A, np.conj(A), C[0, 0], T[0, 0], T[3, 0])
    Q, Qa = _corner(*a), _corner(*map(np.abs, a))
    ref = (Q.conj().T if herm else Q) @ Z
    bound = (4 if cplx else 1) * (Qa.T if herm else Qa) @ np.abs(Z)
    tol = (3 * (38 if prec == "BF16" else 80) + 2 * D * D + 2 * d * D * D + 3) * 2.0 ** -24
    assert np.isfinite(out).all()
    assert np.max(np.abs(out - ref) / bound) < tol


# Exact-digit products: widths of 16, 32, 48 and 64 columns per CTA, one and
# several K blocks (an odd number among them), and more partial sums than CTAs. A
# digit product drops 2^-53 of the row maximum times the column maximum per term
# and sums to 2^-48 relative; of a normal sample the maxima are below twenty times
# the mean product, so 2^-47 of the product of absolute values is a bound.
@pytest.mark.parametrize("M,N,K,op,cplx", [
    (20, 8, 50, 0, False),       # one K block, 8 columns
    (130, 14, 40, 1, True),      # 28 columns, two K blocks
    (300, 69, 333, 2, True),     # 138 columns: three CTAs of 48
    (256, 64, 243, 0, False),    # 64 columns
    (600, 233, 1050, 2, True),   # 466 columns, 33 K blocks: 320 partial sums
])
def test_exact_digit_product(M, N, K, op, cplx):
    rng = np.random.default_rng(M + N)
    opA, B = _normal(rng, (M, K), cplx), _normal(rng, (K, N), cplx)
    A = {0: opA, 1: opA.T, 2: opA.conj().T}[op].copy()
    C = pkg.ctm_gemm_fp64tc(A, B, op)
    assert (np.abs(C - opA @ B) <= 2.0 ** -47 * (np.abs(opA) @ np.abs(B))).all()
