"""Moves replayed from their graphs against moves run directly: two contexts
of the same problem, one with profiling on (which runs every move directly),
must hold the same environment and rangefinders bit for bit after every
iteration. The cases cover one and several lanes, the three arithmetics, dead
columns (a product state, whose repair directions depend on the count of QRs
so far), buffers that grow between moves (an observable in split precision),
a restored checkpoint, and a switch between split and exact-digit moves.
"""
import numpy as np
import pytest

import ctm_synth as S
import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu


def _pair(Lx, Ly, D, chi, cplx, **kw):
    out = []
    for _ in range(2):
        A = (S.product_state_tensors(Lx, Ly, complex_=cplx) if D == 1 else
             S.ipeps_tensors(Lx, Ly, 2, D, complex_=cplx, bond_decay=0.6))
        out.append(pkg.ctm_init(Lx, Ly, [np.array(a) if cplx else a.real for a in A], 2, D, chi,
                                cplx=cplx, opts=pkg.ctm_default_opts(warmup_iters=1, **kw)))
    out[1].ctm_profile_enable(True)
    return out


def _same(a, b):
    sa, sb = a.ctm_save(), b.ctm_save()
    assert sa == sb


@pytest.mark.parametrize("Lx,Ly,D,chi,cplx,kw", [
    (1, 1, 2, 8, False, {}),
    (1, 1, 1, 4, True, {}),                                   # rank one: dead columns
    (2, 3, 2, 6, True, {}),
    (3, 3, 2, 5, False, dict(si_rounds=2)),
    (1, 2, 3, 7, True, dict(prec=pkg.CTM_PREC_SPLIT_BF16)),
    (2, 1, 2, 9, False, dict(prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=float("inf"))),
    (1, 1, 2, 8, True, dict(si_coupled=1)),
])
def test_replayed_moves_equal_direct_ones(Lx, Ly, D, chi, cplx, kw):
    a, b = _pair(Lx, Ly, D, chi, cplx, **kw)
    for it in range(5):
        for c in (a, b):
            c.ctm_converge(0.0, 1)
            if it == 3:
                c.ctm_rdm2(0, 0, 0)
        _same(a, b)
    for r in (2, 0, 0, 1):
        a.ctm_move(r)
        b.ctm_move(r)
        _same(a, b)
    assert a.ctm_si_stats() == b.ctm_si_stats()
    state = a.ctm_save()
    a.ctm_converge(0.0, 2)
    a.ctm_load(state)
    a.ctm_converge(0.0, 1)
    b.ctm_converge(0.0, 1)
    _same(a, b)


def test_refinement_switches_between_recorded_moves():
    a, b = _pair(1, 1, 2, 8, False, prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=1e-3)
    for _ in range(3):
        for c in (a, b):
            c.ctm_converge(0.0, 8)
        _same(a, b)
