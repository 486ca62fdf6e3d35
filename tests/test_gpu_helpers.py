"""Helpers (the W half of a cut beside its X half): a context has them only while it
stays within its footprint and the device has room, gives them up when it needs the
room itself, and computes the same bits with and without them."""
import numpy as np
import pytest

import ctm_synth as S
import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu

SPLIT = dict(prec=pkg.CTM_PREC_SPLIT_BF16)
EXACT = dict(prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=float("inf"))


def _create(Lx, Ly, D, chi, cplx, kw):
    A = S.ipeps_tensors(Lx, Ly, 2, D, complex_=cplx, bond_decay=0.6)
    opts = pkg.ctm_default_opts(warmup_iters=1, warmup_rounds=2, **kw)
    return pkg.ctm_init(Lx, Ly, [np.array(a) if cplx else a.real for a in A], 2, D, chi, cplx=cplx,
                        opts=opts), pkg.ctm_footprint(Lx, Ly, 2, D, chi, cplx, opts)


@pytest.mark.parametrize("Lx,Ly,D,chi,cplx,kw,helpers", [
    (1, 1, 2, 8, False, {}, 1),
    (3, 3, 2, 6, True, {}, 3),
    (1, 1, 3, 20, True, SPLIT, 1),
    (2, 3, 3, 12, False, SPLIT, 3),
    (2, 2, 3, 12, True, EXACT, 2),
    (1, 1, 3, 20, True, dict(prec=pkg.CTM_PREC_SPLIT_BF16, split_refine=1e-2), 1),
])
def test_refused_helpers_change_nothing(Lx, Ly, D, chi, cplx, kw, helpers):
    """Each allocation of a creation and its first two iterations is refused in turn:
    where it was a helper's, the context runs without helpers and gives the same."""
    ref, cap = _create(Lx, Ly, D, chi, cplx, kw)
    ref.ctm_converge(0.0, 3)
    want = ref.ctm_save()
    used, n = ref.ctm_debug_memory()
    assert n == helpers and used <= cap
    without = 0
    for after in range(400):
        pkg.ctm_debug_fail_alloc(after)
        try:
            ctx, _ = _create(Lx, Ly, D, chi, cplx, kw)
            ctx.ctm_converge(0.0, 3)
        except pkg.CTMError as e:
            assert e.status == pkg.CTM_ENOMEM
            continue
        n = ctx.ctm_debug_memory()[1]
        assert ctx.ctm_save() == want
        ctx.ctm_free()
        if n == helpers:
            break
        assert n == 0
        without += 1
    pkg.ctm_debug_fail_alloc(-1)
    assert without >= 10 * helpers


def test_helpers_are_given_up_when_the_context_needs_the_room():
    """At 1x1, D = 4, chi = 64 the footprint has room for the moves with a helper, and
    for an observable's operands only without it."""
    (a, cap), (b, _) = (_create(1, 1, 4, 64, True, SPLIT) for _ in range(2))
    for c in (a, b):
        c.ctm_converge(0.0, 3)
    assert a.ctm_debug_memory()[1] == 1
    assert a.ctm_debug_moves()[1] > 0          # graphs with a helper's kernels: they go with it
    a.ctm_rdm2(0, 0, 0)
    used, n = a.ctm_debug_memory()
    assert n == 0 and used <= cap
    for c in (a, b):
        c.ctm_converge(0.0, 3)
    assert a.ctm_debug_memory()[1] == 0 and b.ctm_debug_memory()[1] == 1
    assert a.ctm_save() == b.ctm_save()
