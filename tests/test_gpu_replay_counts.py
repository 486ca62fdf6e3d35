"""Which moves are replayed from a graph, and replayed against direct moves for
the kernels that a graph can hold: the fp64 small SVD on one to eight CTAs
(k <= 64) and on a cooperative grid (k > 64), the Cholesky factor on one CTA and
on a cluster of eight, the fp32 pre-solve, slice and digit products.

With one warm-up move per direction the first iteration runs directly, the
second too (a direction is recorded after it has run once past its warm-up with
the same buffers), and all moves from the third on are replays.
"""
import pytest

import paper_2607_15158_gb300 as pkg
from test_gpu_replay import _pair, _same

pytestmark = pytest.mark.gpu

SPLIT = dict(prec=pkg.CTM_PREC_SPLIT_BF16)


@pytest.mark.parametrize("Lx,Ly,D,chi,cplx,kw", [
    (1, 1, 2, 8, False, {}),
    (1, 1, 1, 4, True, {}),
    (2, 3, 2, 6, True, {}),
    (1, 1, 2, 14, False, {}),                 # k = 19: SVD on two CTAs
    (1, 2, 2, 24, True, {}),                  # k = 29: four CTAs, factor on one
    (2, 1, 2, 40, True, {}),                  # k = 45: eight CTAs, factor on a cluster
    (1, 1, 3, 64, True, {}),                  # k = 69: cooperative SVD, factor on a cluster
    (2, 2, 2, 100, False, {}),                # k = 105: the same, real, several lanes
    (1, 1, 3, 64, True, SPLIT),
    (2, 2, 3, 20, True, SPLIT),
    (1, 1, 3, 64, False, dict(SPLIT, split_refine=float("inf"))),
])
def test_moves_past_the_second_iteration_are_replays(Lx, Ly, D, chi, cplx, kw):
    a, b = _pair(Lx, Ly, D, chi, cplx, **kw)
    for it in range(4):
        for c in (a, b):
            c.ctm_converge(0.0, 1)
        _same(a, b)
    assert a.ctm_debug_moves() == (8, 8)
    assert b.ctm_debug_moves() == (16, 0)     # profiling: kernel by kernel
    for r in (2, 0, 0, 1):
        a.ctm_move(r)
        b.ctm_move(r)
    _same(a, b)
    assert a.ctm_debug_moves() == (8, 12)


def test_a_grown_buffer_is_followed_by_one_direct_move_per_direction():
    """An observable in split precision, with a contraction of 2^22 multiply-adds or
    more, grows operand buffers that the recorded
    moves use: each direction runs directly once, then is recorded again."""
    a, b = _pair(1, 2, 3, 32, True, **SPLIT)
    for c in (a, b):
        c.ctm_converge(0.0, 4)
    before = a.ctm_debug_moves()
    assert before == (8, 8)
    for c in (a, b):
        c.ctm_rdm2(0, 0, 0)
        c.ctm_converge(0.0, 3)
    _same(a, b)
    assert a.ctm_debug_moves() == (12, 16)


def test_no_replay_into_a_buffer_that_was_freed_and_could_not_be_replaced():
    """An observable frees an operand buffer of the recorded moves to allocate a
    larger one, and the allocation is refused: the observable fails, the next move
    of each direction runs directly (and allocates again), and the environment goes
    on as in a context that never asked for the observable."""
    a, b = _pair(1, 1, 3, 32, True, **SPLIT)
    for c in (a, b):
        c.ctm_converge(0.0, 4)
    assert a.ctm_debug_moves() == (8, 8)
    pkg.ctm_debug_fail_alloc(0)
    with pytest.raises(pkg.CTMError) as e:
        a.ctm_rdm2(0, 0, 0)
    assert e.value.status == pkg.CTM_ENOMEM
    for c in (a, b):
        c.ctm_converge(0.0, 2)
        c.ctm_rdm2(0, 0, 0)
        c.ctm_converge(0.0, 2)
    _same(a, b)
    direct, replayed = a.ctm_debug_moves()
    assert direct == 16 and replayed == 16
