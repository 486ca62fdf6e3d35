"""A context on the caller's stream, on which another thread keeps launching: what
that thread enqueues runs exactly once, also while the context records its moves
as graphs and when it replays them, and the moves are not disturbed."""
import threading

import numpy as np
import pytest

import ctm_synth as S
import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _solve(stream):
    A = S.ipeps_tensors(2, 1, 2, 2, bond_decay=0.6)
    ctx = pkg.ctm_init(2, 1, [np.array(a.real) for a in A], 2, 2, 8, cplx=False,
                       opts=pkg.ctm_default_opts(warmup_iters=1, stream=stream))
    for _ in range(6):
        ctx.ctm_converge(0.0, 1)
    state, moves = ctx.ctm_save(), ctx.ctm_debug_moves()
    ctx.ctm_free()
    return state, moves


def test_launches_of_another_thread_on_the_same_stream():
    alone = _solve(None)
    assert alone[1] == (8, 16)
    s = torch.cuda.Stream()
    count = torch.zeros(1, dtype=torch.int64, device="cuda")
    one = torch.ones(1, dtype=torch.int64, device="cuda")
    count.add_(one)                    # (the first launch loads the kernel)
    count.zero_()
    torch.cuda.synchronize()
    stop, added = threading.Event(), [0]

    def launch():
        with torch.cuda.stream(s):
            while not stop.is_set():
                count.add_(one)
                added[0] += 1

    t = threading.Thread(target=launch)
    t.start()
    try:
        for _ in range(10):
            assert _solve(s.cuda_stream) == alone
    finally:
        stop.set()
        t.join()
    s.synchronize()
    assert added[0] > 0 and int(count) == added[0]
