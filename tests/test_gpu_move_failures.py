"""A move whose buffers are refused on the way leaves its lanes and helpers with
work in flight; the context must be usable at once: with the state restored, it
gives what a context gives that never failed, bit for bit. Every allocation of a
first move is refused in turn."""
import numpy as np
import pytest

import ctm_synth as S
import paper_2607_15158_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,refine", [(1, 1, 0.0), (2, 2, 0.0), (1, 2, float("inf"))])
def test_context_goes_on_after_a_refused_buffer(Lx, Ly, refine):
    D, chi = 3, 20

    def create():
        A = S.ipeps_tensors(Lx, Ly, 2, D, complex_=True, bond_decay=0.6)
        return pkg.ctm_init(Lx, Ly, [np.array(a) for a in A], 2, D, chi, cplx=True,
                            opts=pkg.ctm_default_opts(prec=pkg.CTM_PREC_SPLIT_BF16,
                                                      split_refine=refine, warmup_iters=1))
    ref = create()
    state = ref.ctm_save()
    ref.ctm_converge(0.0, 3)
    want = ref.ctm_save()
    refused = 0
    for after in range(200):
        ctx = create()
        pkg.ctm_debug_fail_alloc(after)
        try:
            ctx.ctm_move(0)
        except pkg.CTMError as e:
            assert e.status == pkg.CTM_ENOMEM
            refused += 1
        else:
            pkg.ctm_debug_fail_alloc(-1)
            break
        ctx.ctm_load(state)
        ctx.ctm_converge(0.0, 3)
        assert ctx.ctm_save() == want, after
        ctx.ctm_free()
    assert refused > 3
