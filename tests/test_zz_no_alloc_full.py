"""rei_solve_noalloc with so large a budget that its array has no room left for the chunk
plans: every CTA plans each chunk then.  (Collected last, as test_zz_no_alloc.py.)"""
import pytest

import paper_2305_18575_gb300 as rei
from workloads import type2_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per,length,n_ic,top", [(6, 6, 25, 13), (6, 6, 40, 13), (10, 7, 70, 12), (13, 9, 129, 11)])
def test_without_room_for_the_plan(per, length, n_ic, top):
    """Searches of some 10^5 candidates, most of them in chunks of the whole grid."""
    i = next(i for i in (type2_instance(s, per, per, length) for s in range(20000)) if i.n_ic == n_ic)
    words = 1 if n_ic <= 32 else 2 if n_ic <= 64 else 4 * ((n_ic + 127) // 128)

    def problem(cap):
        return rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top, mem_budget=cap * (4 * words + 28))

    def noalloc(cap):
        buf, prob = rei._OutBuf(), problem(cap)
        return buf.result(rei.rei_solve_noalloc(prob.p, None, buf.res))

    # the largest cache the array holds: fewer than five arrays' alignment (1280 bytes) are
    # left, and a plan of these costs takes more than 2000
    lo, hi = 1000, 1 << 22
    assert noalloc(lo).status != rei.REI_ESCRATCH and noalloc(hi).status == rei.REI_ESCRATCH
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if noalloc(mid).status == rei.REI_ESCRATCH:
            hi = mid
        else:
            lo = mid
    with rei.Context(device=0) as ctx:
        want = ctx.solve_problem(problem(lo))
    assert want.candidates > 40000
    for _ in range(2):
        got = noalloc(lo)
        assert (got.status, got.cost, got.tree, got.candidates, got.unique, got.levels) == \
            (want.status, want.cost, want.tree, want.candidates, want.unique, want.levels)
