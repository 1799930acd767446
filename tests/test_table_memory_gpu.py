"""A search whose table of exact keys (16 bytes a slot) does not fit the device's memory
goes on with fingerprints (8 bytes) and gives the same result, in no more memory than
slots of 12 bytes would take."""
import pytest

import paper_2305_18575_gb300 as rei
from workloads import type2_instance

pytestmark = pytest.mark.gpu


class Limited(rei.Context):
    """A context whose allocator refuses what would bring it above `limit` bytes."""

    def __init__(self, limit=None):
        import torch
        self.limit, self.held, self.peak = limit, 0, 0

        def alloc(user, nbytes, stream):
            if self.limit is not None and self.held + nbytes > self.limit:
                return None
            self.held += nbytes
            self.peak = max(self.peak, self.held)
            return torch.cuda.caching_allocator_alloc(int(nbytes), 0, int(stream or 0))

        def free(user, ptr, nbytes, stream):
            self.held -= nbytes
            torch.cuda.caching_allocator_delete(ptr)

        self._alloc = rei.rei_alloc(rei.ALLOC_FN(alloc), rei.FREE_FN(free), None)
        self.h = rei.rei_ctx_create(0, self._alloc, torch.cuda.current_stream(0).cuda_stream)
        self._out = rei._OutBuf()


def key(r):
    return (r.status, r.cost, r.tree, r.candidates, r.unique, r.levels)


# initial rows, rows at the end, and the slots of the largest table on the way (the first
# launch's table has four slots a row, the relaunch's two)
@pytest.mark.parametrize("fused,init,slots", [(0, 1 << 18, 1 << 19), (0, 1 << 14, 1 << 19), (1, 1 << 14, 1 << 19),
                                              (1, 1 << 20, 1 << 22)])
@pytest.mark.parametrize("n_ic,seed,top", [(29, 32, 14), (31, 29, 14), (40, None, 13)])
def test_a_table_that_does_not_fit_gives_way_to_fingerprints(n_ic, seed, top, fused, init, slots):
    i = next(i for i in (type2_instance(s, 6, 6, 6) for s in ([seed] if seed else range(20000))) if i.n_ic == n_ic)
    prob = rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top)
    small = rei.Problem(i.alphabet, i.pos, i.neg, max_cost=9)

    def run(limit):
        with Limited(limit) as c:
            c.set_option(rei.REI_OPT_FUSED_STAGE, fused)
            c.set_option(rei.REI_OPT_CACHE_INIT, init)
            c.set_option(rei.REI_OPT_CHUNK, 1 << 18)
            c.set_option(rei.REI_OPT_HANDOVER, 4000)
            got = [key(c.solve_problem(p)) for p in (prob, small, prob)]  # (each leaves the table empty)
            return got, c.peak

    want, peak = run(None)
    assert want[0] == want[2] and want[0][0] != rei.REI_OOM
    assert 1 << 16 < want[0][4] <= 1 << 18
    limit = peak - 4 * slots
    got, less = run(limit)
    assert got == want
    assert less <= limit
