"""A caller's allocator that gives memory at 8-byte boundaries: slots of two words need 16,
so such a context searches with slots of one word, and its results are the same."""
import pytest

import paper_2305_18575_gb300 as rei
from workloads import make_config, type2_instance

pytestmark = pytest.mark.gpu


class Offset(rei.Context):
    """A context whose memory lies 8 bytes behind a 512-byte boundary."""

    def __init__(self):
        import torch

        def alloc(user, nbytes, stream):
            return torch.cuda.caching_allocator_alloc(int(nbytes) + 16, 0, int(stream or 0)) + 8

        def free(user, ptr, nbytes, stream):
            torch.cuda.caching_allocator_delete(ptr - 8)

        self._alloc = rei.rei_alloc(rei.ALLOC_FN(alloc), rei.FREE_FN(free), None)
        self.h = rei.rei_ctx_create(0, self._alloc, torch.cuda.current_stream(0).cuda_stream)
        self._out = rei._OutBuf()


def key(r):
    return (r.status, r.cost, r.tree, r.candidates, r.unique, r.levels)


@pytest.mark.parametrize("fused", [1, 0])
def test_memory_at_8_byte_boundaries(fused):
    """1, 2, 4 and 16 words, a slot per language (|ic| 25) and a hashed one (29), in the first
    launch and handed over from it."""
    sizes = [(6, 6, 25, 12), (6, 6, 29, 12), (6, 6, 40, 12), (10, 7, 70, 11)]
    insts = [(next(i for i in (type2_instance(s, p, p, length) for s in range(20000)) if i.n_ic == n), top)
             for p, length, n, top in sizes]
    insts.append((make_config("wide", 0), 9))
    probs = [rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top) for i, top in insts]
    for handover in (0, 2000):
        with rei.Context(device=0) as a, Offset() as b:
            for c in (a, b):
                c.set_option(rei.REI_OPT_FUSED_STAGE, fused)
                c.set_option(rei.REI_OPT_HANDOVER, handover)
            for k in (0, 1, 2, 3, 4, 2, 0):
                assert key(a.solve_problem(probs[k])) == key(b.solve_problem(probs[k])), k
            assert [key(r)[:5] for r in a.solve_batch(probs)] == [key(r)[:5] for r in b.solve_batch(probs)]
