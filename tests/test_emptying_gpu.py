"""A table emptied in order (256 MiB and more, a row for every 16 slots or fewer, 64 CTAs
or more) with slots of two words: whatever the context solves afterwards finds it empty.
Searches of 3 and 1.2 million languages, without and with an answer (in a chunk whose
languages are marked but not cached), against a table emptied slot by slot."""
import pytest

import paper_2305_18575_gb300 as rei
from workloads import type1_instance

pytestmark = pytest.mark.gpu


def key(r):
    return (r.status, r.cost, r.tree, r.candidates, r.unique, r.levels)


def test_solves_after_an_emptying_in_order_find_the_table_empty():
    i = type1_instance(0, 10, 10, 5)  # |ic| 41
    probs = [rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top, max_errors=errors, mem_budget=8 << 30)
             for top, errors in ((17, 0), (19, 2), (12, 0), (10, 5))]
    with rei.Context(device=0) as by_slot:
        by_slot.set_option(rei.REI_OPT_EXACT_KEYS, 0)  # (one word a slot: 128 MiB at these rows)
        by_slot.set_option(rei.REI_OPT_CACHE_INIT, 1 << 23)
        want = [key(by_slot.solve_problem(p)) for p in probs]
    assert want[0][0] == rei.REI_NOT_FOUND and want[1][0] == want[3][0] == rei.REI_OK
    assert all(16 * w[4] > 1 << 24 for w in want[:2])
    with rei.Context(device=0) as c:
        c.set_option(rei.REI_OPT_CACHE_INIT, 1 << 23)  # (2^24 slots in the relaunch: 256 MiB)
        for order in ((0, 2, 1, 3, 1, 0), (1, 1, 2, 0, 0, 3)):
            for k in order:
                assert key(c.solve_problem(probs[k])) == want[k], (order, k)
