"""Searches of a batch that outgrow their slots continue side by side, each launch on
a share of the GPU.  CTAs of a launch wait for each other, so all of the launches
must fit the GPU together wherever their CTAs lie, also when some widths' CTAs fill an
SM and others' half of one: together they may have at most one CTA an SM."""
import pytest

import paper_2305_18575_gb300 as rei
from workloads import type1_instance, type2_instance

pytestmark = pytest.mark.gpu

SLOT_ROWS = 1 << 18


def outgrowing(n):
    """Searches over |ic| up to 30, 36 - 42 and 60 - 80 (1, 2 and 4 words) that cache
    more languages than a slot holds."""
    kinds = [lambda s: (type1_instance(s, 12, 12, 4), 17), lambda s: (type1_instance(s, 10, 10, 5), 15),
             lambda s: (type2_instance(s, 11, 11, 7), 14)]
    out = []
    for s in range(n):
        i, top = kinds[s % 3](s)
        out.append(rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top, mem_budget=8 << 30))
    return out


@pytest.mark.parametrize("n", [5, 16])
def test_launches_side_by_side_fit_the_gpu_together(n):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    probs = outgrowing(n)
    with rei.Context(device=0) as ctx:
        plain = [ctx.solve_problem(p) for p in probs]
        batch = ctx.solve_batch(probs, warps_per_cta=8, chunk=4096)
    for k, (a, b) in enumerate(zip(plain, batch)):
        assert (a.status, a.cost, a.tree, a.candidates, a.unique) == \
            (b.status, b.cost, b.tree, b.candidates, b.unique), k
    grown = [b for b in batch if b.unique > SLOT_ROWS]
    assert len(grown) >= 4 and len({b.words for b in grown}) == 3
    side_by_side = min(len(grown), 8)
    assert all(b.grid * side_by_side <= sms for b in grown), [(b.words, b.grid) for b in grown]
