"""Parked searches of a batch that go through several group launches.

A group that parks leaves its last command (to leave) and its barrier's arrivals
in the slot's state.  In the next launch the group's first CTA resets them; a CTA
of the group that read the state before that would take the old command for its
own and leave, and the search would end at its next grid barrier.  So the others
wait for the group's release word, which the host zeroes before each launch.
"""
import os
import re

import pytest

import paper_2305_18575_gb300 as rei
from workloads import type2_instance

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_18575_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as fh:
        return fh.read()


def test_a_groups_other_ctas_wait_for_the_reset_state():
    """The order in the kernel: reset, fence, release; the others acquire the
    release before the search's first read of the state."""
    text = source("slots.cu")
    body = text[text.index("k_solve_groups("):]
    body = body[: body.index("\n}\n")]
    reset, fence = body.index("st->cmd_seq = 0"), body.index("__threadfence()")
    give = body.index("atomicExch(&G.release[g]")
    take, search = body.index("ld_acquire_u64(&G.release[g])"), body.index("solve_body<")
    assert reset < fence < give < search and take < search
    assert re.search(r"if \(!s_go\) return;", body[:search])


def test_every_group_launch_starts_with_zeroed_release_words():
    """Both callers zero the words in the copy that brings the groups, on the
    launch's own stream, before the launch."""
    text = source("host.cu")
    launches = [m.start() for m in re.finditer(r"\blaunch_solve_groups\(\(|\blaunch_solve_groups\(S->", text)]
    assert len(launches) == 2
    for at in launches:
        before = text[max(0, at - 4000): at]
        zero = before.rindex("memset(gidx + 2 * ng, 0, 8ull * ng)")
        copy = before.rindex("cudaMemcpyAsync(c->g_idx.p, gidx, 16ull * ng")
        assert zero < copy and "G.release = (unsigned long long *)c->g_idx.p + ng;" in before


@pytest.mark.gpu
@pytest.mark.parametrize("n", [40, 170])
def test_searches_through_several_group_launches_match_plain_solves(n):
    """Searches of some 10^5 candidates, all parked at once, on 7 CTAs and on one
    or two each: far more than a first launch's allowance."""
    insts = [type2_instance(s, 8, 8, 6) for s in range(n)]
    probs = [rei.Problem(i.alphabet, i.pos, i.neg, max_cost=12) for i in insts]
    with rei.Context(device=0) as ctx:
        plain = [ctx.solve_problem(p) for p in probs]
        batch = ctx.solve_batch(probs, warps_per_cta=8, yield_us=1)
        again = ctx.solve_batch(probs, warps_per_cta=8, yield_us=1)  # the slots used again
    for k, (a, b, c) in enumerate(zip(plain, batch, again)):
        for g in (b, c):
            assert (g.status, g.cost, g.tree, g.candidates, g.unique) == \
                (a.status, a.cost, a.tree, a.candidates, a.unique), k
    # (one search launch in the batch and one a group launch; the staging launch beside them)
    rounds = [r.search_launches - 1 for r in batch if r.launches == r.search_launches + 1]
    assert sum(r >= 2 for r in rounds) >= 10, rounds
