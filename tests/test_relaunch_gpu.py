"""The relaunch's tiles and tables at the edges of the language widths: |ic| of
33 and 62 (2 words, exact keys), 63 and 64 (2 words, fingerprints), 65 and 128
(4 words), 129 (8 words), on one to three CTAs so that chunks are large for the
team (2-word candidates in registers), with ragged chunks, and every cached
language compared with the oracle's.  Whole numbers: no tolerance."""
import functools

import pytest

import oracle
import paper_2305_18575_gb300 as rei
from workloads import type2_instance

pytestmark = pytest.mark.gpu

ST = {oracle.OK: rei.REI_OK, oracle.NOT_FOUND: rei.REI_NOT_FOUND, oracle.OOM: rei.REI_OOM}


@functools.lru_cache(maxsize=None)
def spec(n_ic):
    """The first Type 2 specification over {0,1} with |ic| = n_ic."""
    per, top = (6, 6) if n_ic < 45 else (10, 7) if n_ic < 80 else (13, 9)
    return next(i for i in (type2_instance(s, per, per, top) for s in range(20000)) if i.n_ic == n_ic)


def context(grid, chunk, exact=1, handover=800):
    c = rei.Context(device=0)
    c.set_option(rei.REI_OPT_GRID, grid)
    c.set_option(rei.REI_OPT_CHUNK, chunk)
    c.set_option(rei.REI_OPT_EXACT_KEYS, exact)
    c.set_option(rei.REI_OPT_HANDOVER, handover)
    return c


def same(got, ref):
    assert got.status == ST[ref.status]
    assert (got.candidates, got.unique) == (ref.candidates, ref.unique)
    if ref.status == oracle.OK:
        assert (got.cost, got.tree) == (ref.cost, ref.tree)


@pytest.mark.parametrize("n_ic,grid,chunk,exact", [
    (33, 2, 0, 1), (33, 1, 2500, 1), (62, 3, 0, 1), (62, 2, 5003, 1), (63, 2, 0, 1), (64, 2, 3001, 1), (40, 2, 0, 0),
    (40, 0, 0, 1), (65, 2, 0, 1), (128, 3, 4099, 1), (129, 2, 0, 1)])
def test_relaunch_caches_the_oracles_languages(n_ic, grid, chunk, exact):
    i, top = spec(n_ic), 11 if n_ic < 100 else 10
    run = oracle.Run()
    ref = run.solve(i.alphabet, i.pos, i.neg, max_cost=top)
    with context(grid, chunk, exact) as c:
        got = c.solve_keep(rei.Problem(i.alphabet, i.pos, i.neg, max_cost=top))
        same(got, ref)
        assert got.n_ic == n_ic
        rows, op, left, right, _, _ = c.cache_dump(top + 1)
    for k in range(ref.unique):
        lang, oop, ol, orr = run.cache_entry(k, n_ic)
        assert bytes((rows[k][w >> 5] >> (w & 31)) & 1 for w in range(n_ic)) == lang, k
        assert (op[k], left[k], right[k]) == (oop, ol, orr if orr >= 0 else 0xFFFFFFFF), k


@pytest.mark.parametrize("n_ic,errors", [(25, 1), (40, 1), (63, 5), (70, 2)])
def test_answers_and_full_caches_leave_the_table_empty(n_ic, errors):
    """An answer in a chunk whose languages are marked but not appended, a cache
    that fills within a chunk (OnTheFly and out of memory), then the plain
    search again: one context, every result the oracle's."""
    i = spec(n_ic)
    kinds = [dict(max_cost=13, max_errors=errors), dict(max_cost=11, mem_budget=36 * 3000, flags=rei.REI_F_ONTHEFLY),
             dict(max_cost=11, mem_budget=36 * 2500), dict(max_cost=10)]
    with context(2, 0) as c:
        for kw in kinds + kinds[:1] + kinds[3:]:
            flags = kw.get("flags", 0)
            okw = {k: v for k, v in kw.items() if k != "flags"}
            ref = oracle.solve(i.alphabet, i.pos, i.neg, flags=oracle.F_ONTHEFLY if flags else 0, **okw)
            same(c.solve_problem(rei.Problem(i.alphabet, i.pos, i.neg, **kw)), ref)
