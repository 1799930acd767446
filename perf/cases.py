"""Workloads of the REI library as its users run them, through its public calls.

A user has specifications (positive and negative example strings) and wants the
cheapest regular expression of each.  What differs from one use to the next is
the size of a search, not the call: an interactive query ends within a few
hundred candidates, a benchmark specification runs through 10^10 of them.  The
cases cover the five configurations of the repository's own benchmark and tests
(small, medium, wide, batched; the served form's persistent launch has no single
pass to time), the random specifications of the paper's suites (Type 1: strings
uniform over all those up to a length; Type 2: a uniform length first), whose
searches are the deep ones, and the options in use: allowed errors, OnTheFly
mode, device-resident inputs, per-symbol costs, the call that allocates nothing.

Fields of a case
  form      solve (host strings) | device (packed, in device memory) | batch |
            noalloc
  recipe    labelled (strings labelled by a random target expression) | type1 |
            type2
  problems  specifications in one pass (one call each; one call for a batch)
  n_sym, n_pos, n_neg, len_lo, len_hi   the specification; a batch draws
            n_sym, n_pos and n_neg of each problem up to these
  cost_lo, cost_hi   cost of the labelled recipe's target
  costs, sym_costs   cost function, and costs of the symbols ("" = c_sym)
  max_cost, budget_mib, errors, onthefly   as in include/rei.h
"""
import random

import numpy as np
import torch

import paper_2305_18575_gb300 as rei

SYMBOLS = b"0123"


def _case(name, form, recipe, problems, n_sym, n_pos, n_neg, len_lo, len_hi, max_cost, budget_mib, cost_lo=0,
          cost_hi=0, costs="1,1,1,1,1", sym_costs="", errors=0, onthefly=False):
    c = dict(form=form, recipe=recipe, problems=problems, n_sym=n_sym, n_pos=n_pos, n_neg=n_neg, len_lo=len_lo,
             len_hi=len_hi, cost_lo=cost_lo, cost_hi=cost_hi, costs=costs, sym_costs=sym_costs, max_cost=max_cost,
             budget_mib=budget_mib, errors=errors, onthefly=onthefly)
    return dict(c, name=name) if name else c


def listed():
    return [
        # an interactive query, the smallest call: a handful of candidates, all latency
        _case("query_small", "solve", "labelled", 1, 2, 5, 5, 0, 4, 20, 1024, 1, 6),
        # the benchmark's headline: medium specifications one after another, strings from the host
        _case("medium_host", "solve", "labelled", 8, 2, 10, 10, 0, 7, 40, 65536, 10, 14),
        # the same with an expensive star (the headline's second cost vector: searches go several
        # levels deeper), the examples already on the device
        _case("medium_star5_device", "device", "labelled", 4, 2, 10, 10, 0, 7, 40, 65536, 10, 14, costs="1,1,5,1,1"),
        # multiword languages (|ic| 400-500): the wide configuration
        _case("wide_host", "solve", "labelled", 4, 4, 20, 20, 1, 10, 40, 65536, 12, 18),
        # the paper's Type 1 suite at |ic| <= 30, 1-word languages: its hardest rows run 10^9 - 10^10
        # candidates (searched here to cost 26)
        _case("type1_short_deep", "solve", "type1", 1, 2, 12, 12, 0, 4, 26, 65536),
        # Type 1 with strings one longer (|ic| 36-42, 2-word languages), searched to cost 20
        _case("type1_mid_deep", "device", "type1", 1, 2, 10, 10, 0, 5, 20, 16384),
        # Type 1 with longer strings still (|ic| 65-128, 4-word languages)
        _case("type1_long_deep", "solve", "type1", 1, 2, 11, 13, 0, 7, 17, 16384),
        # a random wide specification (|ic| near 1000, 32-word languages) searched to cost 12
        _case("type1_wide_deep", "device", "type1", 1, 4, 20, 20, 0, 10, 12, 16384),
        # noisy examples: two of 24 may be misclassified ("REI with error")
        _case("type2_noisy", "solve", "type2", 2, 2, 12, 12, 0, 6, 17, 8192, errors=2),
        # a small memory budget (16 MiB, about 470 K languages): OnTheFly mode takes over
        _case("type1_onthefly", "solve", "type1", 1, 2, 9, 9, 0, 5, 18, 16, onthefly=True),
        # many uneven specifications at once: the batched configuration
        _case("batch_uneven", "batch", "labelled", 256, 4, 20, 20, 0, 10, 40, 1024, 4, 14),
        # a caller that must not allocate while it solves
        _case("noalloc_medium", "noalloc", "labelled", 4, 2, 10, 10, 0, 7, 40, 16, 10, 14),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["small", "medium", "medium", "wide", "short", "mid", "mid", "long", "deepwide", "noisy",
                       "onthefly", "batch", "batch", "noalloc"])
    host = rng.choice(["solve", "device"])
    cost = rng.choice(["1,1,1,1,1", "1,1,1,1,1", "1,1,5,1,1", "1,2,2,1,1", "2,1,1,1,2"])
    if kind == "small":
        return _case("", host, "labelled", rng.randint(1, 3), rng.choice([2, 3]), rng.randint(2, 7), rng.randint(2, 7),
                     0, rng.randint(3, 5), 20, 1024, 1, rng.randint(3, 7))
    if kind == "medium":
        sym = rng.choice(["", "", "", "1,2"])
        return _case("", host, "labelled", rng.randint(1, 8), 2, rng.randint(6, 13), rng.randint(6, 13), 0,
                     rng.randint(6, 8), 40, 65536, 8, rng.randint(9, 14), costs=cost, sym_costs=sym)
    if kind == "wide":
        return _case("", host, "labelled", rng.randint(1, 4), rng.choice([3, 4]), rng.randint(12, 30),
                     rng.randint(12, 30), 1, rng.randint(8, 12), 40, 65536, 10, rng.randint(12, 18))
    if kind == "short":
        return _case("", host, "type1", 1, 2, rng.randint(7, 12), rng.randint(7, 12), 0, 4, rng.randint(16, 25), 65536)
    if kind == "mid":
        return _case("", host, "type1", 1, 2, rng.randint(8, 13), rng.randint(8, 13), 0, 5, rng.randint(12, 19), 16384)
    if kind == "long":
        return _case("", host, rng.choice(["type1", "type2"]), 1, 2, rng.randint(8, 14), rng.randint(8, 14), 0,
                     rng.randint(6, 9), rng.randint(11, 16), 16384)
    if kind == "deepwide":
        return _case("", host, "type1", 1, rng.choice([3, 4]), rng.randint(9, 30), rng.randint(9, 30), 0,
                     rng.randint(6, 10), rng.randint(8, 11), 16384)
    if kind == "noisy":
        return _case("", "device", "type2", rng.randint(1, 3), 2, rng.randint(8, 13), rng.randint(8, 13), 0,
                     rng.randint(5, 7), rng.randint(12, 17), 8192, errors=rng.randint(1, 4))
    if kind == "onthefly":
        return _case("", host, "type1", 1, 2, rng.randint(7, 12), rng.randint(7, 12), 0, rng.randint(4, 6),
                     rng.randint(13, 18), _log_int(rng, 4, 64), onthefly=True)
    if kind == "batch":
        return _case("", "batch", "labelled", _log_int(rng, 8, 256), rng.randint(2, 4), rng.randint(4, 20),
                     rng.randint(4, 20), 0, rng.randint(6, 10), 40, 1024, 4, rng.randint(8, 14))
    return _case("", "noalloc", "labelled", rng.randint(1, 4), 2, rng.randint(6, 12), rng.randint(6, 12), 0,
                 rng.randint(5, 7), 40, _log_int(rng, 4, 16), 8, rng.randint(9, 13))


# ---- inputs

class _Target:
    """A random expression of `cost` nodes, and which strings it accepts: its position
    automaton (Glushkov), with sets of positions as bit masks."""

    def __init__(self, rng, cost, n_sym):
        self.symbol, self.follow, self.step = [], [], {}
        self.null, self.first, self.last = self._build(rng, cost, n_sym)

    def _link(self, last, first):
        for p in range(len(self.follow)):
            if last >> p & 1:
                self.follow[p] |= first

    def _build(self, rng, cost, n_sym):
        if cost == 1:
            self.symbol.append(chr(SYMBOLS[rng.randrange(n_sym)]))
            self.follow.append(0)
            m = 1 << len(self.symbol) - 1
            return False, m, m
        op = rng.choice("?*.+" if cost >= 3 else "?*")
        if op in "?*":
            _, first, last = self._build(rng, cost - 1, n_sym)
            if op == "*":
                self._link(last, first)
            return True, first, last
        k = rng.randint(1, cost - 2)
        n1, f1, l1 = self._build(rng, k, n_sym)
        n2, f2, l2 = self._build(rng, cost - 1 - k, n_sym)
        if op == "+":
            return n1 or n2, f1 | f2, l1 | l2
        self._link(l1, f2)
        return n1 and n2, f1 | (f2 if n1 else 0), l2 | (l1 if n2 else 0)

    def accepts(self, text):
        if not text:
            return self.null
        at = None
        for ch in text:
            nxt = self.step.get((at, ch))
            if nxt is None:
                nxt, may = 0, self.first if at is None else 0
                for p, sym in enumerate(self.symbol):
                    if at and at >> p & 1:
                        may |= self.follow[p]
                for p, sym in enumerate(self.symbol):
                    if sym == ch:
                        nxt |= may & 1 << p
                self.step[at, ch] = nxt
            at = nxt
            if not at:
                return False
        return bool(at & self.last)


def _text(rng, recipe, n_sym, lo, hi):
    if recipe == "type1":  # uniform over all strings of length <= hi
        x, n = rng.randrange(sum(n_sym ** k for k in range(hi + 1))), 0
        while x >= n_sym ** n:
            x, n = x - n_sym ** n, n + 1
    else:
        n = rng.randint(lo, hi)
    return bytes(rng.choices(SYMBOLS[:n_sym], k=n)).decode()


def _labelled(rng, c, n_sym, n_pos, n_neg):
    tries = 0
    while True:
        target = _Target(rng, rng.randint(c["cost_lo"], c["cost_hi"]), n_sym)
        pos, neg, seen = [], [], set()
        for k in range(4000):
            # (a target that has labelled next to nothing on one side is given up early)
            if k in (200, 1000) and (len(pos) < min(n_pos, n_pos * k / 2000) or len(neg) < min(n_neg, n_neg * k / 2000)):
                break
            s = _text(rng, "labelled", n_sym, c["len_lo"], c["len_hi"])
            if s in seen:
                continue
            seen.add(s)
            side, n = (pos, n_pos) if target.accepts(s) else (neg, n_neg)
            if len(side) < n:
                side.append(s)
                if len(pos) == n_pos and len(neg) == n_neg:
                    return pos, neg
        tries += 1
        if tries % 50 == 0:  # (few strings of this length and so many examples: ask for fewer)
            n_pos, n_neg = max(1, n_pos - 1), max(1, n_neg - 1)


def _random(rng, c, n_sym, n_pos, n_neg):
    texts = {}
    while len(texts) < n_pos + n_neg:
        texts[_text(rng, c["recipe"], n_sym, c["len_lo"], c["len_hi"])] = None
    texts = list(texts)
    return texts[:n_pos], texts[n_pos:]


def _specs(case, seed):
    rng = random.Random("rei:%d" % seed)
    out = []
    for _ in range(case["problems"]):
        k, p, n = case["n_sym"], case["n_pos"], case["n_neg"]
        if case["form"] == "batch":
            k, p, n = rng.randint(2, k), rng.randint(2, p), rng.randint(2, n)
        pos, neg = (_labelled if case["recipe"] == "labelled" else _random)(rng, case, k, p, n)
        out.append((SYMBOLS[:k], [s.encode() for s in pos], [s.encode() for s in neg]))
    return out


def _ints(text):
    return tuple(int(x) for x in text.split(","))


def prepare(case, seed):
    specs = _specs(case, seed)
    kw = dict(costs=_ints(case["costs"]), max_cost=case["max_cost"], mem_budget=case["budget_mib"] << 20)
    state = {"form": case["form"], "specs": specs, "kw": kw}
    if case["form"] != "noalloc":
        state["ctx"] = rei.Context(device=0)
    if case["form"] != "solve" or case["errors"] or case["onthefly"] or case["sym_costs"]:
        make = rei.Problem.on_device if case["form"] == "device" else rei.Problem
        flags = rei.REI_F_ONTHEFLY if case["onthefly"] else 0
        sym = _ints(case["sym_costs"]) if case["sym_costs"] else None
        state["probs"] = [make(a, p, n, max_errors=case["errors"], flags=flags, sym_costs=sym, **kw)
                          for a, p, n in specs]
    if case["form"] == "noalloc":
        rei.load()
        state["stream"] = torch.cuda.current_stream(0).cuda_stream
        state["out"] = rei._OutBuf()
    return state


# ---- one pass

def _noalloc(state):
    out, res = state["out"], []
    for p in state["probs"]:
        out.reset()
        res.append(out.result(rei.rei_solve_noalloc(p.p, state["stream"], out.res)))
    return res


def run(state):
    ctx, probs = state.get("ctx"), state.get("probs")
    if state["form"] == "noalloc":
        res = _noalloc(state)
    elif state["form"] == "batch":
        res = ctx.solve_batch(probs)
    elif probs is not None:
        res = [ctx.solve_problem(p) for p in probs]
    else:
        res = [ctx.solve(a, p, n, **state["kw"]) for a, p, n in state["specs"]]
    # status, cost, counts and the expression (postfix tokens, zero padded) of every problem
    return [np.array([(r.status, r.cost, r.levels, r.candidates, r.unique) for r in res], dtype=np.int64),
            np.frombuffer(b"".join((r.tree or b"").ljust(128, b"\0") for r in res), dtype=np.uint8)]


def exact(case, seed):
    return None  # (whole numbers and bytes only)


# ---- what a pass cannot do without

def _words(texts):
    subs = {s[i:j] for s in texts for i in range(len(s) + 1) for j in range(i, len(s) + 1)}
    n = len(subs)
    return 1 if n <= 32 else 2 if n <= 64 else 4 * ((n + 127) // 128)


def work(case):
    """Every distinct language found is written once with its back-pointers (4 W + 9
    bytes, W its 32-bit words); every candidate is built and tested for precision and
    uniqueness (about 3 word operations a word).  How many candidates a search of
    random inputs takes to a cost: counted on searches of these recipes, about
    2.2e5 * 2.5^(c - 12) over two symbols and 2.0e5 * 4^(c - 9) over four; a labelled
    specification is mostly found at about two thirds of its target's cost (over more
    than two symbols, half)."""
    total_b = total_f = 0.0
    for a, pos, neg in _specs(case, 0):
        w = _words(pos + neg)
        c = case["max_cost"]
        if case["recipe"] == "labelled":
            c = (0.67 if len(a) == 2 else 0.5) * (case["cost_lo"] + case["cost_hi"]) / 2
        cand = max(10.0, 2.2e5 * 2.5 ** (c - 12) if len(a) == 2 else 2.0e5 * 4.0 ** (c - 9))
        uniq = min(0.3 * cand, 0.1 * 2.0 ** 28 if w == 1 else cand, case["budget_mib"] * 2.0 ** 20 / (4 * w + 28))
        total_b += uniq * (4 * w + 9) + sum(map(len, pos + neg))
        total_f += cand * 3 * w
    return {"bytes": total_b, "flops": total_f}
