"""The batch's autotuner tunes every field left open, whatever the others are given as."""
import re

import pytest

import paper_2305_18575_gb300 as rei
from workloads import make_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("given,samples", [(dict(chunk=65536), 2), (dict(chunk=3000), 2), (dict(warps_per_cta=2), 2),
                                           (dict(), 2), (dict(warps_per_cta=2, chunk=65536), 0)])
def test_open_fields_are_tuned(given, samples, monkeypatch, capfd):
    """A sample is one problem a multiprocessor, and two samples stay untimed: a batch of
    four has room for two trials."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    insts = [make_config("small", s) for s in range(40)]
    probs = [rei.Problem(i.alphabet, i.pos, i.neg, max_cost=20) for i in insts]
    monkeypatch.setenv("REI_PHASES", "1")  # (a line on stderr for each launch of a batch)
    with rei.Context(device=0) as ctx:
        plain = [ctx.solve_problem(p) for p in probs]
        capfd.readouterr()
        batch = ctx.solve_batch([probs[k % 40] for k in range(4 * sms)], **given)
    sizes = [int(n) for n in re.findall(r"rei batch of (\d+):", capfd.readouterr().err)]
    assert sizes == [sms] * samples + [(4 - samples) * sms]
    for k, b in enumerate(batch):
        a = plain[k % 40]
        assert (a.status, a.cost, a.tree, a.candidates) == (b.status, b.cost, b.tree, b.candidates), k
