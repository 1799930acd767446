"""rei_solve_noalloc with budgets whose cache its array cannot hold, though its smaller
arrays would fit: REI_ESCRATCH, and nothing runs.  (The GPU part is collected last, as
test_zz_no_alloc.py.)"""
import os
import shutil
import subprocess

import pytest

import paper_2305_18575_gb300 as rei
from workloads import make_config

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_18575_gb300", "csrc")
MAIN = """
#include "sizes.h"
int main() {
    unsigned char *base = (unsigned char *)4096;
    rei::Carve a{base, 0, 10000};
    if (a.take(100) != base || a.take(100) != base + 256) return 1;
    if (a.take(20000)) return 2;  // (too large)
    if (a.take(1)) return 3;      // nothing after it
    rei::Carve b{base, 0, 1000};
    if (b.take(1000) != base || b.take(0) || b.take(1)) return 4;  // (the next piece would start beyond the end)
    rei::Carve c{base, 0, 1000};
    if (c.take((size_t)-1) || c.take(1)) return 5;
    rei::Carve d{base, 0, 1024};
    if (d.take(768) != base || d.take(256) != base + 768 || d.take(1)) return 6;
    return 0;
}
"""


def test_a_piece_that_does_not_fit_ends_the_carving(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", str(tmp_path / "main")], check=True)
    assert subprocess.run([str(tmp_path / "main")]).returncode == 0


@pytest.mark.gpu
@pytest.mark.parametrize("name,seed", [("medium", 16), ("wide", 0)])
def test_every_budget_beyond_the_array_is_refused(name, seed):
    """Caches of 2 and 16 words from a little more than the array holds to 64 times it:
    the table, the languages or both do not fit, the back-pointers alone would."""
    i = make_config(name, seed)

    def solve(budget):
        buf, prob = rei._OutBuf(), rei.Problem(i.alphabet, i.pos, i.neg, max_cost=8, mem_budget=budget)
        return buf.result(rei.rei_solve_noalloc(prob.p, None, buf.res))

    fits = solve(8 << 20)
    assert fits.status in (rei.REI_OK, rei.REI_NOT_FOUND)
    for budget in (72, 80, 96, 128, 160, 192, 256, 320, 512, 1024, 4096):
        assert solve(budget << 20).status == rei.REI_ESCRATCH, budget
    after = solve(8 << 20)
    assert (after.status, after.candidates, after.unique) == (fits.status, fits.candidates, fits.unique)
