"""Sizes of the uniqueness table (csrc/sizes.h), compiled for the host: at most
2^32 slots, whose numbers the search holds in 32 bits, and room enough below that."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_18575_gb300", "csrc")
CAP = 0x7FFF0000  # the most languages a cache holds
MAIN = """
#include <cstdio>
#include <cstdlib>
#include "sizes.h"
int main(int argc, char **argv) {
    for (int i = 1; i + 4 < argc; i += 5)
        printf("%llu\\n", (unsigned long long)rei::table_slots(strtoull(argv[i], 0, 0), strtoull(argv[i + 1], 0, 0),
               strtoull(argv[i + 2], 0, 0), (uint32_t)strtoull(argv[i + 3], 0, 0), atoi(argv[i + 4]) != 0));
    return 0;
}
"""


@pytest.fixture(scope="module")
def table_slots(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("sizes")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def f(rows, cap, chunk, n, direct=0):
        out = subprocess.run([str(d / "main"), *map(str, (rows, cap, chunk, n, direct))], check=True,
                             capture_output=True, text=True)
        return int(out.stdout)
    return f


@pytest.mark.parametrize("n", [27, 30, 31, 32, 33, 40, 62, 64, 129])
@pytest.mark.parametrize("chunk", [1 << 16, 1 << 25, 1 << 26, 1 << 28])
def test_the_largest_tables_slots_are_numbered_in_32_bits(table_slots, n, chunk):
    for rows in (1 << 30, (1 << 30) + 1, CAP - 1, CAP):
        rows = min(rows, 1 << n)
        slots = table_slots(rows, CAP, chunk, n)
        held = min(rows + (chunk if rows >= CAP else 0), 1 << min(n, 40))
        assert slots & (slots - 1) == 0 and slots <= 1 << 32
        # (half full, or the bound: some 1 - 6 % more)
        assert held <= slots // 2 or (slots == 1 << 32 and held <= 0.57 * slots)


def test_smaller_tables_are_at_most_half_full(table_slots):
    assert table_slots(1, 10, 0, 62) == 1024
    assert table_slots(65536, 1 << 20, 4096, 40) == 1 << 17
    assert table_slots(1 << 20, 1 << 20, 4096, 40) == 1 << 22
    assert table_slots(1 << 20, 1 << 20, 4096, 12) == 1 << 13
    assert table_slots(5, 10, 4096, 26, direct=1) == 1 << 26
    assert table_slots((1 << 30) + 1, CAP, 1 << 25, 40) == 1 << 32


PROBE = """
#include <cstdio>
#include "sizes.h"
int main() {
    using rei::probe_first;
    using rei::probe_next;
    const uint64_t top = 0xFFFFFFFFull;
    // the largest table: its last slot is passed over, from either side
    if (probe_first(0x12345678FFFFFFFFull, top) != top - 1 || probe_first(0x12345678FFFFFFFEull, top) != top - 1) return 1;
    if (probe_next(0xFFFFFFFEu, 0xFFFFFFFFu) != 0 || probe_next(0xFFFFFFFDu, 0xFFFFFFFFu) != 0xFFFFFFFEu) return 2;
    if (probe_next(7u, 0xFFFFFFFFu) != 8) return 3;
    if (probe_next(top - 1, top) != 0 || probe_next(top - 2, top) != top - 1 || probe_next(uint64_t(7), top) != 8) return 7;
    // any other: every slot in turn
    for (uint64_t bits = 10; bits < 32; bits++) {
        const uint64_t mask = (1ull << bits) - 1;
        const uint32_t m = (uint32_t)mask;
        if (probe_first(~0ull, mask) != mask || probe_first(~0ull - 1, mask) != mask - 1) return 4;
        if (probe_next(m - 1, m) != m || probe_next(m, m) != 0) return 5;
        if (probe_next(mask - 1, mask) != mask || probe_next(mask, mask) != 0) return 6;
    }
    return 0;
}
"""


def test_probing_passes_over_the_number_that_means_not_marked(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    (tmp_path / "probe.cpp").write_text(PROBE)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "probe.cpp"), "-o", str(tmp_path / "probe")], check=True)
    assert subprocess.run([str(tmp_path / "probe")]).returncode == 0
    # and nothing in the searches probes by itself
    for name in ("search.cuh", "relaunch.cu", "slots.cu", "solve.cu"):
        with open(os.path.join(CSRC, name)) as fh:
            text = fh.read()
        assert "+ 1) & J.table_mask" not in text and "h & J.table_mask" not in text, name
