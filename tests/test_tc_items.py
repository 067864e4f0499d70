"""The work items of the tensor-core passes, on the CPU: at every size the
library accepts there are as many as row units times column chunks, the CTAs'
rounds reach the last of them, and each is the unit and chunk it stands for.

2^25 points, the most an all-pairs run takes, make 2^31 items in the passes with
128-row units: one more than an int holds.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_02226_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "tc_items.h"
// n, rows of a unit, CTAs -> units, chunk, chunks, items, the last item's unit and chunk, visits of it
int main(int argc, char **argv) {
    for (int k = 1; k + 2 < argc; k += 3) {
        const int64_t n = atoll(argv[k]);
        const int rows = atoi(argv[k + 1]), ctas = atoi(argv[k + 2]);
        const int units = (int)((n + rows - 1) / rows), nct = (int)((n + 255) / 256);
        const int ch = tcitems::chunk_tiles(units, nct, ctas), rels = (nct + ch - 1) / ch;
        const auto items = tcitems::count(units, rels);
        const int64_t last = (int64_t)units * rels - 1;
        const tcitems::Item it = tcitems::item(last, units);
        int64_t visits = 0;
        for (int cta = 0; cta < ctas; ++cta)
            for (auto base = decltype(items)(cta); base < items; base += tcitems::round(ctas)) {
                if (last < base || last > tcitems::dealt(base, 31, ctas)) continue;
                for (int lane = 0; lane < 32; ++lane) visits += tcitems::dealt(base, lane, ctas) == last;
            }
        printf("%d %d %d %lld %d %d %lld\n", units, ch, rels, (long long)items, it.unit, it.rel, (long long)visits);
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("items")
    (d / "items.cpp").write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined",
                        "-fno-sanitize-recover", "-I", CSRC, str(d / "items.cpp"), "-o", str(d / "items")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "items")


def test_every_item_is_reached(program):
    sizes = [1, 128, 129, 4096, 32767, 32768, 200_000, 1 << 24, (1 << 25) - 128, (1 << 25) - 127, 1 << 25]
    asked = [(n, rows, ctas) for n in sizes for rows in (128, 256) for ctas in (148, 152)]
    out = subprocess.run([program] + [str(v) for a in asked for v in a], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    lines = out.stdout.splitlines()
    assert len(lines) == len(asked)
    for (n, rows, ctas), line in zip(asked, lines):
        units, ch, rels, items, unit, rel, visits = map(int, line.split())
        assert units == -(-n // rows) and ch in (1, 2, 4, 8, 16) and rels == -(-(-(-n // 256)) // ch)
        assert items == units * rels, f"n={n} rows={rows}"
        assert (unit, rel, visits) == (units - 1, rels - 1, 1), f"n={n} rows={rows}"
    assert any(units * rels > 2**31 - 1 for units, _, rels, *_ in (map(int, ln.split()) for ln in lines))
