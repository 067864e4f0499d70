"""How a batch is cut into parts and its work numbered, on the CPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_02226_gb300", "csrc")


def compiled(tmp_path, text):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "t.cpp").write_text(text)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=undefined",
                        "-fno-sanitize-recover", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(tmp_path / "t")


PARTS = r"""
#include <cstdio>
#include <cstdlib>
#include "batch_items.h"
// count, points of every instance, of every 1000th -> parts, most rows of a part, instances covered
int main(int, char **argv) {
    const int32_t count = atoi(argv[1]);
    const int64_t n = atoll(argv[2]), big = atoll(argv[3]);
    auto size_of = [&](int32_t i) { return i % 1000 ? n : big; };
    long long parts = 0, most = 0, covered = 0;
    for (int32_t i = 0; i < count;) {
        const int32_t end = batchitems::part_end(i, count, size_of);
        if (end <= i) return 1;
        long long rows = 0;
        for (int32_t k = i; k < end; ++k) rows += batchitems::kTileRows * batchitems::tiles_of(size_of(k));
        most = rows > most ? rows : most;
        covered += end - i;
        ++parts;
        i = end;
    }
    printf("%lld %lld %lld\n", parts, most, covered);
}
"""


def test_rows_of_a_part_leave_room_for_a_stride(tmp_path):
    """A row index plus the threads of the largest grid (8 blocks of 256 on up to
    1,024 SMs) stays within an int, whatever the instances are."""
    exe = compiled(tmp_path, PARTS)
    for count, n, big in [(1, 0, 0), (7, 5, 64), (34_000_000, 1, 1), (3_000_000, 300, 4_000_000), (100, 0, 4_194_240)]:
        r = subprocess.run([exe, str(count), str(n), str(big)], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        parts, most, covered = map(int, r.stdout.split())
        assert covered == count and most + 1024 * 8 * 256 <= 2**31 - 1, (count, n, big)
        rows = sum(-(-v // 64) * 64 * k for v, k in ((big, -(-count // 1000)), (n, count - -(-count // 1000))))
        assert parts >= -(-rows // (64 << 20))
