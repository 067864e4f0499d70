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


QUEUE = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "batch_items.h"
// chunk, then the instances' points -> tiles, steps, queue length, entries seen; exits 1 when one is seen twice
int main(int argc, char **argv) {
    const int chunk = atoi(argv[1]), count = argc - 2;
    std::vector<int64_t> n(count), tile0(count), nt(count);
    for (int i = 0; i < count; ++i) n[i] = atoll(argv[2 + i]);
    auto size_of = [&](int32_t i) { return n[i]; };
    const batchitems::Queue q = batchitems::make_queue(count, size_of);
    if (!q.fits) return 1;
    std::vector<int> owner;
    for (int k = 0; k < count; ++k) {
        const int i = q.order.empty() ? k : q.order[k];
        tile0[i] = (int64_t)owner.size();
        nt[i] = batchitems::tiles_of(n[i]);
        owner.insert(owner.end(), nt[i], i);
    }
    std::vector<unsigned> first(batchitems::kMaxSteps + 1);
    const int steps = batchitems::step_table(q, chunk / batchitems::kMinChunk, first.data());
    const unsigned total = (unsigned)owner.size(), len = first[steps];
    std::map<std::pair<int64_t, int64_t>, int> seen;  // (tile, chunk)
    for (int cta = 0; cta < 3; ++cta) {  // each claims every third entry
        int step = 0;
        for (unsigned w = cta; w < len; w += 3) {
            step = batchitems::step_at(w, step, first.data());
            const int64_t T = (int64_t)w - first[step];
            if (T < 0 || T >= (int64_t)total) return 1;
            const int i = owner[T];
            const int64_t nchunk = batchitems::steps_of(nt[i], chunk);
            int64_t c = (T - tile0[i]) / chunk + step;
            if (step >= nchunk) return 1;  // nothing to do
            if (c >= nchunk) c -= nchunk;
            if (seen[{T, c}]++) return 1;
        }
    }
    printf("%u %d %u %zu\n", total, steps, len, seen.size());
}
"""


def test_queue_holds_every_tile_and_chunk_once(tmp_path):
    exe = compiled(tmp_path, QUEUE)
    cases = [[0], [1], [64, 65], [4096, 4097, 0, 1, 8192], [300_000] + [64] * 2000, [1, 9000, 5, 20_000, 4097, 4096] * 5,
             [400_000], [0, 0, 70_000, 3, 70_000, 0]]
    for sizes in cases:
        tiles = [-(-n // 64) for n in sizes]
        for chunk in (64, 256):
            r = subprocess.run([exe, str(chunk)] + [str(n) for n in sizes], capture_output=True, text=True)
            assert r.returncode == 0, (sizes[:8], chunk, r.stderr)
            total, steps, length, seen = map(int, r.stdout.split())
            want = sum(t * -(-t // chunk) for t in tiles)
            assert (total, steps) == (sum(tiles), max(-(-t // chunk) for t in tiles))
            assert length == seen == want, (sizes[:8], chunk)
