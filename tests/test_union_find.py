"""The merge's union-find on the CPU: joins, and what a union returns when it
gives up (its cap on lost races): an index of the forest, and the error bit.
Callers keep the result as a member of the set and read its parent."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1506_02226_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#define __device__
#define __forceinline__ inline
#define DB_EBIT_TIMEOUT 2u
#define DB_UNITE_TRIES 1000
static bool lose = false;  // every race
namespace db {
inline int ld_relaxed(const int *p) { return *p; }
inline void st_relaxed(int *p, int v) { *p = v; }
}
inline int atomicCAS(int *p, int cmp, int v) {
    if (lose) return cmp - 1;
    const int old = *p;
    if (old == cmp) *p = v;
    return old;
}
inline void atomicOr(unsigned *p, unsigned v) { *p |= v; }
#include "union_find.cuh"
int main() {
    const int n = 64;
    std::vector<int> parent(n), set(n);
    for (int i = 0; i < n; ++i) parent[i] = set[i] = i;
    unsigned status = 0, seed = 7;
    for (int k = 0; k < 50; ++k) {
        const int a = (seed = seed * 1664525u + 1013904223u) >> 26, b = (seed = seed * 1664525u + 1013904223u) >> 26;
        const int r = db::uf_unite_root(parent.data(), a, b, &status);
        const int sa = set[a], sb = set[b];
        for (int &s : set) s = s == sa || s == sb ? (sa < sb ? sa : sb) : s;
        if (r != set[a]) return 1;
        for (int i = 0; i < n; ++i)
            if (db::uf_find(parent.data(), i) != set[i]) return 2;
    }
    if (status) return 3;
    lose = true;
    for (int a = 0; a < n; ++a)
        for (int b = 0; b < n; ++b) {
            status = 0;
            const int r = db::uf_unite_root(parent.data(), a, b, &status);
            if (r < 0 || r >= n || (r != set[a] && r != set[b])) return 4;
            if (status != (set[a] == set[b] ? 0u : DB_EBIT_TIMEOUT)) return 5;
            status = 0;
            db::uf_unite(parent.data(), a, b, &status);
            if (status != (set[a] == set[b] ? 0u : DB_EBIT_TIMEOUT)) return 6;
        }
    return 0;
}
"""


def test_union_find(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "uf.cpp").write_text(PROGRAM)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(tmp_path / "uf.cpp"), "-o",
                        str(tmp_path / "uf")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(tmp_path / "uf")]).returncode == 0
