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


SETTLE = r"""
#include <cstdio>
#include <vector>
#define __device__
#define __forceinline__ inline
#define DB_EBIT_TIMEOUT 2u
static void step();  // before every access of the forest
namespace db {
inline int ld_relaxed(const int *p) { step(); return *p; }
inline void st_relaxed(int *p, int v) { step(); *p = v; }
}
inline int atomicCAS(int *p, int, int v) { const int old = *p; *p = v; return old; }
inline void atomicOr(unsigned *p, unsigned v) { *p |= v; }
#include "union_find.cuh"
static std::vector<int> parent, others;  // others: settled, whole, in one thread's way
static int countdown = -1;
static void step() {
    if (countdown < 0 || countdown-- > 0) return;
    for (int v : others) db::uf_settle(parent.data(), v);
    others.clear();
}
int main() {
    const int n = 9;
    for (int fan = 0; fan < 2; ++fan)               // a chain, or a binary tree
        for (int x = 0; x < n; ++x)                 // the thread that is held up,
            for (int at = 0; at < 2 * n; ++at)      // before which of its accesses,
                for (int mask = 0; mask < (1 << n); ++mask) {  // while which others run
                    parent.assign(n, 0);
                    for (int i = 1; i < n; ++i) parent[i] = fan ? (i - 1) / 2 : i - 1;
                    others.clear();
                    for (int v = 0; v < n; ++v)
                        if (v != x && (mask >> v & 1)) others.push_back(v);
                    countdown = at;
                    if (db::uf_settle(parent.data(), x) != 0) return 1;
                    countdown = -1;
                    for (int v : others) db::uf_settle(parent.data(), v);  // (x was done before)
                    for (int v = 0; v < n; ++v)
                        if (v != x && !(mask >> v & 1)) db::uf_settle(parent.data(), v);
                    for (int v = 0; v < n; ++v)
                        if (parent[v] != 0) return 2;
                }
    return 0;
}
"""

def run(tmp_path, text):
    if shutil.which("g++") is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "uf.cpp").write_text(text)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(tmp_path / "uf.cpp"), "-o",
                        str(tmp_path / "uf")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return subprocess.run([str(tmp_path / "uf")]).returncode


def test_union_find(tmp_path):
    assert run(tmp_path, PROGRAM) == 0


def test_settled_nodes_stay_under_their_root(tmp_path):
    """Whatever settles in a thread's way, every node is straight under its root
    once its own thread is done: labels are read through the parents."""
    assert run(tmp_path, SETTLE) == 0
