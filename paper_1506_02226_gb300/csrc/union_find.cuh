// union_find.cuh — the union-find forest of the merge passes (included by
// internal.cuh, which has the relaxed accesses).
#pragma once

namespace db {

// ---------------------------------------------------------------------------
// Lock-free union-find over point indices (replaces the paper's per-target
// merge kernel of Section IV-C).  Invariant: parent[x] <= x, and a root is the
// smallest index of its set, because union always links the larger root under
// the smaller one.  Path halving writes only ancestors, so concurrent halving
// and linking keep the invariant.
// ---------------------------------------------------------------------------
#ifndef DB_UNITE_TRIES
#define DB_UNITE_TRIES (1 << 24)
#endif
constexpr int kUniteTries = DB_UNITE_TRIES;

__device__ __forceinline__ int uf_find(int *parent, int x) {
    while (true) {
        int p = ld_relaxed(parent + x);
        if (p == x) return x;
        int gp = ld_relaxed(parent + p);
        if (gp == p) return p;
        st_relaxed(parent + x, gp);
        x = gp;
    }
}

// Root of x, and x straight under it, for the kernels that leave the forest flat
// (each node settled by a thread of its own, no set joined meanwhile): behind
// such a kernel every settled node's parent is its root, and labels are read
// through it.  Nothing else is written on the way: another thread's uf_find that
// read x's old ancestors would halve the path at x after x has its root, and
// leave an ancestor there that is not one (its points' label is then that of no
// set; 500,000 points in the plane were seen with four such).
__device__ __forceinline__ int uf_settle(int *parent, int x) {
    int r = x;
    for (int p = ld_relaxed(parent + r); p != r; p = ld_relaxed(parent + r)) r = p;
    if (r != x) st_relaxed(parent + x, r);
    return r;
}

// Union of the sets of a and b.  Each failed CAS means another thread linked
// the root first, so the loop makes global progress; the cap only guards
// against a corrupted forest and reports it.
__device__ __forceinline__ void uf_unite(int *parent, int a, int b, unsigned *status) {
    for (int it = 0; it < kUniteTries; ++it) {
        a = uf_find(parent, a);
        b = uf_find(parent, b);
        if (a == b) return;
        if (a > b) {
            int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(parent + b, b, a) == b) return;
    }
    atomicOr(status, DB_EBIT_TIMEOUT);
}

// Union that also returns a root of the merged set (a hint for callers that
// cache it: the value is the set's root at some moment, so any point whose
// parent equals it is in the set).  When the cap is reached it is the smaller of
// the two roots as last seen: an index of the forest in any case, since callers
// keep it as a member and follow its parent.
__device__ __forceinline__ int uf_unite_root(int *parent, int a, int b, unsigned *status) {
    for (int it = 0; it < kUniteTries; ++it) {
        a = uf_find(parent, a);
        b = uf_find(parent, b);
        if (a == b) return a;
        if (a > b) {
            int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(parent + b, b, a) == b) return a;
    }
    atomicOr(status, DB_EBIT_TIMEOUT);
    return a;
}

}  // namespace db
