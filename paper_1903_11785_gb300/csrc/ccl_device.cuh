// ccl_device.cuh -- the union-find of the 26-connected labelling, shared by the
// reconstruction's kernels (kernels_ccl.cu) and the allocation-free call
// (noalloc.cu): lock-free, over a dense int32 array of parents indexed by the
// linear voxel index.
#pragma once

#include "fvv_device.cuh"

namespace fvv {

// Every thread gets a budget of find/union steps for the whole launch; valid
// input never comes near it, and a thread that exhausts it stops, sets
// FVV_FLAG_LOOP and returns, so no launch can run unbounded.
constexpr int kStepBudget = 1 << 22;

// Root of x during the union step, shortening the path on the way (each
// visited node is pointed at its grandparent).  Parents only ever point to
// smaller indices of the same tree, so while unions run the plain stores are
// benign: a store that overwrites a concurrent atomicMin link is made good by
// that union, which retries from the old parent it got back.  This holds for
// k_union only: once k_compress writes a voxel's final root, a shortening
// store from another thread's stale walk could replace it with an
// intermediate node, so k_compress uses find_root_readonly instead.
__device__ __forceinline__ int find_root(int* parent, int x, int& budget) {
    int cur = __ldcg(parent + x);
    if (cur == x || cur < 0) return x;
    int prev = x;
    while (budget > 0) {
        --budget;
        const int next = __ldcg(parent + cur);
        if (next == cur || next < 0) return cur;
        __stcg(parent + prev, next);
        prev = cur;
        cur = next;
    }
    return cur;
}

// Root of x once every union is done, without writing anything.  In
// k_compress the only store to parent[v] is v's own thread writing v's root,
// so a parent entry only ever changes from an ancestor to the root: a walk
// that reads either value still ends at the root, and the root that thread
// writes stays (each non-root voxel ends pointing straight at its root, which
// the two-step lookups of k_stats and k_debug_labels rely on).
__device__ __forceinline__ int find_root_readonly(const int* parent, int x, int& budget) {
    int cur = x;
    while (budget > 0) {
        --budget;
        const int next = __ldcg(parent + cur);
        if (next == cur || next < 0) return cur;
        cur = next;
    }
    return cur;
}

__device__ __forceinline__ void unite(int* parent, int a, int b, int& budget) {
    while (budget > 0) {
        a = find_root(parent, a, budget);
        b = find_root(parent, b, budget);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const int old = atomicMin(parent + a, b);
        if (old == a) return;
        a = old;
    }
}

}  // namespace fvv
