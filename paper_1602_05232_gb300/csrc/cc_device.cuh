// Device primitives of the union-find forest: find and hook.
//
// Forest invariant: parent[x] <= x for every x, with equality exactly at the
// roots. Hooks link a root under a smaller node of another tree, and path
// shortening and compression only repoint a node at one of its ancestors, so
// every write keeps the invariant. Consequences used throughout:
//  * every walk strictly decreases the id, so it ends within n steps (no
//    iteration limit is needed, and none can livelock);
//  * once a node stops being a root it never becomes one again, so only roots
//    are ever linked and only non-roots are ever repointed;
//  * a value read late or early is still an ancestor: two endpoints that reach
//    the same node are connected, whatever else is happening.
#pragma once

#include <cstdint>

#include "cc_internal.cuh"

namespace cc {

// Programmatic dependent launch, device side. pdl_trigger: the kernel launched
// after this one on the stream may start placing its CTAs (it still waits in
// pdl_wait before touching results). pdl_wait: returns once the kernel before
// this one has completed and its writes are visible; immediately when this
// kernel was not launched as a dependent.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// Loads of what the kernel before may still have been writing while this one, its
// dependent, was resident (in pdl_wait, or on its way there). Always ordinary
// loads: the read-only path, which __ldg asks for and which the compiler may take
// for any __restrict__ pointer that the kernel does not write through, is only for
// memory that nothing writes as long as the kernel exists. A pass of the R-MAT
// stream (n = 2^24, tuned) took 3507 us with it and takes 3507, the grid 6328 and 6322.
__device__ __forceinline__ int load_after(const int* p) {
    int x;
    asm volatile("ld.global.s32 %0, [%1];\n" : "=r"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ int4 load_after(const int4* p) {
    int4 x;
    asm volatile("ld.global.v4.s32 {%0, %1, %2, %3}, [%4];\n" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "l"(p));
    return x;
}

__device__ __forceinline__ void flag(DevState* ds, unsigned bit) { atomicOr(&ds->status, bit); }

__device__ __forceinline__ bool in_range(int x, int n) { return (unsigned)x < (unsigned)n; }

// Alignment class of a pair array: 2 = 16-byte, 1 = 8-byte, 0 = 4-byte.
__device__ __forceinline__ int pair_vec_dev(const void* p) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    return (a % 16 == 0) ? 2 : (a % 8 == 0) ? 1 : 0;
}

// Repoints x (not a root) at its ancestor `to`, for finds that shorten paths as
// they go. An atomicMin whose result is not used: it is done where the line
// lives, while a plain store to a line that other SMs are reading costs far
// more on this chip. Measured with 2^18 threads that each write one random word
// and read another, per pair: 0.129 ns with a store and 0.0125 with this on 2^16
// words, 0.035 and 0.0124 on 2^20, 0.022 and 0.0137 on 2^22, 0.035 and 0.032
// on 2^26. It also never raises an entry that another walk has lowered further.
__device__ __forceinline__ void lower(int* parent, int x, int to) { atomicMin(parent + x, to); }

// Root of x's tree, given p = parent[x] already read and p != x. Walks with
// path halving: each visited node is repointed at its grandparent, which
// roughly halves the path for later walks (the Section 5.1 idea of making
// later finds cheaper, done on the way up rather than in a second pass).
__device__ __forceinline__ int find_from(int* parent, int x, int p, DevState* ds) {
    while (true) {
        if (p > x) {  // broken invariant: stop rather than loop
            flag(ds, ST_CORRUPT);
            return x;
        }
        int gp = parent[p];
        if (gp == p) return p;
        lower(parent, x, gp);
        x = gp;
        p = parent[x];
        if (p == x) return x;
    }
}

__device__ __forceinline__ int find_halving(int* parent, int x, DevState* ds) {
    int p = parent[x];
    return p == x ? x : find_from(parent, x, p, ds);
}

// Join the trees of roots-or-former-roots ru and rv: the larger root becomes a
// child of the smaller one with a compare-and-swap that succeeds only while it
// is still a root. If another thread linked it first, continue from its new
// root. Each failed round strictly lowers max(ru, rv), so it ends. Returns 1
// if this call made the link, 0 if the two were already joined.
__device__ __forceinline__ int hook(int* parent, int ru, int rv, DevState* ds) {
    while (ru != rv) {
        int hi = ru > rv ? ru : rv;
        int lo = ru > rv ? rv : ru;
        int old = atomicCAS(parent + hi, hi, lo);
        if (old == hi) return 1;
        if (old > hi) {
            flag(ds, ST_CORRUPT);
            return 0;
        }
        int r = find_halving(parent, old, ds);
        if (hi == ru) ru = r; else rv = r;
    }
    return 0;
}

// Largest-component filter (the large-component skip of Afforest: Sutton,
// Ben-Nun and Barak, IPDPS 2018). Bit x of `big` says that x was in the tree
// of one root R when the bitmap was last written (a full compression pass).
// Trees only ever merge, so two vertices whose bits are set stay connected
// whatever is linked afterwards: a query on them answers 1 and an edge
// between them joins nothing, without a read of the forest. The bitmap is
// n bits (8 MiB for 2^26 vertices), so it stays in L2 while the forest
// lines come and go.
__device__ __forceinline__ bool big_member(const unsigned* __restrict__ big, int x) {
    return (__ldg(big + (x >> 5)) >> (x & 31)) & 1u;
}

// The bitmap a kernel may use: `big` when the handle has one and it marks a
// tree (big_root >= 0), else none. Read after the kernel's wait for the one
// before it (the compression pass that wrote the bitmap).
__device__ __forceinline__ const unsigned* big_active(const unsigned* big, const DevState* ds) {
    return (big && ds->big_root >= 0) ? big : nullptr;
}

// Read-only walk to the root from x with p = parent[x] already read.
__device__ __forceinline__ int walk_root(const int* parent, int x, int p) {
    while (p < x) {
        x = p;
        p = parent[x];
    }
    return x;
}

// Load E pairs starting at pair index e0 of a flat u0 v0 u1 v1 ... array.
// vec: 2 = the array is 16-byte aligned, 1 = 8-byte, 0 = 4-byte. Pairs past k
// are left as (0, 0) and must be ignored by the caller. Streaming loads: each
// pair is read once, so it should not displace the forest from L2.
template <int E>
__device__ __forceinline__ void load_pairs(const int* __restrict__ a, int64_t e0, int64_t k,
                                           int vec, int (&u)[E], int (&v)[E]) {
    if (e0 + E <= k) {
        if (E % 2 == 0 && vec == 2) {
#pragma unroll
            for (int i = 0; i < E / 2; i++) {
                int4 q = __ldcs(reinterpret_cast<const int4*>(a + 2 * e0) + i);
                u[2 * i] = q.x; v[2 * i] = q.y; u[2 * i + 1] = q.z; v[2 * i + 1] = q.w;
            }
            return;
        }
        if (vec >= 1) {
#pragma unroll
            for (int i = 0; i < E; i++) {
                int2 q = __ldcs(reinterpret_cast<const int2*>(a + 2 * e0) + i);
                u[i] = q.x; v[i] = q.y;
            }
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < E; i++) {
        if (e0 + i < k) {
            u[i] = __ldcs(a + 2 * (e0 + i));
            v[i] = __ldcs(a + 2 * (e0 + i) + 1);
        } else {
            u[i] = 0; v[i] = 0;
        }
    }
}

}  // namespace cc
