// Kernels of the plain (one launch per bulk operation) path and their launchers.
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.cuh"

namespace cc {

int pair_vec(const void* p) {
    uintptr_t a = reinterpret_cast<uintptr_t>(p);
    return (a % 16 == 0) ? 2 : (a % 8 == 0) ? 1 : 0;
}

static inline unsigned blocks_for(int64_t work, int64_t per_block) {
    return (unsigned)((work + per_block - 1) / per_block);
}

// Edges (pairs) per thread of a launch with one chunk per thread: as many as
// asked for, but not so many that an SM is left without a CTA. Default options
// (2 per thread, 256 threads), 2 and 1 per thread: minibatches of up to 2^18,
// 30,000 on average, on 10^6 vertices with 50,001 pairs asked after each 894 and
// 854 us for 104 steps; but 434 and 473 for 32 of 2^17, which fill the chip.
static int spread(int ept, int64_t k, int block) {
    thread_local int sms[16] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    int own = 0;
    int& n = dev >= 0 && dev < 16 ? sms[dev] : own;
    if (!n) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    while (ept > 1 && k < (int64_t)ept * block * n) ept /= 2;
    return ept;
}

// ------------------------------------------------------------------ reset

// parent[v] = v: n singletons, the empty graph G_0, with no links made and no
// tree marked (DevState's unions and big_root, which the first CTA sets here:
// as two memsets in front they were two more operations on the stream). Kernels
// that are launched as dependents may read big_root before their own wait; they
// start once all CTAs here have exited, the first one after its write is visible.
// Four vectors per thread: with one, CTAs were launched more slowly than they
// wrote (2^26 vertices in CTAs of 128 threads: 72 -> 39 us, 6.9 TB/s).
__global__ void k_reset(int* __restrict__ parent, int64_t n, DevState* __restrict__ ds) {
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ds->unions = 0ull;
        ds->big_root = -1;
        __threadfence();
    }
    const int64_t q0 = (int64_t)blockIdx.x * blockDim.x * 4 + threadIdx.x;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int64_t v0 = (q0 + (int64_t)i * blockDim.x) * 4;
        if (v0 + 4 <= n) {
            int x = (int)v0;
            reinterpret_cast<int4*>(parent)[v0 / 4] = make_int4(x, x + 1, x + 2, x + 3);
        } else {
            for (int64_t v = v0; v < n; v++) parent[v] = (int)v;
        }
    }
}

cudaError_t launch_reset(int* parent, int64_t n, DevState* ds, int block, bool pdl, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    launch_windowed(k_reset, blocks_for(n, 16LL * block), block, s, nullptr, pdl, parent, n, ds);
    return cudaGetLastError();
}

// ------------------------------------------------------------ Bulk-Update

// Bit i set when this thread's edge i at e0 exists and has both endpoints in
// range, and (with a largest-component bitmap) they are not both marked;
// range errors are flagged here, once per chunk.
template <int E>
__device__ __forceinline__ unsigned edge_mask(int n, const int (&u)[E], const int (&v)[E], int64_t e0,
                                              int64_t k, DevState* __restrict__ ds, const unsigned* bits) {
    unsigned m = 0;
    bool bad = false;
#pragma unroll
    for (int i = 0; i < E; i++) {
        if (e0 + i >= k) continue;
        if (in_range(u[i], n) && in_range(v[i], n)) m |= 1u << i;
        else bad = true;
    }
    if (bad) flag(ds, ST_RANGE);
    if (bits) {  // both endpoints in the marked tree: already joined
#pragma unroll
        for (int i = 0; i < E; i++)
            if (((m >> i) & 1u) && big_member(bits, u[i]) && big_member(bits, v[i])) m &= ~(1u << i);
    }
    return m;
}

// The first parent reads of the edges in m, all issued together (an edge not
// in m reads nothing and keeps its endpoints as their own parents).
template <int E>
__device__ __forceinline__ void gather_parents(const int* parent, unsigned m, const int (&u)[E],
                                               const int (&v)[E], int (&pu)[E], int (&pv)[E]) {
#pragma unroll
    for (int i = 0; i < E; i++) {
        const bool on = (m >> i) & 1u;
        pu[i] = on ? load_after(parent + u[i]) : u[i];
        pv[i] = on ? load_after(parent + v[i]) : v[i];
    }
}

// The rest of the fused pass for edges whose first parents pu, pv were read
// earlier, possibly before other links of this minibatch: a parent read then
// is still an ancestor now (links only put roots under other trees' nodes, and
// splitting only repoints a node at an ancestor), so going on from it reaches
// the current root, and equal values still prove the endpoints joined.
//
// Each edge is two nodes, one of either side, and the larger one is moved up
// until the sides meet or it is a root, which is then linked under the other
// side's node as it stands: ids fall along every path, so that node is not in
// the larger root's tree, and it need not be a root itself. (This is Rem's
// linking, as in Patwary, Blair and Manne, SEA 2010, without its splicing; the
// nodes passed are repointed at their grandparents instead.) A side is read no
// further than the other side makes necessary, where walking both to verified
// roots first reads at least one more node on each. Against that (with compare-and-
// swap or atomicMin on both verified roots), per pass: R-MAT n = 2^22 with a
// compression after each of 32 minibatches 1492 -> 1312 us, 104 ragged
// minibatches 1033 -> 922, R-MAT n = 2^24 without compression 3776 -> 3518, the
// grid 6640 -> 6464; the first minibatch on an empty forest 145 -> 84 us (R-MAT
// n = 2^22), 55 -> 35 (n = 2^20).
//
// The E edges advance in lockstep: all their loads are issued, then all their
// link attempts. An attempt on a node that is no root any more returns its
// parent, which is what a read would have returned: with compare-and-swap the
// node is untouched. With atomicMin (minhook) a parent above lo is lowered to
// lo, which moves the node's subtree into lo's tree; the edge goes on joining
// the displaced parent with lo, so every earlier connection is kept (a
// splitting store that races with the move and undoes it is harmless for the
// same reason). Only a write at a root counts as a link. Each round strictly
// lowers the larger node of every edge, so the loop ends.
//
// A first parent that was a root is tried without another read. With HOOK_AGAIN it
// is read again first: where a minibatch has more edges than the graph vertices, most
// of its edges are joined by others while they wait, and a try for each queues on the
// few words that are left (2^18 edges on 4096 vertices with atomicMin, four
// minibatches: 60 us with both roots verified first, 101 without a second read, 48
// with it; 2^20 on 64 with compare-and-swap 354, 767 and 214).
// One link attempt per distinct hi among the lanes of a whole warp that try
// one: the first of them tries to put hi under its own lo. Returns hi if this
// lane linked it, else hi's parent as this leaves it (p for a lane without a try).
__device__ __forceinline__ int link_grouped(int* parent, bool tries, int hi, int lo, bool minhook, int p) {
    const unsigned full = 0xffffffffu;
    if (!__any_sync(full, tries)) return p;
    const int lane = (int)(threadIdx.x & 31u);
    const int leader = __ffs(__match_any_sync(full, tries ? hi : -1 - lane)) - 1;
    int old = hi;
    if (tries && lane == leader) old = minhook ? atomicMin(parent + hi, lo) : atomicCAS(parent + hi, hi, lo);
    old = __shfl_sync(full, old, leader);
    const int to = __shfl_sync(full, lo, leader);
    if (!tries) return p;
    return lane != leader && (old == hi || (minhook && to < old && old < hi)) ? to : old;
}

template <int E, bool WARP>
__device__ __forceinline__ int join_edges(int* parent, unsigned m, const int (&u)[E], const int (&v)[E],
                                          const int (&pu)[E], const int (&pv)[E], DevState* ds, int hook) {
    const bool minhook = hook & HOOK_MIN, climb = hook & HOOK_CLIMB;
    const int root = hook & HOOK_AGAIN ? -2 : -1;
    int hi[E], lo[E];    // the two nodes of each edge; equal once it is done
    int bhi[E], blo[E];  // the node below each on its path, or -1: it was a root when it was read (-2: and is read again)
    bool any = false;
#pragma unroll
    for (int i = 0; i < E; i++) {
        const bool swap = pu[i] < pv[i];
        const int x = swap ? v[i] : u[i], y = swap ? u[i] : v[i];
        lo[i] = swap ? pu[i] : pv[i];
        hi[i] = !((m >> i) & 1u) ? lo[i] : swap ? pv[i] : pu[i];
        bhi[i] = hi[i] == x ? root : x;
        blo[i] = lo[i] == y ? root : y;
        any |= hi[i] != lo[i];
    }
    int made = 0;
    while (WARP ? __any_sync(0xffffffffu, any) : any) {
        int p[E];
#pragma unroll
        for (int i = 0; i < E; i++) {
            p[i] = hi[i];
            if (hi[i] != lo[i] && bhi[i] != -1) p[i] = parent[hi[i]];
        }
        if (climb) {
            int q[E];
#pragma unroll
            for (int i = 0; i < E; i++) {
                q[i] = lo[i];
                if (hi[i] != lo[i] && blo[i] != -1 && p[i] == hi[i]) q[i] = parent[lo[i]];
            }
#pragma unroll
            for (int i = 0; i < E; i++) {
                if (q[i] >= lo[i]) continue;
                if (blo[i] >= 0) lower(parent, blo[i], q[i]);
                blo[i] = lo[i];
                lo[i] = q[i];
                bhi[i] = -1;  // hi has been read and is a root
                p[i] = -1;    // no attempt in this round
            }
        }
#pragma unroll
        for (int i = 0; i < E; i++) {
            const bool tries = hi[i] != lo[i] && p[i] == hi[i];
            if constexpr (WARP) p[i] = link_grouped(parent, tries, hi[i], lo[i], minhook, p[i]);
            else if (tries) p[i] = minhook ? atomicMin(parent + hi[i], lo[i]) : atomicCAS(parent + hi[i], hi[i], lo[i]);
        }
        any = false;
#pragma unroll
        for (int i = 0; i < E; i++) {
            if (hi[i] == lo[i]) continue;
            if (climb && p[i] < 0) {
                any = true;
                continue;
            }
            if (p[i] >= hi[i]) {  // linked, or a broken invariant: stop rather than loop
                if (p[i] == hi[i]) made++;
                else flag(ds, ST_CORRUPT);
                hi[i] = lo[i];
                continue;
            }
            if (bhi[i] >= 0) lower(parent, bhi[i], p[i]);  // splitting: skip a level
            const int below = hi[i];
            const bool swap = p[i] < lo[i];
            hi[i] = swap ? lo[i] : p[i];
            bhi[i] = swap ? blo[i] : below;
            lo[i] = swap ? p[i] : lo[i];
            blo[i] = swap ? below : blo[i];
            any |= hi[i] != lo[i];
        }
    }
    return made;
}

// One fused pass of Algorithm 2 over E edges: the first parent reads of both
// endpoints of all E edges are issued together; equal parents mean the edge
// joins a tree to itself and is dropped at once (the common case once trees
// are flat, and the self-loop filter of Algorithm 2). The others are joined.
// Returns the number of links made.
template <int E, bool WARP>
__device__ __forceinline__ int update_edges(int* __restrict__ parent, int n, const int (&u)[E], const int (&v)[E],
                                            int64_t e0, int64_t k, DevState* __restrict__ ds, int hook,
                                            const unsigned* bits) {
    const unsigned m = edge_mask<E>(n, u, v, e0, k, ds, bits);
    int pu[E], pv[E];
    gather_parents<E>(parent, m, u, v, pu, pv);
    return join_edges<E, WARP>(parent, m, u, v, pu, pv, ds, hook);
}

// early: the first edges are read before the wait for the previous kernel
// (programmatic dependent launch; see launch_windowed), else after it.
// WARP: the link attempts of a warp are grouped by target (link_grouped), so
// every lane of a warp that has any edge left goes through each round of the
// loop, with no edges of its own if it has none.
template <int E, bool PERSIST, bool WARP>
__global__ void __launch_bounds__(1024)
k_update(int* __restrict__ parent, int n, const int* __restrict__ edges, int64_t k, int vec,
         DevState* __restrict__ ds, int early, int hook, BigArgs fb) {
    pdl_trigger();
    if (!early) pdl_wait();
    if (fb.alt && big_active(fb.big, ds)) {  // the filter is on: the edges were not ordered
        edges = fb.alt;
        vec = pair_vec_dev(fb.alt);
    }
    int made = 0;
    int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * E;
    if (!PERSIST) {
        // with warphook, every lane goes in if any lane of its warp has edges
        bool warp_busy = false;
        if constexpr (WARP) warp_busy = __any_sync(0xffffffffu, e0 < k);
        if (e0 < k || warp_busy) {
            int u[E], v[E];
            load_pairs<E>(edges, e0, k, vec, u, v);
            if (early) pdl_wait();
            made = update_edges<E, WARP>(parent, n, u, v, e0, k, ds, hook, big_active(fb.big, ds));
        }
    } else {
        // persistent grid: loop over chunks, loading the next chunk's edges
        // before walking the current one so their latency overlaps
        const int64_t stride = (int64_t)gridDim.x * blockDim.x * E;
        int u[E], v[E];
        if (e0 < k) load_pairs<E>(edges, e0, k, vec, u, v);
        if (early) pdl_wait();
        const unsigned* bits = big_active(fb.big, ds);
        while (WARP ? __any_sync(0xffffffffu, e0 < k) : e0 < k) {
            const int64_t nx = e0 + stride;
            int nu[E] = {}, nv[E] = {};
            if (nx < k) load_pairs<E>(edges, nx, k, vec, nu, nv);
            made += update_edges<E, WARP>(parent, n, u, v, e0, k, ds, hook, bits);
#pragma unroll
            for (int i = 0; i < E; i++) {
                u[i] = nu[i];
                v[i] = nv[i];
            }
            e0 = nx;
        }
    }
    made = __reduce_add_sync(0xffffffffu, made);
    if ((threadIdx.x & 31) == 0 && made) atomicAdd(&ds->unions, (unsigned long long)made);
}

// --- VARIANT 3: the persistent grid with a two-stage prefetch -------------

// Persistent grid over chunks of E edges per thread. While the walks and
// hooks of chunk c run, the first parent reads of chunk c+1 and the edge
// loads of chunk c+2 are already in flight, so a warp waiting on its deepest
// walk still has the next chunk's gathers outstanding. early: as for k_update.
template <int E, bool WARP>
__global__ void __launch_bounds__(1024)
k_update_deep(int* __restrict__ parent, int n, const int* __restrict__ edges, int64_t k, int vec,
              DevState* __restrict__ ds, int early, int hook, BigArgs fb) {
    pdl_trigger();
    if (!early) pdl_wait();
    if (fb.alt && big_active(fb.big, ds)) {  // as in k_update
        edges = fb.alt;
        vec = pair_vec_dev(fb.alt);
    }
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * E;
    int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * E;
    int made = 0;
    int u0[E] = {}, v0[E] = {}, u1[E] = {}, v1[E] = {};
    if (e0 < k) load_pairs<E>(edges, e0, k, vec, u0, v0);
    if (e0 + stride < k) load_pairs<E>(edges, e0 + stride, k, vec, u1, v1);
    if (early) pdl_wait();
    const unsigned* bits = big_active(fb.big, ds);
    unsigned m0 = e0 < k ? edge_mask<E>(n, u0, v0, e0, k, ds, bits) : 0u;
    int pu0[E], pv0[E];
    gather_parents<E>(parent, m0, u0, v0, pu0, pv0);
    while (WARP ? __any_sync(0xffffffffu, e0 < k) : e0 < k) {
        const int64_t e1 = e0 + stride, e2 = e1 + stride;
        const unsigned m1 = e1 < k ? edge_mask<E>(n, u1, v1, e1, k, ds, bits) : 0u;
        int pu1[E], pv1[E];
        gather_parents<E>(parent, m1, u1, v1, pu1, pv1);
        int u2[E] = {}, v2[E] = {};
        if (e2 < k) load_pairs<E>(edges, e2, k, vec, u2, v2);
        made += join_edges<E, WARP>(parent, m0, u0, v0, pu0, pv0, ds, hook);
#pragma unroll
        for (int i = 0; i < E; i++) {
            u0[i] = u1[i]; v0[i] = v1[i]; pu0[i] = pu1[i]; pv0[i] = pv1[i];
            u1[i] = u2[i]; v1[i] = v2[i];
        }
        m0 = m1;
        e0 = e1;
    }
    made = __reduce_add_sync(0xffffffffu, made);
    if ((threadIdx.x & 31) == 0 && made) atomicAdd(&ds->unions, (unsigned long long)made);
}

template <int E>
static void update_deep_inst(const int* edges, int64_t k, int vec, int* parent, int n, DevState* ds,
                             int block, const cudaAccessPolicyWindow* window, int pdl, int hook,
                             int warphook, BigArgs fb, cudaStream_t s) {
    int64_t g = (k + (int64_t)E * block - 1) / ((int64_t)E * block);
    if (warphook) {
        const int64_t cap = resident_grid<k_update_deep<E, true>>(block);
        if (g > cap) g = cap;
        launch_windowed(k_update_deep<E, true>, (unsigned)g, block, s, window, pdl != 0, parent, n, edges, k,
                        vec, ds, (int)(pdl == 2), hook, fb);
        return;
    }
    const int64_t cap = resident_grid<k_update_deep<E, false>>(block);
    if (g > cap) g = cap;
    launch_windowed(k_update_deep<E, false>, (unsigned)g, block, s, window, pdl != 0, parent, n, edges, k, vec,
                    ds, (int)(pdl == 2), hook, fb);
}

// --- VARIANT 5: per-CTA list of open edges ---------------------------------
//
// A persistent grid over tiles of blockDim * E edges. Every thread reads its
// E edges' first parents (independent loads, as in the filter pass of
// variant 4); the open edges (parents differ) go to a list in shared memory,
// and then all threads of the CTA walk and hook that list together, two
// listed edges per thread at a time, while the edge loads and first parent
// reads of the CTA's next tile are already in flight. So the walks of the few
// open edges are spread over every thread of the CTA instead of stalling the
// warp that happened to load them. Two barriers per tile; the list's counter
// is double-buffered so that a count is cleared only after every thread has
// read it.
template <int E>
__global__ void __launch_bounds__(1024, 1)  // without the minimum, E = 1 and 2 were held to 32 registers and spilled
k_update_tiles(int* __restrict__ parent, int n, const int* __restrict__ edges, int64_t k, int vec,
               DevState* __restrict__ ds, int early, int hook, BigArgs fb) {
    extern __shared__ int4 open_list[];  // blockDim.x * E entries: (u, v, parent[u], parent[v])
    __shared__ unsigned n_open[2];
    pdl_trigger();
    if (!early) pdl_wait();
    if (fb.alt && big_active(fb.big, ds)) {  // as in k_update
        edges = fb.alt;
        vec = pair_vec_dev(fb.alt);
    }
    const int64_t T = (int64_t)blockDim.x * E;
    const int64_t tiles = (k + T - 1) / T;
    if (threadIdx.x == 0) n_open[0] = n_open[1] = 0u;
    int made = 0;
    int64_t t = blockIdx.x;
    int u[E] = {}, v[E] = {}, pu[E], pv[E];
    unsigned m = 0;
    int64_t e0 = t * T + (int64_t)threadIdx.x * E;
    if (t < tiles && e0 < k) load_pairs<E>(edges, e0, k, vec, u, v);
    if (early) pdl_wait();
    const unsigned* bits = big_active(fb.big, ds);
    if (t < tiles && e0 < k) m = edge_mask<E>(n, u, v, e0, k, ds, bits);
    gather_parents<E>(parent, m, u, v, pu, pv);
    __syncthreads();  // counters cleared
    const unsigned lane = threadIdx.x & 31u;
    for (int sel = 0; t < tiles; t += gridDim.x, sel ^= 1) {
        // append this thread's open edges (one atomic per warp)
        unsigned open = 0;
#pragma unroll
        for (int i = 0; i < E; i++)
            if (((m >> i) & 1u) && pu[i] != pv[i]) open |= 1u << i;
        const int mine = __popc(open);
        int incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= (unsigned)d) incl += y;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        unsigned base = 0;
        if (lane == 31 && total) base = atomicAdd(&n_open[sel], (unsigned)total);
        base = __shfl_sync(0xffffffffu, base, 31) + (unsigned)(incl - mine);
#pragma unroll
        for (int i = 0; i < E; i++)
            if ((open >> i) & 1u) open_list[base++] = make_int4(u[i], v[i], pu[i], pv[i]);
        __syncthreads();  // A: the list of this tile is complete
        const unsigned cnt = n_open[sel];
        if (threadIdx.x == 0) n_open[sel ^ 1] = 0u;  // last read before the previous B
        // the next tile's edges and first parents, in flight during the walks
        const int64_t t1 = t + gridDim.x;
        const int64_t e1 = t1 * T + (int64_t)threadIdx.x * E;
        int nu[E] = {}, nv[E] = {};
        unsigned m1 = 0;
        if (t1 < tiles && e1 < k) {
            load_pairs<E>(edges, e1, k, vec, nu, nv);
            m1 = edge_mask<E>(n, nu, nv, e1, k, ds, bits);
        }
        int npu[E], npv[E];
        gather_parents<E>(parent, m1, nu, nv, npu, npv);
        // walk and hook the list, two entries per thread at a time
        for (unsigned j = 2u * threadIdx.x; j < cnt; j += 2u * blockDim.x) {
            const int4 a = open_list[j];
            const int4 b = j + 1 < cnt ? open_list[j + 1] : a;
            const unsigned on = j + 1 < cnt ? 3u : 1u;
            const int lu[2] = {a.x, b.x}, lv[2] = {a.y, b.y}, lpu[2] = {a.z, b.z}, lpv[2] = {a.w, b.w};
            made += join_edges<2, false>(parent, on, lu, lv, lpu, lpv, ds, hook);
        }
        __syncthreads();  // B: the list has been walked; it may be refilled
#pragma unroll
        for (int i = 0; i < E; i++) {
            u[i] = nu[i]; v[i] = nv[i]; pu[i] = npu[i]; pv[i] = npv[i];
        }
        m = m1;
    }
    made = __reduce_add_sync(0xffffffffu, made);
    if ((threadIdx.x & 31) == 0 && made) atomicAdd(&ds->unions, (unsigned long long)made);
}

template <int E>
static void update_tiles_inst(const int* edges, int64_t k, int vec, int* parent, int n, DevState* ds, int block,
                              const cudaAccessPolicyWindow* window, int pdl, int hook, BigArgs fb,
                              cudaStream_t s) {
    const size_t smem = sizeof(int4) * (size_t)block * E;
    if (smem > 48 * 1024)  // the largest list (1024 threads x 4 edges) needs 64 KiB
        cudaFuncSetAttribute(k_update_tiles<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int64_t g = (k + (int64_t)E * block - 1) / ((int64_t)E * block);
    const int64_t cap = resident_grid<k_update_tiles<E>>(block, smem);
    if (g > cap) g = cap;
    launch_windowed_smem(k_update_tiles<E>, (unsigned)g, block, smem, s, window, pdl != 0, parent, n, edges, k, vec, ds,
                         (int)(pdl == 2), hook, fb);
}

// HOOK_AGAIN from this many edges per vertex. Four minibatches of 2^16 to 2^20
// uniform or skewed edges on 16 to 2^18 vertices take 1.00 of the time with it at
// half an edge per vertex, 0.92 at one, 0.86 at two, 0.82 at four and less from there;
// but sixteen of 2^16 uniform edges on 2^16 vertices 1.01 to 1.02.
static bool dense(int64_t k, int n) { return k >= 2 * (int64_t)n; }

// --- VARIANT 4: filter pass + live-edge pass ------------------------------
//
// Once the forest is shallow, almost every edge of a minibatch already has
// parent[u] == parent[v] (its endpoints were joined before), and only a few
// percent need walks and a hook. Pass 1 streams all edges and does only those
// first parent reads -- every warp's loads are independent, so the pass runs
// at the rate of the gathers -- and appends each edge that is still open as
// (u, v, parent[u], parent[v]) to a compact list. Pass 2 walks and hooks only
// the listed edges, from the parents pass 1 read (still ancestors; see
// join_edges). The two list counters alternate between minibatches: pass 1
// of minibatch i appends through count[sel] and zeroes count[sel ^ 1] for
// minibatch i + 1, after the wait that orders it behind everything before it.

template <int E>
__global__ void __launch_bounds__(1024)
k_update_filter(const int* __restrict__ parent, int n, const int* __restrict__ edges, int64_t k, int vec,
                int4* __restrict__ live, unsigned* __restrict__ count, int sel, DevState* __restrict__ ds,
                int early, BigArgs fb) {
    pdl_trigger();
    if (!early) pdl_wait();
    if (fb.alt && big_active(fb.big, ds)) {  // as in k_update
        edges = fb.alt;
        vec = pair_vec_dev(fb.alt);
    }
    const int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * E;
    int u[E] = {}, v[E] = {};
    if (e0 < k) load_pairs<E>(edges, e0, k, vec, u, v);
    if (early) pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) count[sel ^ 1] = 0u;
    const unsigned m = e0 < k ? edge_mask<E>(n, u, v, e0, k, ds, big_active(fb.big, ds)) : 0u;
    int pu[E], pv[E];
    gather_parents<E>(parent, m, u, v, pu, pv);
    unsigned open = 0;
#pragma unroll
    for (int i = 0; i < E; i++)
        if (((m >> i) & 1u) && pu[i] != pv[i]) open |= 1u << i;
    // one atomic per warp: an exclusive scan of the lanes' open counts
    const unsigned lane = threadIdx.x & 31u;
    const int mine = __popc(open);
    int incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= (unsigned)d) incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) return;
    unsigned base = 0;
    if (lane == 31) base = atomicAdd(count + sel, (unsigned)total);
    base = __shfl_sync(0xffffffffu, base, 31) + (unsigned)(incl - mine);
#pragma unroll
    for (int i = 0; i < E; i++)
        if ((open >> i) & 1u) live[base++] = make_int4(u[i], v[i], pu[i], pv[i]);
}

// Pass 2: two listed edges per thread per step, in lockstep.
template <bool WARP>
__global__ void __launch_bounds__(1024)
k_update_live(int* __restrict__ parent, const int4* __restrict__ live, const unsigned* __restrict__ count,
              int sel, DevState* __restrict__ ds, int hook) {
    pdl_trigger();
    pdl_wait();
    const int64_t m = (unsigned)load_after(reinterpret_cast<const int*>(count) + sel);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * 2;
    int made = 0;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 2;
         WARP ? __any_sync(0xffffffffu, i < m) : i < m; i += stride) {
        const int4 zero = make_int4(0, 0, 0, 0);
        const int4 a = i < m ? load_after(live + i) : zero;
        const int4 b = i + 1 < m ? load_after(live + i + 1) : a;
        const unsigned on = i + 1 < m ? 3u : i < m ? 1u : 0u;
        const int u[2] = {a.x, b.x}, v[2] = {a.y, b.y}, pu[2] = {a.z, b.z}, pv[2] = {a.w, b.w};
        made += join_edges<2, WARP>(parent, on, u, v, pu, pv, ds, hook);
    }
    made = __reduce_add_sync(0xffffffffu, made);
    if ((threadIdx.x & 31) == 0 && made) atomicAdd(&ds->unions, (unsigned long long)made);
}

template <int E>
static void update_filter_inst(const int* edges, int64_t k, int vec, const int* parent, int n, int4* live,
                               unsigned* count, int sel, DevState* ds, int block,
                               const cudaAccessPolicyWindow* window, int pdl, BigArgs fb,
                               cudaStream_t s) {
    const int64_t g = (k + (int64_t)E * block - 1) / ((int64_t)E * block);
    launch_windowed(k_update_filter<E>, (unsigned)g, block, s, window, pdl != 0, parent, n, edges, k, vec,
                    live, count, sel, ds, (int)(pdl == 2), fb);
}

cudaError_t launch_update_split(int* parent, int n, const int* edges, int64_t k, DevState* ds, Launch cfg,
                                int4* live, unsigned* count, int sel, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    if (dense(k, n)) cfg.hook |= HOOK_AGAIN;
    const int vec = pair_vec(edges);
    switch (cfg.ept) {
        case 1: update_filter_inst<1>(edges, k, vec, parent, n, live, count, sel, ds, cfg.block, cfg.window, cfg.pdl, BigArgs{cfg.big, cfg.alt}, s); break;
        case 2: update_filter_inst<2>(edges, k, vec, parent, n, live, count, sel, ds, cfg.block, cfg.window, cfg.pdl, BigArgs{cfg.big, cfg.alt}, s); break;
        case 4: update_filter_inst<4>(edges, k, vec, parent, n, live, count, sel, ds, cfg.block, cfg.window, cfg.pdl, BigArgs{cfg.big, cfg.alt}, s); break;
        default: return cudaErrorInvalidValue;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // pass 2 on a grid of resident CTAs, capped by the most it could have to do
    int64_t g = (k + 2LL * cfg.block - 1) / (2LL * cfg.block);
    if (cfg.warphook) {
        const int64_t cap = resident_grid<k_update_live<true>>(cfg.block);
        if (g > cap) g = cap;
        launch_windowed(k_update_live<true>, (unsigned)g, cfg.block, s, cfg.window, cfg.pdl != 0, parent,
                        (const int4*)live, (const unsigned*)count, sel, ds, cfg.hook);
    } else {
        const int64_t cap = resident_grid<k_update_live<false>>(cfg.block);
        if (g > cap) g = cap;
        launch_windowed(k_update_live<false>, (unsigned)g, cfg.block, s, cfg.window, cfg.pdl != 0, parent,
                        (const int4*)live, (const unsigned*)count, sel, ds, cfg.hook);
    }
    return cudaGetLastError();
}


template <int E, bool PERSIST, bool WARP>
static void update_inst2(const int* edges, int64_t k, int vec, int* parent, int n, DevState* ds,
                         int block, const cudaAccessPolicyWindow* window, int pdl, int hook,
                         BigArgs fb, cudaStream_t s) {
    int64_t g = (k + (int64_t)E * block - 1) / ((int64_t)E * block);
    if (PERSIST) {
        const int64_t cap = resident_grid<k_update<E, PERSIST, WARP>>(block);
        if (g > cap) g = cap;
    }
    launch_windowed(k_update<E, PERSIST, WARP>, (unsigned)g, block, s, window, pdl != 0, parent, n, edges, k,
                    vec, ds, (int)(pdl == 2), hook, fb);
}

template <int E, bool PERSIST>
static void update_inst(const int* edges, int64_t k, int vec, int* parent, int n, DevState* ds,
                        int block, const cudaAccessPolicyWindow* window, int pdl, int hook,
                        int warphook, BigArgs fb, cudaStream_t s) {
    if (warphook)
        update_inst2<E, PERSIST, true>(edges, k, vec, parent, n, ds, block, window, pdl, hook, fb, s);
    else
        update_inst2<E, PERSIST, false>(edges, k, vec, parent, n, ds, block, window, pdl, hook, fb, s);
}

// A small minibatch on a small forest in one CTA, with the forest in shared
// memory: loaded, joined as in join_edges, flattened and written back, so that
// no compression is left to do. Bound by latency: the chains of dependent
// reads and links that many edges on few vertices make (most of all on an empty
// forest) take tens of cycles a step here instead of hundreds of nanoseconds a
// step in L2, and one launch takes the place of two: four minibatches of 4096
// edges on an empty forest of 4096 vertices, each with a query, 37.4 -> 34.3 us.
constexpr int kSmallBlock = 1024;

__global__ void __launch_bounds__(kSmallBlock)
k_update_small(int* __restrict__ parent, int n, const int* __restrict__ edges, int k, int vec,
               DevState* __restrict__ ds, int early) {
    extern __shared__ int4 small_forest[];
    int* sp = reinterpret_cast<int*>(small_forest);
    __shared__ int part[kSmallBlock / 32];
    pdl_trigger();
    const int tid = threadIdx.x;
    int u[2] = {}, v[2] = {};
    if (!early) pdl_wait();
    if (2 * tid < k) load_pairs<2>(edges, 2 * tid, k, vec, u, v);
    if (early) pdl_wait();
    const int quads = n / 4;
    for (int c = tid; c < quads; c += kSmallBlock) small_forest[c] = reinterpret_cast<const int4*>(parent)[c];
    if (tid < n - 4 * quads) sp[4 * quads + tid] = parent[4 * quads + tid];
    __syncthreads();
    int made = 0;
    bool bad = false;
    for (int i0 = 2 * tid; i0 < k; i0 += 2 * kSmallBlock) {
        int nu[2] = {}, nv[2] = {};
        if (i0 + 2 * kSmallBlock < k) load_pairs<2>(edges, i0 + 2 * kSmallBlock, k, vec, nu, nv);
#pragma unroll
        for (int i = 0; i < 2; i++) {
            if (i0 + i >= k) continue;
            if (!(in_range(u[i], n) && in_range(v[i], n))) {
                bad = true;
                continue;
            }
            int hi = u[i] > v[i] ? u[i] : v[i], lo = u[i] > v[i] ? v[i] : u[i], bhi = -1, blo = -1;
            while (hi != lo) {
                volatile int* vp = sp;
                int p = vp[hi];
                if (p == hi) {
                    p = atomicCAS(sp + hi, hi, lo);
                    if (p == hi) {
                        made++;
                        break;
                    }
                }
                if (p > hi) {  // broken invariant: stop rather than loop
                    flag(ds, ST_CORRUPT);
                    break;
                }
                if (bhi >= 0) vp[bhi] = p;  // splitting: skip a level
                const int below = hi;
                const bool swap = p < lo;
                hi = swap ? lo : p;
                bhi = swap ? blo : below;
                lo = swap ? p : lo;
                blo = swap ? below : blo;
            }
        }
#pragma unroll
        for (int i = 0; i < 2; i++) {
            u[i] = nu[i];
            v[i] = nv[i];
        }
    }
    if (bad) flag(ds, ST_RANGE);
    made = __reduce_add_sync(0xffffffffu, made);
    if ((tid & 31) == 0) part[tid >> 5] = made;
    __syncthreads();
    if (tid == 0) {
        int t = 0;
        for (int w = 0; w < kSmallBlock / 32; w++) t += part[w];
        if (t) atomicAdd(&ds->unions, (unsigned long long)t);
    }
    for (int c = tid; c < quads; c += kSmallBlock) {
        const int4 q = small_forest[c];
        const int4 w = make_int4(walk_root(sp, q.x, sp[q.x]), walk_root(sp, q.y, sp[q.y]),
                                 walk_root(sp, q.z, sp[q.z]), walk_root(sp, q.w, sp[q.w]));
        reinterpret_cast<int4*>(parent)[c] = w;
    }
    if (tid < n - 4 * quads) {
        const int x = sp[4 * quads + tid];
        parent[4 * quads + tid] = walk_root(sp, x, sp[x]);
    }
}

bool small_update(int64_t n, int64_t k, bool compress) {
    return n <= kSmallVertices && k <= (compress ? kSmallEdges : kSmallEdges / 2);
}

cudaError_t launch_update_small(int* parent, int n, const int* edges, int64_t k, DevState* ds, int pdl,
                                cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    launch_windowed_smem(k_update_small, 1u, kSmallBlock, sizeof(int4) * (size_t)((n + 3) / 4), s, nullptr, pdl != 0,
                         parent, n, edges, (int)k, pair_vec(edges), ds, (int)(pdl == 2));
    return cudaGetLastError();
}

// Variant 0 takes the tile kernel (variant 5) in CTAs of 128 threads from this
// many edges, about one wave of its tiles, and one chunk per thread below.
// Whole passes with a compression after each minibatch, 2 edges per thread, one
// chunk per thread (256 threads) against tiles (128): R-MAT n = 2^22 with 2^20
// edges a minibatch 1277 and 926 us, 2^18 583 and 540, 2^17 470 and 518; a 3001 x
// 3001 mesh 1225 and 888 with 2^20, 1042 and 992 with 2^18; R-MAT n = 2^24 with
// 2^22 2230 and 1315; 50,000 edges on 10^6 vertices 931 and 1098. Tiles of 256
// threads: 995 us with 2^20, 535 with 2^18.
constexpr int64_t kTileEdges = 1 << 18;

cudaError_t launch_update(int* parent, int n, const int* edges, int64_t k, DevState* ds,
                          Launch cfg, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    const int vec = pair_vec(edges);
    if (dense(k, n)) cfg.hook |= HOOK_AGAIN;
    if (cfg.variant == 0 && k >= kTileEdges) {
        cfg.variant = 5;
        cfg.block = 128;
    } else if (cfg.variant == 0) {
        cfg.ept = spread(cfg.ept, k, cfg.block);
    }
#define CC_UPD(E, P) update_inst<E, P>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, cfg.variant ? cfg.warphook : 0, BigArgs{cfg.big, cfg.alt}, s)
    switch (cfg.variant * 8 + cfg.ept) {
        case 1: case 9: CC_UPD(1, false); break;
        case 2: case 10: CC_UPD(2, false); break;
        case 4: case 12: CC_UPD(4, false); break;
        case 17: CC_UPD(1, true); break;
        case 18: CC_UPD(2, true); break;
        case 20: CC_UPD(4, true); break;
        case 25: update_deep_inst<1>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, cfg.warphook, BigArgs{cfg.big, cfg.alt}, s); break;
        case 26: update_deep_inst<2>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, cfg.warphook, BigArgs{cfg.big, cfg.alt}, s); break;
        case 28: update_deep_inst<4>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, cfg.warphook, BigArgs{cfg.big, cfg.alt}, s); break;
        case 41: update_tiles_inst<1>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, BigArgs{cfg.big, cfg.alt}, s); break;
        case 42: update_tiles_inst<2>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, BigArgs{cfg.big, cfg.alt}, s); break;
        case 44: update_tiles_inst<4>(edges, k, vec, parent, n, ds, cfg.block, cfg.window, cfg.pdl, cfg.hook, BigArgs{cfg.big, cfg.alt}, s); break;
        default: return cudaErrorInvalidValue;
    }
#undef CC_UPD
    return cudaGetLastError();
}

// ------------------------------------------------------------- Bulk-Query

template <int E>
__device__ __forceinline__ void store_answers(uint8_t* __restrict__ out, int64_t e0, int64_t k,
                                              bool ovec, const uint8_t (&a)[E]) {
    if (ovec && e0 + E <= k) {
        if (E == 4) {
            uchar4 w = make_uchar4(a[0], a[E > 1 ? 1 : 0], a[E > 2 ? 2 : 0], a[E > 3 ? 3 : 0]);
            __stcs(reinterpret_cast<uchar4*>(out + e0), w);
            return;
        }
        if (E == 2) {
            uchar2 w = make_uchar2(a[0], a[E > 1 ? 1 : 0]);
            __stcs(reinterpret_cast<uchar2*>(out + e0), w);
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < E; i++)
        if (e0 + i < k) out[e0 + i] = a[i];
}

// One chunk of Algorithm 1: the E pairs (u, v) of this thread, answers in a.
// Returns whether a pair had an id outside [0, n). MODE as for k_query. With
// a largest-component bitmap, a pair whose endpoints are both marked is
// answered 1 from the bitmap alone: it reads no parent and walks nothing.
//
// Ids fall along every path, so a root that is larger than the other side's node
// cannot be that side's root: the pair is answered 0 there, and the other side is
// not read any further. Otherwise the larger node is replaced by its parent; nodes
// that meet answer 1.
//  LAZY: only the larger node is moved up, and the smaller endpoint's parent is read
//        only once the larger one's has not decided the pair. On a large forest the
//        kernel is bound by the gathers (one line per clock and SM from L2, 71 G/s from
//        DRAM), so what is not read is what it gains: reading both endpoints and walking
//        both to their roots, a pass over the R-MAT stream (n = 2^24, 128 x 2^20 pairs,
//        no compression) took 4.25 ms and now takes 3.89; the 8192 x 8192 grid (32 x 2^22
//        pairs) 8.48 and now 7.01. Otherwise both nodes are read in a round and both
//        moved up, which takes fewer rounds one after the other.
template <int E, int MODE, bool LAZY>
__device__ __forceinline__ bool query_chunk(int* __restrict__ parent, int n, const int (&u)[E], const int (&v)[E],
                                            int64_t e0, int64_t k, uint8_t (&a)[E],
                                            DevState* __restrict__ ds, const unsigned* bits) {
    int hi[E], lo[E];
    bool act[E];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < E; i++) {
        bool ok = e0 + i < k;
        if (ok && !(in_range(u[i], n) && in_range(v[i], n))) {
            ok = false;
            bad = true;
        }
        a[i] = ok && u[i] == v[i];
        act[i] = ok && u[i] != v[i];
        hi[i] = u[i] > v[i] ? u[i] : v[i];
        lo[i] = u[i] > v[i] ? v[i] : u[i];
    }
    if (bits) {
#pragma unroll
        for (int i = 0; i < E; i++)
            if (act[i] && big_member(bits, hi[i]) && big_member(bits, lo[i])) {
                a[i] = 1;
                act[i] = false;
            }
    }
    int p[E], q[E];
    if constexpr (MODE == 2) {
#pragma unroll
        for (int i = 0; i < E; i++) {
            p[i] = act[i] ? load_after(parent + hi[i]) : 0;
            if (!LAZY) q[i] = act[i] ? load_after(parent + lo[i]) : 0;
        }
        if (LAZY) {
#pragma unroll
            for (int i = 0; i < E; i++)  // p > lo: lo's root is another; p == lo: lo is the root
                q[i] = act[i] && p[i] < lo[i] ? load_after(parent + lo[i]) : lo[i];
        }
#pragma unroll
        for (int i = 0; i < E; i++)
            if (act[i]) a[i] = p[i] == q[i];
        return bad;
    }
    // the node below hi (lo) on its walk, which is repointed past it (MODE 1); -1 at the endpoint
    int bhi[E], blo[E];
#pragma unroll
    for (int i = 0; i < E; i++) bhi[i] = blo[i] = -1;
    if constexpr (!LAZY) {
#pragma unroll
        for (int i = 0; i < E; i++) {
            p[i] = q[i] = 0;
            if (!act[i]) continue;
            p[i] = load_after(parent + hi[i]);
            q[i] = load_after(parent + lo[i]);
        }
#pragma unroll
        for (int i = 0; i < E; i++) {
            if (!act[i]) continue;
            if (p[i] > hi[i] || q[i] > lo[i]) flag(ds, ST_CORRUPT);
            a[i] = p[i] == q[i] || p[i] == lo[i];
            // decided, or one of them is a root above the other side's node
            if (a[i] || p[i] >= hi[i] || (q[i] >= lo[i] && p[i] < lo[i])) {
                act[i] = false;
                continue;
            }
            bhi[i] = hi[i];
            blo[i] = q[i] < lo[i] ? lo[i] : -1;
            const bool swap = p[i] < q[i];
            hi[i] = swap ? q[i] : p[i];
            lo[i] = swap ? p[i] : q[i];
            const int t = bhi[i];
            bhi[i] = swap ? blo[i] : t;
            blo[i] = swap ? t : blo[i];
        }
    }
    while (true) {
        bool any = false;
#pragma unroll
        for (int i = 0; i < E; i++) {
            p[i] = q[i] = 0;
            if (!act[i]) continue;
            p[i] = load_after(parent + hi[i]);
            q[i] = lo[i];
            if constexpr (!LAZY) q[i] = load_after(parent + lo[i]);
            any = true;
        }
        if (!any) break;
#pragma unroll
        for (int i = 0; i < E; i++) {
            if (!act[i]) continue;
            if (p[i] >= hi[i] || q[i] > lo[i]) {  // a root above lo's id, or a broken invariant: not connected
                if (p[i] > hi[i] || q[i] > lo[i]) flag(ds, ST_CORRUPT);
                act[i] = false;
                continue;
            }
            int beside = blo[i];
            if (MODE == 1 && bhi[i] >= 0) lower(parent, bhi[i], p[i]);  // splitting: skip a level
            if constexpr (!LAZY) {
                if (MODE == 1 && blo[i] >= 0 && q[i] < lo[i]) lower(parent, blo[i], q[i]);
                if (q[i] < lo[i]) beside = lo[i];
            }
            if (p[i] == lo[i] || p[i] == q[i]) {
                a[i] = 1;
                act[i] = false;
                continue;
            }
            const bool swap = p[i] < q[i];
            const int below = hi[i];
            hi[i] = swap ? q[i] : p[i];
            lo[i] = swap ? p[i] : q[i];
            bhi[i] = swap ? beside : below;
            blo[i] = swap ? below : beside;
        }
    }
    return bad;
}

// Algorithm 1 over E pairs per thread. Lanes of a warp own consecutive pairs,
// so the pair loads (16 B per lane) and the answer stores (E bytes per lane)
// are coalesced across the warp. The E walks of a thread advance in lockstep,
// so their loads overlap.
//  MODE 0: read-only finds.
//  MODE 1: finds with path splitting: every node walked over is repointed at
//          its grandparent.
//  MODE 2: flat forest (every tree of height <= 1): the parents decide.
// LAZY: see query_chunk.
// PERSIST: a persistent grid that loads the next chunk's pairs before working
// on the current one, so those loads overlap the parent reads.
// early: as for k_update.
template <int E, int MODE, bool PERSIST, bool LAZY>
__global__ void __launch_bounds__(1024)
k_query(int* __restrict__ parent, int n, const int* __restrict__ pairs, int64_t k, int vec,
        uint8_t* __restrict__ out, int ovec, DevState* __restrict__ ds, int early,
        const unsigned* __restrict__ big) {
    pdl_trigger();
    if (!early) pdl_wait();
    int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * E;
    if (e0 >= k) return;
    bool bad = false;
    int u[E], v[E];
    uint8_t a[E];
    load_pairs<E>(pairs, e0, k, vec, u, v);
    if (early) pdl_wait();
    const unsigned* bits = big_active(big, ds);
    if (!PERSIST) {
        bad = query_chunk<E, MODE, LAZY>(parent, n, u, v, e0, k, a, ds, bits);
        store_answers<E>(out, e0, k, ovec != 0, a);
    } else {
        const int64_t stride = (int64_t)gridDim.x * blockDim.x * E;
        while (e0 < k) {
            const int64_t nx = e0 + stride;
            int nu[E] = {}, nv[E] = {};
            if (nx < k) load_pairs<E>(pairs, nx, k, vec, nu, nv);
            bad |= query_chunk<E, MODE, LAZY>(parent, n, u, v, e0, k, a, ds, bits);
            store_answers<E>(out, e0, k, ovec != 0, a);
#pragma unroll
            for (int i = 0; i < E; i++) {
                u[i] = nu[i];
                v[i] = nv[i];
            }
            e0 = nx;
        }
    }
    if (bad) flag(ds, ST_RANGE);
}

// Algorithm 1 with the warp as the unit of work. A warp takes chunks of
// 32 * CH consecutive pairs; each lane keeps S pairs in flight, and every
// round advances each unfinished walk one step (read-only, as MODE 0: all
// of a lane's loads of a round are independent). A finished pair writes its
// answer, and its slot takes the next pair of the chunk at once: a ballot
// over the finished slots gives each a distinct index, so the lanes whose
// walks are short keep working while another lane walks a long path, instead
// of idling until the warp's longest walk ends. A pair whose first parents
// are equal is answered after its first round.
template <int S, int CH>
__global__ void __launch_bounds__(1024)
k_query_warp(const int* __restrict__ parent, int n, const int* __restrict__ pairs, int64_t k, int vec,
             uint8_t* __restrict__ out, DevState* __restrict__ ds) {
    pdl_trigger();
    pdl_wait();
    const unsigned full = 0xffffffffu;
    const int lane = (int)(threadIdx.x & 31u);
    const unsigned lt = (1u << lane) - 1u;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    bool bad = false, corrupt = false;
    for (int64_t base = warp * 32 * CH; base < k; base += nwarps * 32 * CH) {
        const int64_t end = base + 32 * CH < k ? base + 32 * CH : k;
        int64_t next = base;  // warp-uniform: the next pair of the chunk not yet taken
        int64_t idx[S];
        int xu[S], pu[S], xv[S], pv[S];
        bool act[S], eq[S];
#pragma unroll
        for (int j = 0; j < S; j++) {
            act[j] = false;
            eq[j] = false;
            idx[j] = 0;
            xu[j] = pu[j] = xv[j] = pv[j] = 0;
        }
        bool take[S];
#pragma unroll
        for (int j = 0; j < S; j++) take[j] = true;
        while (true) {
            // hand the next pairs of the chunk to the slots that are free
#pragma unroll
            for (int j = 0; j < S; j++) {
                const unsigned want = __ballot_sync(full, take[j]);
                if (take[j]) {
                    idx[j] = next + __popc(want & lt);
                    act[j] = idx[j] < end;
                    if (act[j]) {
                        int u, v;
                        if (vec >= 1) {
                            const int2 q = __ldcs(reinterpret_cast<const int2*>(pairs) + idx[j]);
                            u = q.x;
                            v = q.y;
                        } else {
                            u = __ldcs(pairs + 2 * idx[j]);
                            v = __ldcs(pairs + 2 * idx[j] + 1);
                        }
                        if (!(in_range(u, n) && in_range(v, n))) {
                            bad = true;
                            out[idx[j]] = 0;
                            act[j] = false;
                        } else {
                            xu[j] = u;
                            xv[j] = v;
                            pu[j] = load_after(parent + u);
                            pv[j] = load_after(parent + v);
                            eq[j] = pu[j] == pv[j];
                        }
                    }
                    take[j] = false;
                }
                next += __popc(want);
            }
            bool any = false;
#pragma unroll
            for (int j = 0; j < S; j++) any |= act[j];
            if (!__any_sync(full, any) && next >= end) break;
            // one step of every unfinished walk; finished pairs answer and free their slot
#pragma unroll
            for (int j = 0; j < S; j++) {
                if (!act[j]) {
                    take[j] = next < end;  // an idle slot takes a pair while the chunk has any
                    continue;
                }
                if (!eq[j] && pu[j] < xu[j]) {
                    xu[j] = pu[j];
                    pu[j] = load_after(parent + xu[j]);
                }
                if (!eq[j] && pv[j] < xv[j]) {
                    xv[j] = pv[j];
                    pv[j] = load_after(parent + xv[j]);
                }
                if (eq[j] || (pu[j] >= xu[j] && pv[j] >= xv[j])) {
                    if (!eq[j] && (pu[j] > xu[j] || pv[j] > xv[j])) corrupt = true;
                    out[idx[j]] = (uint8_t)(eq[j] || xu[j] == xv[j]);
                    act[j] = false;
                    take[j] = true;
                }
            }
        }
    }
    if (bad) flag(ds, ST_RANGE);
    if (corrupt) flag(ds, ST_CORRUPT);
}

template <int E, int MODE, bool PERSIST, bool LAZY>
static void query_one(unsigned g, int block, const cudaAccessPolicyWindow* window, int pdl, cudaStream_t s,
                      int* parent, int n, const int* pairs, int64_t k, int vec, uint8_t* out, int ovec,
                      DevState* ds, const unsigned* big) {
    if (PERSIST) {
        const int c = resident_grid<k_query<E, MODE, PERSIST, LAZY>>(block);
        if (g > (unsigned)c) g = (unsigned)c;
    }
    launch_windowed(k_query<E, MODE, PERSIST, LAZY>, g, block, s, window, pdl != 0, parent, n, pairs, k, vec, out,
                    ovec, ds, (int)(pdl == 2), big);
}

template <int MODE, bool LAZY>
static void query_inst(unsigned g, Launch cfg, cudaStream_t s, int* parent, int n,
                       const int* pairs, int64_t k, int vec, uint8_t* out, int ovec, DevState* ds) {
#define CC_Q(E, P) query_one<E, MODE, P, LAZY>(g, cfg.block, cfg.window, cfg.pdl, s, parent, n, pairs, k, vec, out, ovec, ds, cfg.big)
    const bool persist = cfg.query_variant == 1;
    switch (cfg.ept) {
        case 1: if (persist) CC_Q(1, true); else CC_Q(1, false); break;
        case 2: if (persist) CC_Q(2, true); else CC_Q(2, false); break;
        default: if (persist) CC_Q(4, true); else CC_Q(4, false); break;
    }
#undef CC_Q
}

// LAZY of query_chunk from this many pairs and vertices. Fewer pairs leave the
// latency of a round unhidden (50,001 on 10^6 vertices: 0.1 us more a query). Smaller
// forests stay near the SMs: 2^20 pairs on a forest that two updates left deep, lazy
// and not, 9.5 and 7.9 us for n = 2^10, 12.0 and 10.5 for 2^16, 14.4 and 13.7 for 2^20. On
// larger ones, passes of 6 to 24 minibatches of 2^17 to 2^21 edges and pairs without
// compression take 1.00 to 1.08 times as long without it for n = 2^22 to 2^24 and
// 1.00 to 1.17 for 2^26.
constexpr int64_t kLazyPairs = 1 << 17;
constexpr int kLazyVertices = 1 << 22;

cudaError_t launch_query(int* parent, int n, const int* pairs, int64_t k, uint8_t* out,
                         DevState* ds, int mode, Launch cfg, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    if (cfg.query_variant == 2) {  // warp-cooperative, read-only walks whatever the mode
        constexpr int kS = 2, kCH = 16;
        const int64_t warps = (k + 32 * kCH - 1) / (32 * kCH);
        int64_t g = (warps * 32 + cfg.block - 1) / cfg.block;
        const int64_t cap = resident_grid<k_query_warp<kS, kCH>>(cfg.block);
        if (g > cap) g = cap;
        launch_windowed(k_query_warp<kS, kCH>, (unsigned)g, cfg.block, s, cfg.window, cfg.pdl != 0, (const int*)parent,
                        n, pairs, k, pair_vec(pairs), out, ds);
        return cudaGetLastError();
    }
    if (cfg.qept) cfg.ept = cfg.qept;
    if (cfg.query_variant == 0) cfg.ept = spread(cfg.ept, k, cfg.block);
    const int vec = pair_vec(pairs);
    const int ovec = (reinterpret_cast<uintptr_t>(out) % cfg.ept) == 0;
    const unsigned g = blocks_for(k, (int64_t)cfg.ept * cfg.block);
    const bool lazy = k >= kLazyPairs && n >= kLazyVertices;
#define CC_QM(M) if (lazy) query_inst<M, true>(g, cfg, s, parent, n, pairs, k, vec, out, ovec, ds); \
                 else query_inst<M, false>(g, cfg, s, parent, n, pairs, k, vec, out, ovec, ds)
    switch (mode) {
        case 2: CC_QM(2); break;
        case 1: CC_QM(1); break;
        default: CC_QM(0); break;
    }
#undef CC_QM
    return cudaGetLastError();
}

// ------------------------------------------------------------ compression

// Every vertex is pointed at its root (4 consecutive vertices per thread, one
// 16-byte read of their parents). The parents of the four parents are read at
// once, a root's own too, and where all are roots, as most are, nothing is left to
// do; else the four walks go on from there in lockstep. That straight path is what
// bounds the pass, which issues its instructions at 60 % of the rate: with one loop
// from the vertices up it took 10.0 us for 4.2 million R-MAT vertices and takes
// 8.3, 45 and 34 for 33.6 million, 21.6 and 20.5 for 9 million of a mesh. Only
// entries that change are written. With OUT, the roots are also written to
// out[] -- the minimum-id labels, since the root is the smallest id of its
// tree. No hooks run concurrently, so the roots are fixed for the whole pass.
// With BIG, the pass also rewrites the largest-component bitmap: bit v = (the
// root of v is ds->big_root), one 32-bit word per 8 lanes (a warp covers 128
// consecutive vertices); every lane of a warp takes part, so threads past n
// do not leave early. (Counting the marked vertices here, one atomic per warp
// on one word, doubled the pass: launch_big_count does it on demand.) With BIG
// four parents are written back as one vector if any changed: these passes come
// after several minibatches, so that most have (2^26 vertices of the grid: 178 ->
// 158 us a pass, and 148 with the straight path); where one minibatch went before, single stores are the faster
// ones (2^25 vertices of an R-MAT graph: 45 and 48 us).
// As a dependent launch it starts while the update drains, where a plain launch
// costs a boundary of about 2 us on each side (ragged minibatches on 10^6
// vertices, three kernels a step: 1250 -> 1011 us for 104 steps). It has no
// explicit trigger, so its own dependents start as its CTAs exit: with one after
// the wait, the kernels that follow all came in at once to wait (1195 us).
template <bool OUT, bool BIG>
__global__ void __launch_bounds__(1024)
k_compress_all(int* __restrict__ parent, int64_t n, int* __restrict__ out,
               DevState* __restrict__ ds, unsigned* __restrict__ big) {
    pdl_wait();
    const int64_t v0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    if (!BIG && v0 >= n) return;
    const bool full = v0 + 4 <= n;
    int p0[4], x[4], p[4];
    bool done = full;  // every vertex points at its root already
    if (full) {
        const int v = (int)v0;
        const int4 q = *reinterpret_cast<const int4*>(parent + v0);
        p0[0] = q.x; p0[1] = q.y; p0[2] = q.z; p0[3] = q.w;
#pragma unroll
        for (int i = 0; i < 4; i++) x[i] = p0[i] < v + i ? p0[i] : v + i;  // never past v, in a broken forest either
#pragma unroll
        for (int i = 0; i < 4; i++) p[i] = parent[x[i]];
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (x[i] != p0[i]) p[i] = p0[i];
            done &= p[i] == x[i];
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            p[i] = p0[i] = v0 + i < n ? parent[v0 + i] : 0;
            x[i] = v0 + i < n ? (int)(v0 + i) : 0;  // past n: a walk of length 0
        }
    }
    bool changed = false;
    if (!done) {
        while (true) {
            bool any = false;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                if (p[i] < x[i]) {
                    x[i] = p[i];
                    p[i] = parent[x[i]];
                    any = true;
                }
            }
            if (!any) break;
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            if (p[i] > x[i]) flag(ds, ST_CORRUPT);
            if ((!BIG || !full) && (full || v0 + i < n) && x[i] != p0[i]) parent[v0 + i] = x[i];
            changed |= x[i] != p0[i];
        }
    }
    if (BIG && full && changed) reinterpret_cast<int4*>(parent)[v0 / 4] = make_int4(x[0], x[1], x[2], x[3]);
    if (OUT) {
        if (full) {
            reinterpret_cast<int4*>(out)[v0 / 4] = make_int4(x[0], x[1], x[2], x[3]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (v0 + i < n) out[v0 + i] = x[i];
        }
    }
    if (BIG) {
        const int R = ds->big_root;  // the same for every thread
        if (R < 0) return;
        unsigned nib = 0;
#pragma unroll
        for (int i = 0; i < 4; i++)
            if ((full || v0 + i < n) && x[i] == R) nib |= 1u << i;
        const unsigned lane = threadIdx.x & 31u;
        unsigned w = nib << ((lane & 7u) * 4u);
        w |= __shfl_xor_sync(0xffffffffu, w, 1);
        w |= __shfl_xor_sync(0xffffffffu, w, 2);
        w |= __shfl_xor_sync(0xffffffffu, w, 4);
        if ((lane & 7u) == 0 && v0 < n) big[v0 >> 5] = w;  // word v0 / 32 holds vertices v0 .. v0 + 31
    }
}

// ds->big_members += the set bits of words[0, nwords): one atomic per CTA.
__global__ void __launch_bounds__(256)
k_big_count(const unsigned* __restrict__ words, int64_t nwords, DevState* __restrict__ ds) {
    __shared__ unsigned part[8];
    unsigned c = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nwords; i += (int64_t)gridDim.x * blockDim.x)
        c += (unsigned)__popc(words[i]);
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long t = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += part[w];
        if (t) atomicAdd(&ds->big_members, t);
    }
}

cudaError_t launch_big_count(const unsigned* words, int64_t nwords, DevState* ds, cudaStream_t s) {
    if (nwords <= 0) return cudaSuccess;
    int64_t g = (nwords + 255) / 256;
    if (g > 1024) g = 1024;
    k_big_count<<<(unsigned)g, 256, 0, s>>>(words, nwords, ds);
    return cudaGetLastError();
}

// The root of the largest tree, estimated (the sampling step of Afforest's
// large-component skip): kBigSample vertices, spread over [0, n) by the
// golden-ratio sequence, are walked to their roots (read-only); the roots go
// into a shared-memory hash table with a count each, and the most frequent
// one (the smaller id on a tie) becomes ds->big_root if at least min_share of
// the sample reached it, else -1. One CTA of kBigSample threads.
__global__ void __launch_bounds__(kBigSample)
k_big_pick(const int* parent, int64_t n, int min_share, DevState* __restrict__ ds) {
    pdl_wait();
    constexpr int kSlots = 2 * kBigSample;
    __shared__ int key[kSlots];
    __shared__ int cnt[kSlots];
    __shared__ unsigned long long best[kBigSample / 32];
    const int t = threadIdx.x;
    for (int i = t; i < kSlots; i += blockDim.x) {
        key[i] = -1;
        cnt[i] = 0;
    }
    // x = floor(frac((t + 1) * phi) * n), in [0, n)
    const uint64_t h = (uint64_t)(t + 1) * 0x9E3779B97F4A7C15ull;
    const int x = (int)(((h >> 32) * (uint64_t)n) >> 32);
    const int r = walk_root(parent, x, parent[x]);
    __syncthreads();
    unsigned slot = ((unsigned)r * 0x9E3779B1u) >> 21;  // 11 bits: kSlots slots
    for (int probe = 0; probe < kSlots; probe++) {       // at most kBigSample keys: a free slot exists
        const int prev = atomicCAS(&key[slot], -1, r);
        if (prev == -1 || prev == r) {
            atomicAdd(&cnt[slot], 1);
            break;
        }
        slot = (slot + 1) & (kSlots - 1);
    }
    __syncthreads();
    // (count, then the smaller id) as one 64-bit key; the maximum wins
    unsigned long long mine = 0;
    for (int i = t; i < kSlots; i += blockDim.x)
        if (cnt[i]) {
            const unsigned long long c = ((unsigned long long)cnt[i] << 32) | (unsigned)(0x7fffffff - key[i]);
            if (c > mine) mine = c;
        }
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mine, d);
        if (o > mine) mine = o;
    }
    if ((t & 31) == 0) best[t >> 5] = mine;
    __syncthreads();
    if (t == 0) {
        unsigned long long b = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++)
            if (best[w] > b) b = best[w];
        const int count = (int)(b >> 32);
        const int root = 0x7fffffff - (int)(b & 0xffffffffu);
        ds->big_root = (b && count >= min_share) ? root : -1;
    }
}

cudaError_t launch_big_pick(const int* parent, int64_t n, int min_share, DevState* ds, bool pdl, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    launch_windowed(k_big_pick, 1u, kBigSample, s, nullptr, pdl, parent, n, min_share, ds);
    return cudaGetLastError();
}

cudaError_t launch_compress_all(int* parent, int64_t n, int* out, DevState* ds, int block, bool pdl,
                                cudaStream_t s, unsigned* big) {
    const unsigned g = blocks_for(n, 4LL * block);
    // labels into a buffer without 16-byte alignment: compress, then copy
    int* direct = reinterpret_cast<uintptr_t>(out) % 16 == 0 ? out : nullptr;
    if (direct) {
        if (big) launch_windowed(k_compress_all<true, true>, g, block, s, nullptr, pdl, parent, n, direct, ds, big);
        else launch_windowed(k_compress_all<true, false>, g, block, s, nullptr, pdl, parent, n, direct, ds, big);
    } else {
        if (big) launch_windowed(k_compress_all<false, true>, g, block, s, nullptr, pdl, parent, n, direct, ds, big);
        else launch_windowed(k_compress_all<false, false>, g, block, s, nullptr, pdl, parent, n, direct, ds, big);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && out && !direct)
        e = cudaMemcpyAsync(out, parent, (size_t)n * sizeof(int), cudaMemcpyDeviceToDevice, s);
    return e;
}

// Section 5.1's pragmatic compression for the endpoints of an edge array:
// find the root, then walk the path again pointing every node at it.
template <int E>
__global__ void __launch_bounds__(1024)
k_compress_touched(int* __restrict__ parent, int n, const int* __restrict__ edges, int64_t k,
                   int vec, DevState* __restrict__ ds) {
    pdl_wait();
    const int64_t e0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * E;
    if (e0 >= k) return;
    int u[E], v[E];
    load_pairs<E>(edges, e0, k, vec, u, v);
#pragma unroll
    for (int j = 0; j < 2 * E; j++) {
        const int i = j >> 1;
        int x = (j & 1) ? v[i] : u[i];
        if (e0 + i >= k || !in_range(x, n)) continue;
        int p = parent[x];
        if (p >= x) continue;
        const int r = walk_root(parent, x, p);
        while (p != r && p < x) {
            lower(parent, x, r);
            x = p;
            p = parent[x];
        }
    }
}

cudaError_t launch_compress_touched(int* parent, int n, const int* edges, int64_t k,
                                    DevState* ds, Launch cfg, cudaStream_t s) {
    if (k <= 0) return cudaSuccess;
    const int vec = pair_vec(edges);
    const unsigned g = blocks_for(k, (int64_t)cfg.ept * cfg.block);
    switch (cfg.ept) {
        case 1: launch_windowed(k_compress_touched<1>, g, cfg.block, s, nullptr, cfg.pdl != 0, parent, n, edges, k, vec, ds); break;
        case 2: launch_windowed(k_compress_touched<2>, g, cfg.block, s, nullptr, cfg.pdl != 0, parent, n, edges, k, vec, ds); break;
        default: launch_windowed(k_compress_touched<4>, g, cfg.block, s, nullptr, cfg.pdl != 0, parent, n, edges, k, vec, ds); break;
    }
    return cudaGetLastError();
}

// ------------------------------------------------------- label validation

// Checks an array loaded from outside and counts its roots: LABELS wants
// 0 <= a[v] <= v and a[a[v]] == a[v], else only 0 <= a[v] <= v. Bound by the
// stream of n ids plus, for labels, the gather of each label's own label (one
// hot line where a giant component holds most ids). Each thread has four
// quadruples, whose loads (16 bytes where the array allows it) and then gathers
// are all in flight together, and a CTA makes ONE atomic on the root counter:
// with one per warp, 2^25 ids queued 2^20 atomics on that word and the pass took
// 668 us; on a resident grid with a quadruple per thread and step 49; now 35.
template <bool LABELS>
__global__ void __launch_bounds__(256)
k_validate(const int* __restrict__ a, int64_t n, int vec, DevState* __restrict__ ds) {
    __shared__ int part[8];
    constexpr int Q = 4;
    const int64_t first = (int64_t)blockIdx.x * (256 * 4 * Q);
    int roots = 0;
    bool bad = false;
    if (vec && first + 256 * 4 * Q <= n) {
        int x[Q][4], y[Q][4];
        const int v0 = (int)first + 4 * (int)threadIdx.x;
#pragma unroll
        for (int j = 0; j < Q; j++) {
            const int4 q = *reinterpret_cast<const int4*>(a + v0 + 1024 * j);
            x[j][0] = q.x; x[j][1] = q.y; x[j][2] = q.z; x[j][3] = q.w;
        }
        if (LABELS) {
#pragma unroll
            for (int j = 0; j < Q; j++)
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const int v = v0 + 1024 * j + i;
                    y[j][i] = a[(unsigned)x[j][i] < (unsigned)v ? x[j][i] : v];  // stays in range
                }
        }
#pragma unroll
        for (int j = 0; j < Q; j++)
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const int v = v0 + 1024 * j + i;
                bad |= (unsigned)x[j][i] > (unsigned)v || (LABELS && y[j][i] != x[j][i]);
                roots += x[j][i] == v;
            }
    } else {
        for (int j = 0; j < Q * 4; j++) {
            const int64_t v = first + 256 * j + threadIdx.x;
            if (v >= n) break;
            const int x = a[v];
            const bool in = x >= 0 && (int64_t)x <= v;
            bad |= !in || (LABELS && a[x] != x);
            roots += (int64_t)x == v;
        }
    }
    if (bad) atomicOr(&ds->checked.bad, 1u);
    roots = __reduce_add_sync(0xffffffffu, roots);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = roots;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < 8; w++) t += part[w];
        if (t) atomicAdd(&ds->checked.roots, (unsigned long long)t);
    }
}

template <bool LABELS>
static cudaError_t validate(const int* a, int64_t n, DevState* ds, cudaStream_t s) {
    k_validate<LABELS><<<blocks_for(n, 4096), 256, 0, s>>>(a, n, pair_vec(a) == 2, ds);
    return cudaGetLastError();
}

// dst = src, n ids (dst 16-byte aligned). With ADOPT the forest becomes src,
// which has been validated: also unions links made, no tree marked; and the
// last ids go first, whose lines the validation has left in L2 (2^25 ids, with
// the device-to-device copy, the copy of the counter, the memset and the second
// synchronisation that it replaces: 20 us less of a 252 us restart).
template <bool ADOPT>
__global__ void __launch_bounds__(256)
k_copy_ids(const int* src, int64_t n, int vec, int* dst, DevState* __restrict__ ds, unsigned long long unions) {
    pdl_wait();
    if (ADOPT && blockIdx.x == 0 && threadIdx.x == 0) {
        ds->unions = unions;
        ds->big_root = -1;
        __threadfence();  // before any dependent starts, as in k_reset
    }
    const unsigned b = ADOPT ? gridDim.x - 1 - blockIdx.x : blockIdx.x;
    const int64_t v0 = ((int64_t)b * blockDim.x + threadIdx.x) * 4;
    if (v0 + 4 <= n) {
        int4 q;
        if (vec) q = *reinterpret_cast<const int4*>(src + v0);
        else q = make_int4(src[v0], src[v0 + 1], src[v0 + 2], src[v0 + 3]);
        *reinterpret_cast<int4*>(dst + v0) = q;
    } else {
        for (int64_t v = v0; v < n; v++) dst[v] = src[v];
    }
}

cudaError_t launch_adopt(const int* src, int64_t n, int* parent, DevState* ds, unsigned long long unions,
                         cudaStream_t s) {
    k_copy_ids<true><<<blocks_for(n, 1024), 256, 0, s>>>(src, n, pair_vec(src) == 2, parent, ds, unions);
    return cudaGetLastError();
}

cudaError_t launch_copy_ids(const int* parent, int64_t n, int* out, bool pdl, cudaStream_t s) {
    launch_windowed(k_copy_ids<false>, blocks_for(n, 1024), 256, s, nullptr, pdl, parent, n, 1, out,
                    (DevState*)nullptr, 0ull);
    return cudaGetLastError();
}

cudaError_t launch_validate_forest(const int* p, int64_t n, DevState* ds, cudaStream_t s) {
    return validate<false>(p, n, ds, s);
}

cudaError_t launch_validate_labels(const int* lab, int64_t n, DevState* ds, cudaStream_t s) {
    return validate<true>(lab, n, ds, s);
}

}  // namespace cc
