// Bulk-Find (Algorithm 4; Section 4): the roots of a set S of vertices with
// path compression for the whole set, in ONE cooperative kernel launch.
//
// Phase I walks up from all of S at once, one level per grid barrier: the
// frontier F_0 = removeDup(S), and every node of F_i that is not a root sends
// its parent on to F_{i+1} unless the parent was already visited or another
// flow got there first in this level (both are one atomic exchange on an
// epoch-stamped mark array, so "visited" never has to be cleared). This counts
// the traversed vertices and the levels. Every level's frontier holds at most
// |S| entries (each traversed node is on some query's path, and a path has
// one node per level).
//
// Phase II points every traversed node at its root. Algorithm 4 hands the
// roots back down the recorded paths through the Response Distributor, an
// index of all recorded (parent, node) pairs, because there a path that many
// queries share must be walked once only. Here each query walks its own path
// twice, first to the root (before the first barrier, while nothing is
// written) and then again to repoint it, which the writes of the others only
// shorten. The index cost more than it saved: a hash, a counting sort of all
// pairs and two or three kernels with a host round trip for every level going
// up and again going down, 243 us for 2^16 vertices of a flat R-MAT forest of
// 2^20 (13 launches); the walks are gathers that L2 serves. Now
// 21 us (65 against 265 us for 2^20 vertices). The work is the sum of the path
// lengths, also where paths are shared: 2^20 vertices at the ends of 350 chains of
// 3000 take 21 ms, 16 of them 10, a barrier for each level; with a launch for each
// 165 and 156 ms.
//
// What bounds it: the barriers (about 1.3 us each, one for the seed and one
// for each level) for small S, the gathers of the walks and the marks for
// large S. The grid is no larger than S needs, which keeps the barriers cheap.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "cc_append.cuh"
#include "cc_device.cuh"
#include "cc_internal.cuh"

namespace cc {

namespace {

constexpr int kBfBlock = 512;

// Whether this thread is the first of the call to reach x (x >= 0), among the
// lanes with `on`. Many nodes share a parent (a big tree's root) and query
// sets repeat popular vertices: within a warp one lane per distinct vertex
// stamps it, and a read that already shows this call's stamp skips the
// exchange, so they do not queue on one mark word. All lanes must call it.
__device__ __forceinline__ bool first_visit(bool on, int x, int* mark, int epoch) {
    const unsigned act = __ballot_sync(0xffffffffu, on);
    if (!on) return false;
    const unsigned g = __match_any_sync(act, x);
    return (unsigned)(__ffs(g) - 1) == (threadIdx.x & 31u) &&
           *(volatile const int*)(mark + x) != epoch && atomicExch(mark + x, epoch) != epoch;
}

// The forest may come from union by size, so the walks go on until p == x
// rather than rely on decreasing ids, and stop after n steps (a cycle, which
// is reported). parent, front and the counters are read and written by
// different CTAs between barriers: no read-only loads on them.
__global__ void __launch_bounds__(kBfBlock)
k_bulk_find(const int* S, int64_t k, int n, int* parent, int* mark, int epoch, int* front0,
            int* front1, int* roots, BulkFindCounters* c, int* res, uint8_t* __restrict__ out,
            DevState* ds) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x;
    const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
    BulkFindCounters::Stats* st = &c->stats[epoch & 1];
    // F_0, the roots, and the longest path
    unsigned depth = 0;
    for (int64_t i0 = first; i0 < k; i0 += stride) {  // block-uniform
        const int64_t i = i0 + threadIdx.x;
        const int s = i < k ? S[i] : -1;
        const bool ok = in_range(s, n);
        if (i < k && !ok) flag(ds, ST_RANGE);
        append1_block(first_visit(ok, s, mark, epoch), s, front0, &c->front[0]);
        if (i < k) {
            int x = s;
            if (ok) {
                unsigned d = 0;
                for (int p = parent[x]; p != x; d++) {
                    if (d > (unsigned)n) {
                        flag(ds, ST_CORRUPT);
                        break;
                    }
                    x = p;
                    p = parent[x];
                }
                depth = d > depth ? d : depth;
            }
            roots[i] = ok ? x : -1;
        }
    }
    grid.sync();
    depth = __reduce_max_sync(0xffffffffu, depth);
    if ((threadIdx.x & 31) == 0 && depth) atomicMax(&st->depth, depth);
    // Phase I: three frontier counters in turn, so that the one being cleared
    // is neither read nor appended through in the same level; all are zero at
    // the end, for the next call
    unsigned traversed = 0;
    int level = 0;
    for (;; level++) {
        const unsigned count = *(volatile const unsigned*)&c->front[level % 3];
        if (leader) c->front[(level + 2) % 3] = 0u;
        if (count == 0) break;
        const int* from = level & 1 ? front1 : front0;
        int* to = level & 1 ? front0 : front1;
        for (int64_t i0 = first; i0 < (int64_t)count; i0 += stride) {
            const int64_t i = i0 + threadIdx.x;
            int v = 0, p = 0;
            if (i < (int64_t)count) {
                v = from[i];
                p = parent[v];
            }
            traversed += p != v;
            append1_block(first_visit(p != v, p, mark, epoch), p, to, &c->front[(level + 1) % 3]);
        }
        grid.sync();
    }
    traversed = __reduce_add_sync(0xffffffffu, traversed);
    if ((threadIdx.x & 31) == 0 && traversed) atomicAdd(&st->traversed, (unsigned long long)traversed);
    if (leader) {
        st->levels = (unsigned)level;
        c->stats[(epoch + 1) & 1] = {};
    }
    // Phase II
    for (int64_t i = first + threadIdx.x; i < k; i += stride) {
        const int r = roots[i];
        if (r >= 0) {
            int x = S[i];
            for (int steps = 0; x != r && steps <= n; steps++) {
                const int p = parent[x];
                if (p == r) break;
                parent[x] = r;
                x = p;
            }
        }
        if (res) res[i] = r;
    }
    if (out)
        for (int64_t i = first + threadIdx.x; 2 * i + 1 < k; i += stride) {
            const int a = roots[2 * i], b = roots[2 * i + 1];
            out[i] = (uint8_t)(a >= 0 && a == b);
        }
}

// The same where every tree is known to have height at most one (after a full
// compression with no update since): a root is one gather away, nothing has to
// be repointed, and no frontier has to be kept, since Phase I has one level,
// or two where some S[i]'s root is not itself in S. Two launches that overlap
// their neighbours take the place of the cooperative kernel's launch, three
// barriers and two appends: 7.5 us against
// 21 us for 2^16 vertices, 22 against 65 us for 2^20.
// Counts are summed per CTA of a resident grid: with an atomic and two stores
// per warp on the same words, 2^20 vertices took 129 us instead of 22.
__global__ void __launch_bounds__(kBfBlock)
k_bulk_find_flat(const int* S, int64_t k, int n, const int* parent, int* mark, int epoch, int* roots,
                 BulkFindCounters* c, int* res, uint8_t* __restrict__ out, DevState* ds) {
    __shared__ unsigned part[kBfBlock / 32];
    pdl_trigger();
    pdl_wait();
    BulkFindCounters::Stats* st = &c->stats[epoch & 1];
    unsigned traversed = 0;
    bool any = false;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < k; i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + threadIdx.x;
        const int s = i < k ? S[i] : -1;
        const bool ok = in_range(s, n);
        if (i < k && !ok) flag(ds, ST_RANGE);
        const int r = ok ? parent[s] : -1;
        any |= ok;
        traversed += first_visit(ok, s, mark, epoch) && r != s;
        const int other = __shfl_down_sync(0xffffffffu, r, 1);
        if (i >= k) continue;
        roots[i] = r != s ? r : -1;  // what k_bulk_find_flat_levels has to look up
        if (res) res[i] = r;
        // S holds pairs: the even one of two lanes answers
        if (out && (i & 1) == 0) out[i >> 1] = (uint8_t)(r >= 0 && r == other);
    }
    traversed = __reduce_add_sync(0xffffffffu, traversed);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = traversed;
    any = __syncthreads_or(any);
    if (threadIdx.x == 0 && any) {
        unsigned long long t = 0;
        for (int w = 0; w < kBfBlock / 32; w++) t += part[w];
        if (t) atomicAdd(&st->traversed, t);
        st->levels = 1u;  // every writer writes the same
        st->depth = 1u;   // read only where something was traversed
    }
}

__global__ void __launch_bounds__(kBfBlock)
k_bulk_find_flat_levels(const int* roots, int64_t k, const int* mark, int epoch, BulkFindCounters* c) {
    pdl_trigger();
    pdl_wait();
    bool two = false;
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = first; i < k && !two; i += (int64_t)gridDim.x * blockDim.x) {
        const int r = roots[i];
        two = r >= 0 && mark[r] != epoch;
    }
    two = __syncthreads_or(two);
    if (threadIdx.x == 0 && two) c->stats[epoch & 1].levels = 2u;
    if (first == 0) c->stats[(epoch + 1) & 1] = {};
}

}  // namespace

// ---------------------------------------------------------------- driver

static cudaError_t grow(int** p, int64_t* cap, int64_t need) {
    if (need <= *cap) return cudaSuccess;
    int64_t c = *cap ? *cap : 1024;
    while (c < need) c *= 2;
    int* q = nullptr;
    cudaError_t e = cudaMalloc(&q, sizeof(int) * (size_t)c);
    if (e != cudaSuccess) return e;
    cudaFree(*p);
    *p = q;
    *cap = c;
    return cudaSuccess;
}

void bulk_find_free(BulkFindState& b) {
    cudaFree(b.mark);
    cudaFree(b.front[0]);
    cudaFree(b.front[1]);
    cudaFree(b.roots);
    cudaFree(b.res);
    cudaFree(b.count);
    b = BulkFindState{};
}

static cudaError_t launch(BulkFindState& b, int* parent, int n, const int* S, int64_t k, int* res,
                          uint8_t* out, DevState* ds, bool flat, bool pdl, cudaStream_t s) {
    // A graph would keep this call's stamp, and buffers that a larger call frees.
    if (capturing(s)) return cudaErrorStreamCaptureUnsupported;
    cudaError_t e = cudaSuccess;
    if (!b.mark) {
        BulkFindCounters* count = nullptr;
        int* mark = nullptr;
        e = cudaMalloc(&count, sizeof(BulkFindCounters));
        if (e == cudaSuccess) e = cudaMalloc(&mark, sizeof(int) * (size_t)n);
        if (e == cudaSuccess) e = cudaMemsetAsync(mark, 0, sizeof(int) * (size_t)n, s);
        if (e != cudaSuccess) {
            cudaFree(count);
            cudaFree(mark);
            return e;
        }
        b.mark = mark;
        b.count = count;
        b.epoch = 0;
        b.dirty = true;
    }
    if (b.dirty) {
        e = cudaMemsetAsync(b.count, 0, sizeof(BulkFindCounters), s);
        if (e != cudaSuccess) return e;
    }
    if (b.epoch >= 0x7ffffff0) {  // stamps would wrap: start over
        e = cudaMemsetAsync(b.mark, 0, sizeof(int) * (size_t)n, s);
        if (e == cudaSuccess) e = cudaMemsetAsync(b.count, 0, sizeof(BulkFindCounters), s);
        if (e != cudaSuccess) return e;
        b.epoch = 0;
    }
    if (k > b.cap_front) {  // cudaFree waits for the calls that use the old buffers
        int64_t c0 = b.cap_front, c1 = b.cap_front, c2 = b.cap_front;
        e = grow(&b.front[0], &c0, k);
        if (e == cudaSuccess) e = grow(&b.front[1], &c1, k);
        if (e == cudaSuccess) e = grow(&b.roots, &c2, k);
        if (e != cudaSuccess) return e;
        b.cap_front = c0;
    }
    int epoch = ++b.epoch;
    b.dirty = true;  // until everything is launched
    const int64_t need = (k + kBfBlock - 1) / kBfBlock;
    if (flat) {
        const int64_t cap = resident_grid<k_bulk_find_flat>(kBfBlock);
        const unsigned grid = (unsigned)std::min(cap, need);
        launch_windowed(k_bulk_find_flat, grid, kBfBlock, s, nullptr, pdl, S, k, n, (const int*)parent,
                        b.mark, epoch, b.roots, b.count, res, out, ds);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        launch_windowed(k_bulk_find_flat_levels, grid, kBfBlock, s, nullptr, pdl, (const int*)b.roots, k,
                        (const int*)b.mark, epoch, b.count);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        b.launches += 2;
    } else {
        const int64_t cap = resident_grid<k_bulk_find>(kBfBlock);
        void* args[] = {&S, &k, &n, &parent, &b.mark, &epoch, &b.front[0], &b.front[1], &b.roots,
                        &b.count, &res, &out, &ds};
        e = launch_fitting((unsigned)std::min(cap, need), [&](unsigned grid) {
            return cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(k_bulk_find), dim3(grid),
                                               dim3(kBfBlock), args, 0, s);
        });
        if (e != cudaSuccess) return e;
        b.launches += 1;
    }
    b.dirty = false;
    return cudaSuccess;
}

cudaError_t bulk_find(BulkFindState& b, int* parent, int n, const int* S, int64_t k, int* res,
                      DevState* ds, bool flat, bool pdl, cudaStream_t s) {
    return launch(b, parent, n, S, k, res, nullptr, ds, flat, pdl, s);
}

cudaError_t bulk_find_query(BulkFindState& b, int* parent, int n, const int* pairs, int64_t k,
                            uint8_t* out, DevState* ds, bool flat, bool pdl, cudaStream_t s) {
    return launch(b, parent, n, pairs, 2 * k, nullptr, out, ds, flat, pdl, s);
}

}  // namespace cc
