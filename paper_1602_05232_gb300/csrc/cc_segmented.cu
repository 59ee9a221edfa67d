// Batched form: many independent graphs, each with its own ordered list of
// Bulk-Update / Bulk-Query minibatches of any size (Section 1: minibatches
// need not be equal), all executed by ONE persistent kernel.
//
// Every graph g owns the slice parent[seg_off[g] .. seg_off[g+1]) of one
// forest, with its own local ids. A CTA claims a whole graph from a work
// queue (largest work first) and runs that graph's operations in list order,
// separated by __syncthreads(), so each bulk operation completes before the
// next one starts. A graph of at most `smem_cap` vertices is worked on in
// shared memory: its slice is loaded as 16-bit local ids (up to 65,536
// vertices = 128 KiB), finds and hooks use shared-memory atomics, and the
// slice is written back flattened (every vertex pointing at its root). Larger
// graphs are worked on in place in global memory with the plain path's
// find/hook. The work queue counter is the only scratch and is reset before
// every launch.
#include <cstdint>

#include "cc_device.cuh"
#include "cc_internal.cuh"

namespace cc {

namespace {

// --- shared-memory forest primitives (same invariant: sp[x] <= x) ---------

__device__ __forceinline__ int sroot(const volatile unsigned short* sp, int x) {
    int p = sp[x];
    while (p < x) {
        x = p;
        p = sp[x];
    }
    return x;
}

// Joins the ends of E edges whose parents have been read (equal ones are done),
// in lockstep; returns the links made. The larger of an edge's two nodes is
// moved up, repointing the nodes passed at their grandparents, until the sides
// meet or it is a root, which is linked under the other node (join_edges of the
// plain path, in shared memory, where a store costs no more than an atomic).
template <int E>
__device__ __forceinline__ int sjoin(volatile unsigned short* sp, const int (&u)[E], const int (&v)[E],
                                     const int (&pu)[E], const int (&pv)[E]) {
    int hi[E], lo[E], bhi[E], blo[E];  // the nodes and those below them; a node itself where it is a root endpoint
    bool any = false;
#pragma unroll
    for (int j = 0; j < E; j++) {
        const bool s = pu[j] < pv[j];
        hi[j] = s ? pv[j] : pu[j];
        lo[j] = s ? pu[j] : pv[j];
        bhi[j] = s ? v[j] : u[j];
        blo[j] = s ? u[j] : v[j];
        any |= hi[j] != lo[j];
    }
    int made = 0;
    while (any) {
        any = false;
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (hi[j] == lo[j]) continue;
            int p = hi[j] == bhi[j] ? hi[j] : sp[hi[j]];
            if (p == hi[j])
                p = atomicCAS(const_cast<unsigned short*>(sp) + hi[j], (unsigned short)hi[j], (unsigned short)lo[j]);
            if (p == hi[j]) {
                made++;
                hi[j] = lo[j];
                continue;
            }
            if (bhi[j] != hi[j]) sp[bhi[j]] = (unsigned short)p;
            const int below = hi[j];
            const bool swap = p < lo[j];
            hi[j] = swap ? lo[j] : p;
            bhi[j] = swap ? blo[j] : below;
            lo[j] = swap ? p : lo[j];
            blo[j] = swap ? below : blo[j];
            any |= hi[j] != lo[j];
        }
    }
    return made;
}

// Bit j: the ends of pair j, whose parents have been read, have the same root,
// in a forest that does not change meanwhile (a Bulk-Query between barriers).
// Only the larger node of a pair is moved up: a root above the other side's
// node is not that side's root, and nodes that meet are.
template <int E>
__device__ __forceinline__ unsigned ssame(const unsigned short* sp, const int (&pu)[E], const int (&pv)[E]) {
    int hi[E], lo[E];
    unsigned same = 0, act = 0;
#pragma unroll
    for (int j = 0; j < E; j++) {
        hi[j] = pu[j] < pv[j] ? pv[j] : pu[j];
        lo[j] = pu[j] < pv[j] ? pu[j] : pv[j];
        if (hi[j] == lo[j]) same |= 1u << j;
        else act |= 1u << j;
    }
    while (act) {
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (!((act >> j) & 1u)) continue;
            const int p = sp[hi[j]];
            if (p == lo[j]) same |= 1u << j;
            if (p == lo[j] || p == hi[j]) act &= ~(1u << j);
            hi[j] = p < lo[j] ? lo[j] : p;
            lo[j] = p < lo[j] ? p : lo[j];
        }
    }
    return same;
}

// Points every vertex of the slice at its root, four vertices per thread and
// step. No other writes than these go on; all threads of the CTA take part.
__device__ __forceinline__ void sflatten(unsigned short* sp, int ng) {
    for (int v0 = threadIdx.x * 4; v0 < ng; v0 += blockDim.x * 4) {
        if (v0 + 4 <= ng) {
            const ushort4 q = *reinterpret_cast<const ushort4*>(sp + v0);
            const ushort4 g = make_ushort4(sp[q.x], sp[q.y], sp[q.z], sp[q.w]);
            if (g.x == q.x && g.y == q.y && g.z == q.z && g.w == q.w) continue;
            *reinterpret_cast<ushort4*>(sp + v0) =
                make_ushort4((unsigned short)sroot(sp, g.x), (unsigned short)sroot(sp, g.y),
                             (unsigned short)sroot(sp, g.z), (unsigned short)sroot(sp, g.w));
        } else {
            for (int v = v0; v < ng; v++) sp[v] = (unsigned short)sroot(sp, v);
        }
    }
}

// One operation as staged in shared memory, and how many are staged at a time.
struct StagedOp {
    const int* data;
    uint8_t* out;
    unsigned k;
    int kind;
};
constexpr int kStagedOps = 512;

// Asynchronous copies global -> shared, each thread's own: a thread waits only
// for its own groups, so the ring needs no barrier.
__device__ __forceinline__ void async_copy(void* dst, const int* src, int bytes) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (bytes == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
    else if (bytes == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// All but the newest `left` groups of this thread are complete (left in 1..3).
__device__ __forceinline__ void async_wait(int left) {
    if (left == 3) asm volatile("cp.async.wait_group 3;\n" ::: "memory");
    else if (left == 2) asm volatile("cp.async.wait_group 2;\n" ::: "memory");
    else asm volatile("cp.async.wait_group 1;\n" ::: "memory");
}

// The operations [ob, oe) of one graph in shared memory. An operation is cut
// into chunks of blockDim * E pairs (at least one), and a barrier separates
// consecutive operations. Bound by instruction issue and the latency between
// two barriers: a graph's operations are small (a few chunks, often one), so
// whatever a chunk waits for is waited for by all threads. So
//  - the operations' descriptors are staged in shared memory, and each thread's
//    pairs of the next `depth - 1` chunks, across operations (their data does not
//    depend on results), are in flight to its own slots of a ring there;
//  - a warp without pairs in a chunk goes straight on to the barrier;
//  - the parents of all E pairs are read first, and only what they leave open is
//    walked, in lockstep;
//  - after an operation the slice is flattened, once as many pairs as it has
//    vertices have gone by since the last time and anything has been linked, so
//    that the parents decide nearly all pairs, and all of a query while nothing
//    more is linked.
// 1024 uniform graphs of 2^8 to 2^16 vertices (4 edges per vertex, 36,000
// operations): 713 -> 640 us with 1024 threads and 2 pairs each, 1011 -> 904 with
// 512 and 1, 838 -> 755 with 1024 and 4. Of this, the ring and the staging alone
// were worth 2 %, with the skip 8 %, the flattening 2 % more. Flattening after every
// half as many pairs cost 1 %. Returns the number of links made.
template <int E>
__device__ __forceinline__ int seg_run_smem(unsigned short* sp, int ng, int2* ring, int depth, StagedOp* staged,
                                            const SegOp* __restrict__ ops, int ob, int oe, DevState* ds) {
    const unsigned chunk = blockDim.x * E;
    const unsigned mine = threadIdx.x * E;
    int made = 0, linked = 0;
    bool bad = false, flat = false;
    unsigned since = 0;
    for (; ob < oe; ob += kStagedOps) {
        const int count = oe - ob < kStagedOps ? oe - ob : kStagedOps;
        for (int i = threadIdx.x; i < count; i += blockDim.x)
            staged[i] = {ops[ob + i].data, ops[ob + i].out, (unsigned)ops[ob + i].k, ops[ob + i].kind};
        __syncthreads();
        // the next chunk to be fetched: of operation f, from pair foff on, into ring slot fs
        int f = 0, fs = 0;
        unsigned foff = 0;
        auto fetch = [&] {
            if (f < count) {
                const int* data = staged[f].data;
                const unsigned k = staged[f].k, i0 = foff + mine;
                if (i0 < k) {
                    const int* src = data + 2 * (size_t)i0;
                    int2* dst = ring + (size_t)fs * chunk + mine;
                    const int vec = pair_vec_dev(src);
                    if (E % 2 == 0 && vec == 2 && i0 + E <= k) {
#pragma unroll
                        for (int j = 0; j < E / 2; j++) async_copy(dst + 2 * j, src + 4 * j, 16);
                    } else {
#pragma unroll
                        for (int j = 0; j < E; j++)
                            if (i0 + j < k) {
                                if (vec) {
                                    async_copy(dst + j, src + 2 * j, 8);
                                } else {
                                    async_copy(&dst[j].x, src + 2 * j, 4);
                                    async_copy(&dst[j].y, src + 2 * j + 1, 4);
                                }
                            }
                    }
                }
                foff += chunk;
                if (foff >= k) {
                    foff = 0;
                    f++;
                }
            }
            async_commit();
            fs = fs + 1 == depth ? 0 : fs + 1;
        };
        for (int i = 1; i < depth; i++) fetch();
        int o = 0, slot = 0;
        unsigned off = 0;
        while (o < count) {
            fetch();
            async_wait(depth - 1);
            const unsigned k = staged[o].k, i0 = off + mine;
            if (i0 < k) {  // a warp without pairs goes on to the barrier
                int u[E], v[E], pu[E], pv[E];
                unsigned in = 0;  // pairs that exist and are in range
#pragma unroll
                for (int j = 0; j < E; j++) {
                    pu[j] = pv[j] = 0;
                    if (i0 + j >= k) continue;
                    const int2 q = ring[(size_t)slot * chunk + mine + j];
                    u[j] = q.x;
                    v[j] = q.y;
                    if (in_range(u[j], ng) && in_range(v[j], ng)) {
                        in |= 1u << j;
                        pu[j] = sp[u[j]];
                        pv[j] = sp[v[j]];
                    } else {
                        bad = true;
                    }
                }
                if (staged[o].kind == CC_OP_UPDATE) {
                    linked += sjoin<E>(sp, u, v, pu, pv);
                } else {
                    uint8_t* out = staged[o].out;
                    unsigned same = 0;
                    if (flat) {
#pragma unroll
                        for (int j = 0; j < E; j++) same |= (unsigned)(pu[j] == pv[j]) << j;
                    } else {
                        same = ssame<E>(sp, pu, pv);
                    }
#pragma unroll
                    for (int j = 0; j < E; j++)
                        if (i0 + j < k) out[i0 + j] = (uint8_t)(((same & in) >> j) & 1u);
                }
            }
            slot = slot + 1 == depth ? 0 : slot + 1;
            off += chunk;
            if (off >= k) {
                off = 0;
                o++;
                since = since + k < since ? 0xffffffffu : since + k;
                if (__syncthreads_or(linked)) flat = false;
                made += linked;
                linked = 0;
                if (!flat && since >= (unsigned)ng) {
                    sflatten(sp, ng);
                    __syncthreads();
                    flat = true;
                    since = 0;
                }
            }
        }
    }
    if (bad) flag(ds, ST_RANGE);
    return made;
}

// --- the same operations in place on the global forest (large graphs) ----

template <int E>
__device__ __forceinline__ int seg_update_global(int* parent, int64_t base, int ng,
                                                 const SegOp& op, DevState* ds) {
    const int vec = pair_vec_dev(op.data);
    int made = 0;
    bool bad = false;
    for (int64_t i = (int64_t)threadIdx.x * E; i < op.k; i += (int64_t)blockDim.x * E) {
        int u[E], v[E];
        load_pairs<E>(op.data, i, op.k, vec, u, v);
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (i + j >= op.k) break;
            if (!(in_range(u[j], ng) && in_range(v[j], ng))) {
                bad = true;
                continue;
            }
            const int gu = (int)(base + u[j]), gv = (int)(base + v[j]);
            made += hook(parent, find_halving(parent, gu, ds), find_halving(parent, gv, ds), ds);
        }
    }
    if (bad) flag(ds, ST_RANGE);
    return made;
}

template <int E>
__device__ __forceinline__ void seg_query_global(int* parent, int64_t base, int ng,
                                                 const SegOp& op, DevState* ds) {
    const int vec = pair_vec_dev(op.data);
    bool bad = false;
    for (int64_t i = (int64_t)threadIdx.x * E; i < op.k; i += (int64_t)blockDim.x * E) {
        int u[E], v[E];
        load_pairs<E>(op.data, i, op.k, vec, u, v);
#pragma unroll
        for (int j = 0; j < E; j++) {
            if (i + j >= op.k) break;
            uint8_t a = 0;
            if (in_range(u[j], ng) && in_range(v[j], ng)) {
                const int gu = (int)(base + u[j]), gv = (int)(base + v[j]);
                a = (uint8_t)(walk_root(parent, gu, parent[gu]) == walk_root(parent, gv, parent[gv]));
            } else {
                bad = true;
            }
            op.out[i + j] = a;
        }
    }
    if (bad) flag(ds, ST_RANGE);
}

}  // namespace

template <int E>
__global__ void __launch_bounds__(1024, 1)
k_segmented(int* __restrict__ parent, const int64_t* __restrict__ seg_off, SegTables t,
            unsigned* __restrict__ queue, DevState* __restrict__ ds, int smem_cap, int depth) {
    extern __shared__ int4 seg_smem[];  // staged operations, ring of pairs, slice (seg_smem_bytes)
    StagedOp* staged = reinterpret_cast<StagedOp*>(seg_smem);
    int2* ring = reinterpret_cast<int2*>(staged + kStagedOps);
    unsigned short* sp = reinterpret_cast<unsigned short*>(ring + (size_t)depth * blockDim.x * E);
    __shared__ int s_idx;
    int made = 0;
    const int nactive = *t.nactive;
    for (;;) {
        if (threadIdx.x == 0) s_idx = (int)atomicAdd(queue, 1u);
        __syncthreads();
        const int idx = s_idx;
        __syncthreads();  // all have read s_idx before thread 0 may overwrite it
        if (idx >= nactive) break;
        const int g = t.order[idx];
        const int64_t base = seg_off[g];
        const int ng = (int)(seg_off[g + 1] - base);
        const int ob = t.op_begin[g], oe = t.op_begin[g + 1];
        if (ng <= smem_cap) {
            // four loads in flight per thread, then the tail one at a time
            int v = threadIdx.x;
            for (; v + 3 * (int)blockDim.x < ng; v += 4 * blockDim.x) {
                int pv[4];
#pragma unroll
                for (int j = 0; j < 4; j++) pv[j] = __ldcs(parent + base + v + j * blockDim.x);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const int w = v + j * blockDim.x;
                    int64_t l = (int64_t)pv[j] - base;
                    if (l < 0 || l > w) {  // not a forest of this slice: keep w alone
                        flag(ds, ST_CORRUPT);
                        l = w;
                    }
                    sp[w] = (unsigned short)l;
                }
            }
            for (; v < ng; v += blockDim.x) {
                const int64_t pv = (int64_t)parent[base + v] - base;
                if (pv < 0 || pv > v) {  // not a forest of this slice: keep v alone
                    flag(ds, ST_CORRUPT);
                    sp[v] = (unsigned short)v;
                } else {
                    sp[v] = (unsigned short)pv;
                }
            }
            __syncthreads();
            made += seg_run_smem<E>(sp, ng, ring, depth, staged, t.ops, ob, oe, ds);
            for (int v = threadIdx.x; v < ng; v += blockDim.x)
                parent[base + v] = (int)(base + sroot(sp, v));
            __syncthreads();  // the slice is out before the buffer is reused
        } else {
            for (int o = ob; o < oe; o++) {
                const SegOp op = t.ops[o];
                if (op.kind == CC_OP_UPDATE) made += seg_update_global<E>(parent, base, ng, op, ds);
                else seg_query_global<E>(parent, base, ng, op, ds);
                __syncthreads();
            }
        }
    }
    made = __reduce_add_sync(0xffffffffu, made);
    if ((threadIdx.x & 31) == 0 && made) atomicAdd(&ds->unions, (unsigned long long)made);
}

static size_t seg_smem_bytes(const SegLaunch& cfg) {
    if (cfg.smem_cap == 0) return 0;  // no graph is worked on in shared memory
    return sizeof(StagedOp) * kStagedOps + sizeof(int2) * (size_t)cfg.depth * cfg.block * cfg.ept +
           sizeof(unsigned short) * (size_t)cfg.smem_cap;
}

template <int E>
static cudaError_t seg_prepare(SegLaunch& cfg) {
    int per_sm = 0, dev = 0, sms = 0, most = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    // three chunks ahead, fewer where the ring would not fit beside the largest slice
    for (cfg.depth = 4; cfg.depth > 2 && seg_smem_bytes(cfg) > (size_t)most; cfg.depth--) {
    }
    const size_t smem = seg_smem_bytes(cfg);
    e = cudaFuncSetAttribute(k_segmented<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_segmented<E>, cfg.block, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cfg.grid = per_sm * sms;
    if (cfg.max_ctas > 0 && cfg.grid > cfg.max_ctas) cfg.grid = cfg.max_ctas;
    return cudaSuccess;
}

cudaError_t prepare_segmented(SegLaunch& cfg) {
    switch (cfg.ept) {
        case 1: return seg_prepare<1>(cfg);
        case 2: return seg_prepare<2>(cfg);
        default: return seg_prepare<4>(cfg);
    }
}

cudaError_t launch_segmented(int* parent, const int64_t* seg_off, const SegTables& t,
                             unsigned* queue, DevState* ds, const SegLaunch& cfg, cudaStream_t s) {
    if (cfg.grid < 1) return cudaErrorInvalidConfiguration;
    const size_t smem = seg_smem_bytes(cfg);
    switch (cfg.ept) {
        case 1: k_segmented<1><<<cfg.grid, cfg.block, smem, s>>>(parent, seg_off, t, queue, ds, cfg.smem_cap, cfg.depth); break;
        case 2: k_segmented<2><<<cfg.grid, cfg.block, smem, s>>>(parent, seg_off, t, queue, ds, cfg.smem_cap, cfg.depth); break;
        default: k_segmented<4><<<cfg.grid, cfg.block, smem, s>>>(parent, seg_off, t, queue, ds, cfg.smem_cap, cfg.depth); break;
    }
    return cudaGetLastError();
}

}  // namespace cc
