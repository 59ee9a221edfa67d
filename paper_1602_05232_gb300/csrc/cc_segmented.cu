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
// in lockstep; returns the links made. Both nodes of an edge are read in a round,
// their loads in flight together, and moved up, repointing the nodes passed at their
// grandparents, until the sides meet or the larger node is a root, which is linked
// under the other's parent at once: with the loads of all E edges before their
// links, more of these came too late (the 1024 graphs of seg_run_ring 591 -> 612 us).
// These walks are bound by latency, so moving up the larger node only, as the plain
// path does (join_edges), which reads less in more rounds, is slower: 612 us there,
// and 400 graphs of 32,768 vertices, 4 minibatches of 16,384 edges and pairs each, 256
// threads and two pairs each, 1047 us against 915.
template <int E>
__device__ __forceinline__ int sjoin(volatile unsigned short* sp, const int (&u)[E], const int (&v)[E],
                                     const int (&pu)[E], const int (&pv)[E]) {
    int hi[E], lo[E], bhi[E], blo[E];  // the nodes and those below them; a node itself where it was read as a root
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
            int p = hi[j] != bhi[j] ? sp[hi[j]] : hi[j];
            const int q = lo[j] != blo[j] ? sp[lo[j]] : lo[j];
            if (p == hi[j]) {
                p = atomicCAS(const_cast<unsigned short*>(sp) + hi[j], (unsigned short)hi[j], (unsigned short)q);
                if (p == hi[j]) {
                    made++;
                    hi[j] = lo[j];
                    continue;
                }
            }
            if (bhi[j] != hi[j]) sp[bhi[j]] = (unsigned short)p;
            if (blo[j] != lo[j] && q != lo[j]) sp[blo[j]] = (unsigned short)q;
            const int above = p == lo[j] ? q : p;  // the sides meet at lo: done
            const int bh = hi[j], bl = lo[j];
            const bool swap = above < q;
            hi[j] = swap ? q : above;
            bhi[j] = swap ? bl : bh;
            lo[j] = swap ? above : q;
            blo[j] = swap ? bh : bl;
            any |= hi[j] != lo[j];
        }
    }
    return made;
}

// Bit j: the ends of pair j, whose parents have been read, have the same root,
// in a forest that does not change meanwhile (a Bulk-Query between barriers).
// Nodes that meet have the same root, and a root above the other side's node is
// not that side's root, so the larger node is moved up. With one pair per thread
// the other one too, whose load is in flight with the first's; with more, the
// pairs' loads are in flight with each other, and reading less is faster (the 1024
// graphs of seg_run_ring: 1 %).
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
            const int p = sp[hi[j]], q = E == 1 ? sp[lo[j]] : lo[j];
            const bool meet = p == lo[j] || p == q;
            if (meet) same |= 1u << j;
            if (meet || p == hi[j]) act &= ~(1u << j);
            hi[j] = p < q ? q : p;
            lo[j] = p < q ? p : q;
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

// The pairs u, v of one thread, `count` of them, as part of an operation on the
// slice: joined, or answered into out. Returns the links made.
template <int E>
__device__ __forceinline__ int seg_chunk(unsigned short* sp, int ng, const int (&u)[E], const int (&v)[E], unsigned count,
                                         int kind, uint8_t* out, bool flat, bool& bad) {
    int pu[E], pv[E];
    unsigned in = 0;  // pairs that exist and are in range
#pragma unroll
    for (int j = 0; j < E; j++) {
        pu[j] = pv[j] = 0;
        if (j >= count) continue;
        if (in_range(u[j], ng) && in_range(v[j], ng)) {
            in |= 1u << j;
            pu[j] = sp[u[j]];
            pv[j] = sp[v[j]];
        } else {
            bad = true;
        }
    }
    if (kind == CC_OP_UPDATE) return sjoin<E>(sp, u, v, pu, pv);
    unsigned same = 0;
    if (flat) {
#pragma unroll
        for (int j = 0; j < E; j++) same |= (unsigned)(pu[j] == pv[j]) << j;
    } else {
        same = ssame<E>(sp, pu, pv);
    }
#pragma unroll
    for (int j = 0; j < E; j++)
        if (j < count) out[j] = (uint8_t)(((same & in) >> j) & 1u);
    return 0;
}

// The end of an operation of k pairs: a barrier, and the slice flattened once as
// many pairs as it has vertices have gone by since the last time and anything has
// been linked, if more operations follow. So the parents decide nearly all pairs,
// and all of a query while nothing more is linked.
__device__ __forceinline__ void seg_end_op(unsigned short* sp, int ng, unsigned k, bool more, int& linked, int& made,
                                           bool& flat, unsigned& since) {
    since = since + k < since ? 0xffffffffu : since + k;
    if (__syncthreads_or(linked)) flat = false;
    made += linked;
    linked = 0;
    if (!flat && since >= (unsigned)ng && more) {
        sflatten(sp, ng);
        __syncthreads();
        flat = true;
        since = 0;
    }
}

// The operations [ob, oe) of one graph in shared memory. An operation is cut
// into chunks of blockDim * E pairs (at least one), and a barrier separates
// consecutive operations. Bound by instruction issue and the latency between
// two barriers: a graph's operations are small (a few chunks, often one), so
// whatever a chunk waits for is waited for by all threads. So a warp without pairs
// in a chunk goes straight on to the barrier, the parents of all E pairs are read
// first, and only what they leave open is walked, in lockstep; and the next chunks'
// pairs, across operations (their data does not depend on results), are in flight:
// for one pair per thread the next chunk's, in registers (this function), for more
// those of `depth - 1` chunks (seg_run_ring). The ring's bookkeeping is worth it only
// where a chunk has more work: submits of 150 to 1000 graphs of 8192 to 60,000
// vertices with 4 minibatches of half as many edges and pairs, 512 threads, one pair
// each: 266-662 us with registers, 341-836 with the ring. Returns the links made.
template <int E>
__device__ __forceinline__ int seg_run_regs(unsigned short* sp, int ng, const SegOp* __restrict__ ops, int ob, int oe,
                                            DevState* ds) {
    const unsigned chunk = blockDim.x * E;
    const unsigned mine = threadIdx.x * E;
    int made = 0, linked = 0;
    bool bad = false, flat = false;
    unsigned since = 0, off = 0, k = 0;
    const int* data = nullptr;  // the current operation, field by field
    uint8_t* out = nullptr;
    int kind = 0, u[E] = {}, v[E] = {};
    if (ob < oe) {
        data = ops[ob].data; out = ops[ob].out; k = (unsigned)ops[ob].k; kind = ops[ob].kind;
        if (mine < k) load_pairs<E>(data, mine, k, pair_vec_dev(data), u, v);
    }
    for (int o = ob; o < oe;) {
        // where the next chunk is, and its loads
        int o2 = o, kind2 = kind;
        unsigned off2 = off + chunk, k2 = k;
        const int* data2 = data;
        uint8_t* out2 = out;
        if (off2 >= k) {
            o2 = o + 1;
            off2 = 0;
            if (o2 < oe) {
                data2 = ops[o2].data; out2 = ops[o2].out; k2 = (unsigned)ops[o2].k; kind2 = ops[o2].kind;
            }
        }
        int nu[E] = {}, nv[E] = {};
        if (o2 < oe && off2 + mine < k2) load_pairs<E>(data2, off2 + mine, k2, pair_vec_dev(data2), nu, nv);
        const unsigned i0 = off + mine;
        if (i0 < k) linked += seg_chunk<E>(sp, ng, u, v, k - i0, kind, out + i0, flat, bad);
        if (o2 != o) seg_end_op(sp, ng, k, o2 < oe, linked, made, flat, since);
#pragma unroll
        for (int j = 0; j < E; j++) {
            u[j] = nu[j];
            v[j] = nv[j];
        }
        o = o2; off = off2; data = data2; out = out2; k = k2; kind = kind2;
    }
    if (bad) flag(ds, ST_RANGE);
    return made;
}

// One operation as staged in shared memory, and how many are at a time (none for
// one pair per thread, which has no ring). A number the compiler knows: as an
// argument of the kernel it cost 2.5 % of the submit below.
template <int E>
constexpr int kStagedOps = E == 1 ? 0 : 64;
struct StagedOp {
    const int* data;
    uint8_t* out;
    unsigned k;
    int kind;
};

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

// The same with the operations' descriptors staged in shared memory, kStagedOps at a
// time, and each thread's pairs of the next `depth - 1` chunks in flight to its own
// slots of a ring there. 1024 uniform graphs of 2^8 to 2^16 vertices (4 edges per
// vertex, 36,000 operations), 1024 threads and 2 pairs each: the submit 690 -> 591 us
// with all of this. Flattening after every half as many pairs cost 1 %.
template <int E>
__device__ __forceinline__ int seg_run_ring(unsigned short* sp, int ng, int2* ring, int depth, StagedOp* staged,
                                            const SegOp* __restrict__ ops, int ob, int oe, DevState* ds) {
    const unsigned chunk = blockDim.x * E;
    const unsigned mine = threadIdx.x * E;
    int made = 0, linked = 0;
    bool bad = false, flat = false;
    unsigned since = 0;
    for (; ob < oe; ob += kStagedOps<E>) {
        const int count = oe - ob < kStagedOps<E> ? oe - ob : kStagedOps<E>;
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
            if (i0 < k) {
                int u[E], v[E];
#pragma unroll
                for (int j = 0; j < E; j++)
                    if (i0 + j < k) {
                        const int2 q = ring[(size_t)slot * chunk + mine + j];
                        u[j] = q.x;
                        v[j] = q.y;
                    }
                linked += seg_chunk<E>(sp, ng, u, v, k - i0, staged[o].kind, staged[o].out + i0, flat, bad);
            }
            slot = slot + 1 == depth ? 0 : slot + 1;
            off += chunk;
            if (off >= k) {
                off = 0;
                o++;
                seg_end_op(sp, ng, k, o < count || ob + count < oe, linked, made, flat, since);
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

// One pair per thread is held to 40 registers, with which three CTAs of 512
// threads fit on an SM (45 without the limit).
template <int E>
__global__ void __maxnreg__(E == 1 ? 40 : 64)
k_segmented(int* __restrict__ parent, const int64_t* __restrict__ seg_off, SegTables t,
            unsigned* __restrict__ queue, DevState* __restrict__ ds, int smem_cap, int depth) {
    extern __shared__ int4 seg_smem[];  // staged operations, ring of pairs (both empty for E = 1), slice
    StagedOp* staged = reinterpret_cast<StagedOp*>(seg_smem);
    int2* ring = reinterpret_cast<int2*>(staged + kStagedOps<E>);
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
            if constexpr (E == 1) made += seg_run_regs<E>(sp, ng, t.ops, ob, oe, ds);
            else made += seg_run_ring<E>(sp, ng, ring, depth, staged, t.ops, ob, oe, ds);
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
    const int staged = cfg.ept == 1 ? kStagedOps<1> : kStagedOps<2>;
    return sizeof(StagedOp) * staged + sizeof(int2) * (size_t)cfg.depth * cfg.block * cfg.ept +
           sizeof(unsigned short) * (size_t)cfg.smem_cap;
}

// The depth of the ring is the largest that costs no resident CTA, which pay more: a
// slice of 32,768 vertices leaves 11 KiB to each of three CTAs of an SM, and with a
// depth of 4 and 512 staged operations, which leave room for two, submits of graphs
// of 256 to 32,768 vertices at that cap took 1.1 to 1.5 times as long (256 threads,
// two pairs each). With one pair per thread there is no ring, and depth is 0.
template <int E>
static cudaError_t seg_depth(SegLaunch& cfg, int dev, int* ctas) {
    int most = 0;
    cudaFuncAttributes own;
    cudaError_t e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&own, k_segmented<E>);
    if (e != cudaSuccess) return e;
    const size_t room = (size_t)most - own.sharedSizeBytes;
    e = cudaFuncSetAttribute(k_segmented<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room);
    int best = E == 1 ? 0 : 2;
    *ctas = 0;
    for (int depth = best; depth <= (E == 1 ? 0 : 4) && e == cudaSuccess; depth++) {
        cfg.depth = depth;
        int per_sm = 0;
        if (seg_smem_bytes(cfg) <= room)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_segmented<E>, cfg.block, seg_smem_bytes(cfg));
        if (per_sm < *ctas) break;
        best = depth;
        *ctas = per_sm;
    }
    cfg.depth = best;
    return e;
}

template <int E>
static cudaError_t seg_prepare(SegLaunch& cfg) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    thread_local int of[3] = {-1, 0, 0}, depth, ctas;  // the last answer, and what it was for
    if (of[0] == dev && of[1] == cfg.block && of[2] == cfg.smem_cap) {
        cfg.depth = depth;
    } else {
        of[0] = -1;
        e = seg_depth<E>(cfg, dev, &ctas);
        if (e != cudaSuccess) return e;
        depth = cfg.depth;
        of[0] = dev;
        of[1] = cfg.block;
        of[2] = cfg.smem_cap;
    }
    if (ctas < 1) return cudaErrorInvalidConfiguration;
    cfg.grid = ctas * sms;
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
