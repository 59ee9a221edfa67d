"""Kernels at the sizes where their tiling, their remainders and their dispatch
rules change, against numpy and the CPU oracle."""
from __future__ import annotations

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05232_gb300 import _build, cc as ccmod
    _build.build_cc()
    ccmod.load()
    return ccmod


def dev(a, shift=0):
    """An int32 device copy whose address is 4 * shift bytes past a 16-byte boundary."""
    a = np.ascontiguousarray(a, dtype=np.int32)
    buf = torch.empty(a.size + 4, dtype=torch.int32, device="cuda")
    out = buf[shift:shift + a.size].view(a.shape)
    out.copy_(torch.from_numpy(a))
    return out


# ---------------------------------------------------------------- checkpoints

@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 5, 1023, 1025, 700_001, 3_000_000])
def test_validation_counts_roots_and_finds_each_fault(cc, n, shift):
    r = np.random.default_rng(n)
    first = r.integers(0, n, size=n)
    lab = np.minimum(first, np.arange(n))       # a label below v, or v itself
    lab = np.where(lab[lab] == lab, lab, np.arange(n)).astype(np.int32)
    assert (lab[lab] == lab).all()
    f = cc.Forest(n)
    f.load_labels(dev(lab, shift))
    assert f.components() == int((lab == np.arange(n)).sum())
    for at in (0, 1):                           # flat: copied; into any 4-byte-aligned place
        out = torch.full((n + 2,), -7, dtype=torch.int32, device="cuda")
        f.labels(out[at:at + n])
        assert np.array_equal(out[at:at + n].cpu().numpy(), lab) and int(out[n + at:].max()) == -7
    f.load_forest(dev(lab, shift))
    assert np.array_equal(f.labels().cpu().numpy(), lab)        # not known to be flat
    f.load_forest(dev(lab, shift))
    assert f.components() == int((lab == np.arange(n)).sum())
    for v in {0, n // 2, n - 1}:                # one id above its own place, or negative
        for x in (-1, v + 1):
            bad = lab.copy()
            bad[v] = x
            for load in (f.load_labels, f.load_forest):
                with pytest.raises(cc.CCError) as ex:
                    load(dev(bad, shift))
                assert ex.value.status == cc.CC_ERR_LABELS
    roots = np.flatnonzero(lab == np.arange(n))
    kids = np.flatnonzero(lab != np.arange(n))
    if len(kids) and len(roots) > 1:            # a chain of two: a forest, but no labelling
        chain = lab.copy()
        v = int(kids[-1])
        mid = int(kids[kids < v][-1]) if (kids < v).any() else -1
        if mid >= 0:
            chain[v] = mid
            with pytest.raises(cc.CCError):
                f.load_labels(dev(chain, shift))
            f.load_forest(dev(chain, shift))


# ------------------------------------------------------------------ Bulk-Find

def levels_up(par, S):
    """Phase I levels, as the frontiers of Algorithm 4 run."""
    seen, front, count = set(S), set(S), 0
    while front:
        count += 1
        front = {int(par[v]) for v in front if par[v] != v} - seen
        seen |= front
    return count


@pytest.mark.parametrize("k", [1, 31, 511, 512, 513, 4096, 1_500_001])
@pytest.mark.parametrize("shape", ["flat", "random", "chain"])
def test_bulk_find_at_block_and_grid_edges(cc, k, shape):
    import oracle
    n = 5000 if shape != "random" else 60_001
    r = np.random.default_rng(k)
    par = np.arange(n, dtype=np.int32)
    if shape == "flat":
        par[1:] = np.where(r.random(n - 1) < 0.5, 0, par[1:])
    elif shape == "chain":
        par[1:] = np.arange(n - 1)
        par[::700] = np.arange(0, n, 700)
    else:
        par[1:] = (r.random(n - 1) * np.arange(1, n)).astype(np.int32)
    S = r.integers(0, n, size=k).astype(np.int32)
    want_par, want_res, want_t = oracle.bulk_find(par, S)
    f = cc.Forest(n)
    for again in range(2):      # the counters and stamps of the first call must not show in the second
        if shape == "flat" and again:
            f.load_labels(dev(par))     # known to be flat: the kernels without frontiers
        else:
            f.load_forest(dev(par))
        Sd = dev(S, shift=1)
        res = f.bulk_find(Sd, Sd if again else None)    # the roots may replace S itself
        assert np.array_equal(res.cpu().numpy(), want_res)
        assert np.array_equal(f.parent().cpu().numpy(), want_par)
        t, up, down = f.bulk_find_stats()
        depth = np.zeros(n, dtype=np.int64)
        for v in range(1, n):
            depth[v] = 0 if par[v] == v else depth[par[v]] + 1
        assert t == want_t and up == levels_up(par, S.tolist())
        assert down == (int(depth[S].max()) + 1 if want_t else 0)
        if again:                       # the same through Bulk-Query: S as pairs
            f.set_option("bulk_find", 1)
            m = k - k % 2
            got = f.bulk_query(dev(S[:m], shift=1).view(-1, 2)).cpu().numpy()
            assert np.array_equal(got, (want_res[0:m:2] == want_res[1:m:2]).astype(np.uint8))
            f.set_option("bulk_find", 0)
    f.sync()
    S[0] = n                    # an id outside [0, n): no root, and reported
    got = f.bulk_find(dev(S)).cpu().numpy()
    assert got[0] == -1 and np.array_equal(got[1:], want_res[1:])
    with pytest.raises(cc.CCError) as ex:
        f.sync()
    assert ex.value.status == cc.CC_ERR_RANGE


# ----------------------------------------------------------------- Bulk-Query

def roots_of(par):
    r = par.copy()
    while not np.array_equal(r[r], r):
        r = r[r]
    return r


@pytest.mark.parametrize("shape", ["flat", "random", "chains", "singletons"])
@pytest.mark.parametrize("k", [1, 3, (1 << 17) - 1, 1 << 17, (1 << 17) + 5])
def test_query_walks_answer_as_the_roots_do(cc, k, shape):
    """Both sides of the size rule (two parents read at once, or the larger
    endpoint's first), every walk mode, on forests of several heights."""
    n = 100_003
    r = np.random.default_rng(k)
    par = np.arange(n, dtype=np.int32)
    if shape == "flat":
        par[1:] = np.where(r.random(n - 1) < 0.6, r.integers(0, 3, n - 1), par[1:])
        par[:3] = 0, 1, 2
    elif shape == "random":
        par[1:] = np.where(r.random(n - 1) < 0.9, (r.random(n - 1) * np.arange(1, n)).astype(np.int32), par[1:])
    elif shape == "chains":
        par[40:] = np.arange(n - 40)
    root = roots_of(par)
    q = r.integers(0, n, size=(k, 2)).astype(np.int32)
    q[::7, 1] = q[::7, 0]
    q[1::11, 1] = par[q[1::11, 0]]
    q[2::11, 1] = root[q[2::11, 0]]
    want = (root[q[:, 0]] == root[q[:, 1]]).astype(np.uint8)
    for mode in (0, 1, 2):
        for extra in ({}, {"query_pairs_per_thread": 1}, {"query_pairs_per_thread": 4, "query_variant": 1},
                      {"query_pairs_per_thread": 4, "block": 64}):
            f = cc.Forest(n, query_halving=mode, **extra)
            if shape == "flat":
                f.load_labels(dev(root))
            else:
                f.load_forest(dev(par))
            for shift in (0, 1):
                assert np.array_equal(f.bulk_query(dev(q, shift)).cpu().numpy(), want), (mode, extra)
            got = f.parent().cpu().numpy()      # the walks may only have skipped levels
            assert (got <= par).all() and np.array_equal(roots_of(got), root)
            f.sync()
            bad = q.copy()
            bad[-1] = n, 0
            got = f.bulk_query(dev(bad)).cpu().numpy()
            assert got[-1] == 0 and np.array_equal(got[:-1], want[:-1])
            with pytest.raises(cc.CCError):
                f.sync()


# ---------------------------------------------------------------- Bulk-Update

@pytest.mark.parametrize("ept", [1, 2, 4])
@pytest.mark.parametrize("k", [1, (1 << 18) - 1, 1 << 18, (1 << 18) + 127])
def test_update_on_both_sides_of_the_tile_rule(cc, k, ept):
    """Whole minibatches on a sparse, a dense and an already joined forest."""
    import oracle
    r = np.random.default_rng(k + ept)
    for n in (1000, 150_001, 2_000_003):
        ref = oracle.OracleUF(n)
        f = cc.Forest(n, edges_per_thread=ept)
        g = cc.Forest(n, edges_per_thread=ept, compress_every=0, hook=1)
        for step in range(3):
            e = r.integers(0, n, size=(k, 2)).astype(np.int32)
            e[::5] = np.sort(e[::5], axis=1)
            e[1::9, 0] = n // 2                     # a hub
            ref.bulk_update(e)
            for x in (f, g):
                x.bulk_update(dev(e, shift=step % 2))
                assert x.components() == ref.components
        for x in (f, g):
            assert np.array_equal(x.labels().cpu().numpy(), ref.labels())
            x.sync()
            bad = np.array([[0, n], [-1, 0], [0, 1]], dtype=np.int32).repeat(max(1, k // 3), axis=0)
            x.bulk_update(dev(bad))
            with pytest.raises(cc.CCError):
                x.sync()


@pytest.mark.parametrize("n", [1, 2, 5, 1023, 4096, 8191, 8192, 8193])
@pytest.mark.parametrize("k", [1, 2, 2047, 2049, 4096, 4097])
def test_small_update_equals_the_general_one(cc, n, k):
    """Both sides of the size rule, on an empty forest, on a deep one that was
    loaded and between larger minibatches, for every compression policy."""
    import oracle
    r = np.random.default_rng(n * 5000 + k)
    par = np.maximum(np.arange(n) - 1 - r.integers(0, 3, n), 0).astype(np.int32)
    par = np.where(r.random(n) < 0.3, np.arange(n), par).astype(np.int32)
    batches = [r.integers(0, n, size=(x, 2)).astype(np.int32) for x in (k, k, 6000, k)]
    batches[1][: k // 2] = batches[0][: k // 2]
    for opts in ({}, {"compress_every": 0}, {"compress_every": 2, "hook": 1}, {"compress_scope": 1}, {"pdl": 2}):
        f, g = cc.Forest(n, **opts), cc.Forest(n, **{**opts, "update_variant": 1})
        for start in ("empty", "loaded"):
            ref = oracle.OracleUF(n)
            if start == "loaded":
                for x in (f, g):
                    x.reset()
                    x.load_forest(dev(par))
                ref.bulk_update(np.stack([np.arange(n, dtype=np.int32), par], axis=1))
            for i, e in enumerate(batches):
                ref.bulk_update(e)
                q = dev(r.integers(0, n, size=(777, 2)).astype(np.int32))
                for x in (f, g):
                    x.bulk_update(dev(e, shift=i % 2))
                    assert x.components() == ref.components, (opts, start, i)
                    assert np.array_equal(x.bulk_query(q).cpu().numpy(), ref.bulk_query(q.cpu().numpy()))
            for x in (f, g):
                assert np.array_equal(x.labels().cpu().numpy(), ref.labels())
                x.sync()
    bad = np.array([[0, 0], [n, 0], [0, -1]], dtype=np.int32)[np.arange(min(k, 3))]
    f = cc.Forest(n)
    f.bulk_update(dev(bad))
    assert f.components() == n
    if len(bad) > 1:
        with pytest.raises(cc.CCError) as ex:
            f.sync()
        assert ex.value.status == cc.CC_ERR_RANGE


# --------------------------------------------------------------- batched form

@pytest.mark.parametrize("opts", [{}, {"seg_block": 1024, "seg_edges_per_thread": 2},
                                  {"seg_block": 64, "seg_edges_per_thread": 4},
                                  {"seg_block": 1024, "seg_edges_per_thread": 4},
                                  {"seg_block": 256, "seg_smem_cap": 3000}])
def test_batched_operations_of_all_lengths(cc, opts):
    """More operations than are staged at once, empty ones, lengths around the
    chunks of every launch shape, and data at 4, 8 and 16-byte alignment."""
    import oracle
    r = np.random.default_rng(7)
    sizes = [1, 2, 700, 3001, 65536]
    f = cc.Forest.segmented(sizes, **opts)
    refs = [oracle.OracleUF(n) for n in sizes]
    lengths = [0, 1, 2, 3, 63, 64, 65, 255, 256, 257, 1023, 1025, 2047, 2048, 2049, 4095, 4097, 0, 9000]
    ops, want, outs = [], [], []
    for step in range(2):
        for g, n in enumerate(sizes):
            # 1400 short operations on one graph: more than two stagings
            for i, k in enumerate([1] * 1400 if g == 2 and step else lengths * (2 if n > 2 else 1)):
                p = r.integers(0, n, size=(k, 2)).astype(np.int32)
                d = dev(p, shift=i % 4)
                if i % 2:
                    out = torch.full((k + 1,), 7, dtype=torch.uint8, device="cuda")
                    ops.append((g, cc.OP_QUERY, d, out[i % 3 == 0:][:k]))
                    want.append(refs[g].bulk_query(p))
                    outs.append(ops[-1][3])
                else:
                    ops.append((g, cc.OP_UPDATE, d, None))
                    refs[g].bulk_update(p)
        f.submit(ops if step else ops[:])
        f.sync()
        for got, exp in zip(outs, want):
            assert np.array_equal(got.cpu().numpy(), exp)
        ops, want, outs = [], [], []
        lab = f.labels().cpu().numpy()
        for g, ref in enumerate(refs):
            a, b = f.offsets[g], f.offsets[g + 1]
            assert np.array_equal(lab[a:b] - a, ref.labels())
    bad = [(4, cc.OP_UPDATE, dev([[0, 65536], [3, 4]]), None)]
    f.submit(bad)
    with pytest.raises(cc.CCError) as ex:
        f.sync()
    assert ex.value.status == cc.CC_ERR_RANGE


# ------------------------------------------------------- captured and replayed

@pytest.mark.parametrize("opts", [{}, {"pdl": 2, "compress_every": 2, "big_filter": 100, "edge_order": 6},
                                  {"pdl": 0, "compress_every": 0, "query_halving": 1}])
@pytest.mark.parametrize("n,k", [(3000, 1000), (200_000, 300_000)])
def test_a_captured_pass_replays_on_new_inputs(cc, opts, n, k):
    """The dependent launches, the small update and the tiles inside a CUDA
    graph, replayed after the inputs have changed."""
    import oracle
    r = np.random.default_rng(n)
    st = torch.cuda.Stream()
    edges = [torch.empty((k, 2), dtype=torch.int32, device="cuda") for _ in range(3)]
    pairs = torch.empty((5000, 2), dtype=torch.int32, device="cuda")
    out = torch.empty((3, 5000), dtype=torch.uint8, device="cuda")
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    f = cc.Forest(n, stream=st, **opts)

    def fill():
        for e in edges:
            e.copy_(torch.from_numpy(r.integers(0, n, size=(k, 2)).astype(np.int32)))
        pairs.copy_(torch.from_numpy(r.integers(0, n, size=(5000, 2)).astype(np.int32)))
        torch.cuda.synchronize()

    def one_pass():
        f.reset()
        for e, o in zip(edges, out):
            f.bulk_update(e)
            f.bulk_query(pairs, o)
        f.labels(labels)

    fill()
    one_pass()                              # scratch of the first calls
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        one_pass()
    for _ in range(2):
        fill()
        g.replay()
        torch.cuda.synchronize()
        ref = oracle.OracleUF(n)
        q = pairs.cpu().numpy()
        for e, o in zip(edges, out):
            ref.bulk_update(e.cpu().numpy())
            assert np.array_equal(o.cpu().numpy(), ref.bulk_query(q))
        assert np.array_equal(labels.cpu().numpy(), ref.labels())
        f.sync()


@pytest.mark.parametrize("recorded", ["update", "labels"])
@pytest.mark.parametrize("n,k", [(3000, 1000), (200_000, 60_000)])
def test_labels_and_bulk_find_do_not_trust_a_forest_that_a_graph_changes(cc, recorded, n, k):
    """A replayed update changes a forest that the handle last saw compressed,
    and recorded labels run on a forest that was updated since: neither may
    take the copy of, or the short Bulk-Find on, a flat forest."""
    import oracle
    r = np.random.default_rng(n + k)
    st = torch.cuda.Stream()
    e = torch.empty((k, 2), dtype=torch.int32, device="cuda")
    labels = torch.empty(n, dtype=torch.int32, device="cuda")
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    found = torch.empty_like(ids)
    f = cc.Forest(n, stream=st, compress_every=0, update_variant=1)
    ref = oracle.OracleUF(n)

    def fill():
        # a path through the ids in steps of random length: deep trees
        x = np.sort(r.choice(n, size=k + 1, replace=False)).astype(np.int32)
        p = np.stack([x[1:], x[:-1]], axis=1)
        e.copy_(torch.from_numpy(p))
        torch.cuda.synchronize()
        ref.bulk_update(p)

    def check():
        torch.cuda.synchronize()
        assert np.array_equal(labels.cpu().numpy(), ref.labels())

    fill()
    f.bulk_update(e)
    f.labels(labels)        # flat from here, as the handle sees it
    f.bulk_find(ids, found)
    check()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        f.bulk_update(e) if recorded == "update" else f.labels(labels)
    for _ in range(3):
        fill()
        if recorded == "update":
            g.replay()
            torch.cuda.synchronize()
            f.bulk_find(ids, found)
            torch.cuda.synchronize()
            assert np.array_equal(found.cpu().numpy(), ref.labels())
            fill()
            g.replay()
            torch.cuda.synchronize()
            f.labels(labels)
        else:
            f.bulk_update(e)
            torch.cuda.synchronize()
            g.replay()
        check()
    f.sync()


def test_bulk_find_is_refused_under_capture(cc):
    """Its scratch may be freed by a later, larger call, and its stamp is the call's."""
    st = torch.cuda.Stream()
    f = cc.Forest(5000, stream=st)
    ids = torch.arange(5000, dtype=torch.int32, device="cuda")
    e = torch.tensor([[1, 2], [2, 3]], dtype=torch.int32, device="cuda")
    found = torch.empty_like(ids)
    out = torch.empty(2, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    f.bulk_find(ids, found)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        with pytest.raises(cc.CCError) as ex:
            f.bulk_find(ids, found)
        assert ex.value.status == cc.CC_ERR_CUDA
        f.bulk_update(e)
        f.bulk_query(e, out)
    g.replay()
    torch.cuda.synchronize()
    assert out.tolist() == [1, 1] and f.components() == 4998
    f.bulk_find(ids[:4], found[:4])
    torch.cuda.synchronize()
    assert found[:4].tolist() == [0, 1, 1, 1]
