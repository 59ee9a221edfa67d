"""What a handle may know about a forest that CUDA graphs read and change:
work that is only recorded has not run, and a graph may be replayed at any time."""
from __future__ import annotations

import contextlib
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

M = 1000                # groups of four vertices
N = 4 * M


@pytest.fixture(scope="module")
def cc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1602_05232_gb300 import _build, cc as ccmod
    _build.build_cc()
    ccmod.load()
    return ccmod


def groups(*ij):
    """The pairs (4g + i, 4g + j) of every group g, on the device."""
    base = 4 * np.arange(M)[:, None, None] + np.array(ij)[None]
    return torch.from_numpy(base.reshape(-1, 2).astype(np.int32)).cuda()


def deepen(f, e):
    """Joins each group by two updates that leave vertex 3 two links below its root."""
    f.bulk_update(e[0])
    f.bulk_update(e[1])


def edges():
    return groups((0, 1), (2, 3)), groups((1, 3))


def all_pairs():
    return groups((0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3))


ROOTS = np.repeat(4 * np.arange(M), 4)


def record(st, fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        fn()
    return g


def test_query_after_the_replay_of_an_update(cc):
    """The forest was reset, then a graph made it deep."""
    st = torch.cuda.Stream()
    e, q = edges(), all_pairs()
    out = torch.zeros(q.shape[0], dtype=torch.uint8, device="cuda")
    f = cc.Forest(N, stream=st, compress_every=0, update_variant=1)
    torch.cuda.synchronize()
    g = record(st, lambda: deepen(f, e))
    f.reset()
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    f.bulk_query(q, out)
    torch.cuda.synchronize()
    assert out.all()


@pytest.mark.parametrize("link", [0, 1])
def test_recorded_query_on_a_forest_that_is_deep_by_then(cc, link):
    """A query recorded while the forest was flat, replayed after updates."""
    st = torch.cuda.Stream()
    e, q = edges(), all_pairs()
    out = torch.zeros(q.shape[0], dtype=torch.uint8, device="cuda")
    f = cc.Forest(N, stream=st, compress_every=0, update_variant=1, link=link, update_schedule=link)
    torch.cuda.synchronize()
    f.compress()
    g = record(st, lambda: f.bulk_query(q, out))
    deepen(f, e)
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()
    assert out.all()


RECORDED = {
    "labels": lambda f, e: f.labels(),
    "compress": lambda f, e: f.compress(),
    "reset": lambda f, e: f.reset(),
    "small update": lambda f, e: f.bulk_update(e[0]),
    "compressing update": lambda f, e: f.bulk_update(e[0]),
    "update, then compress": lambda f, e: (deepen(f, e), f.compress()),
}


@pytest.mark.parametrize("ask", ["labels", "find", "query"])
@pytest.mark.parametrize("recorded", RECORDED)
def test_recorded_work_has_not_flattened_anything(cc, recorded, ask):
    """A deep forest, work that flattens it recorded but not run, then a call."""
    st = torch.cuda.Stream()
    e, q = edges(), all_pairs()
    out = torch.zeros(q.shape[0], dtype=torch.uint8, device="cuda")
    ids = torch.arange(N, dtype=torch.int32, device="cuda")
    f = cc.Forest(N, stream=st, compress_every=0, update_variant=1)

    def check():
        torch.cuda.synchronize()
        if ask == "query":
            out.zero_()
            torch.cuda.synchronize()
            f.bulk_query(q, out)
            torch.cuda.synchronize()
            assert out.all()
        else:
            got = f.labels() if ask == "labels" else f.bulk_find(ids)
            torch.cuda.synchronize()
            assert np.array_equal(got.cpu().numpy(), ROOTS)

    torch.cuda.synchronize()
    deepen(f, e)
    assert f.depth()[0] == 2
    f.set_option("update_variant", 0 if recorded == "small update" else 1)
    f.set_option("compress_every", int(recorded == "compressing update"))
    g = record(st, lambda: RECORDED[recorded](f, e))
    check()
    f.reset()
    f.set_option("update_variant", 1)
    f.set_option("compress_every", 0)
    if recorded != "reset":
        deepen(f, e)
        torch.cuda.synchronize()
        g.replay()
        check()


def test_recorded_calls_see_what_was_recorded_before_them(cc):
    """Within one capture: flat after the compression, not before and not after
    the next update, whatever the forest is when the graph is replayed."""
    st = torch.cuda.Stream()
    e, q = edges(), all_pairs()
    outs = torch.zeros((3, q.shape[0]), dtype=torch.uint8, device="cuda")
    labels = torch.empty((2, N), dtype=torch.int32, device="cuda")
    f = cc.Forest(N, stream=st, compress_every=0, update_variant=1)
    torch.cuda.synchronize()

    def step():
        f.bulk_query(q, outs[0])
        f.compress()
        f.bulk_query(q, outs[1])
        f.labels(labels[0])
        f.reset()
        deepen(f, e)
        f.bulk_query(q, outs[2])
        f.labels(labels[1])

    g = record(st, step)
    for _ in range(2):
        deepen(f, e)
        outs.zero_()
        labels.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert outs.all()
        assert np.array_equal(labels.cpu().numpy(), np.stack([ROOTS, ROOTS]))


@contextlib.contextmanager
def foreign_capture():
    """While a stream that the legacy stream synchronises with is captured, which
    work given to the legacy stream is refused by and ends."""
    try:
        rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    except OSError:
        pytest.skip("no CUDA runtime library to create a blocking stream with")
    st, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(st)) == 0
    assert rt.cudaStreamBeginCapture(st, 0) == 0
    try:
        yield
    finally:
        rt.cudaStreamEndCapture(st, ctypes.byref(graph))
        rt.cudaGetLastError()
        assert rt.cudaStreamDestroy(st) == 0


def test_a_refused_call_does_not_fail_the_next(cc):
    f = cc.Forest(N, stream=0)
    labels = torch.zeros(N, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    with foreign_capture():
        with pytest.raises(cc.CCError) as ex:
            f.load_labels(labels)
        assert ex.value.status == cc.CC_ERR_CUDA
    f.compress()
    assert f.components() == N


def test_another_streams_capture_is_not_this_forests(cc):
    """Nothing was recorded, so once the forest is compressed the two-kernel
    Bulk-Find for flat forests is back."""
    e = edges()[0]
    ids = torch.arange(N, dtype=torch.int32, device="cuda")
    f = cc.Forest(N, stream=0)
    f.submit([(0, cc.OP_UPDATE, e, None)])
    f.sync()
    with foreign_capture():
        with pytest.raises(cc.CCError):
            f.submit([(0, cc.OP_UPDATE, e, None)])
    f.compress()
    before = f.kernel_stats()["query"]
    found = f.bulk_find(ids)
    torch.cuda.synchronize()
    assert f.kernel_stats()["query"] - before == 2
    assert np.array_equal(found.cpu().numpy(), np.arange(N) // 2 * 2)


def test_statistics_asked_for_during_a_capture(cc):
    """They are on the device, where a capture cannot wait for them; it is not ended."""
    st = torch.cuda.Stream()
    e, q = edges(), all_pairs()
    out = torch.zeros(q.shape[0], dtype=torch.uint8, device="cuda")
    f = cc.Forest(N, stream=st)
    torch.cuda.synchronize()
    f.bulk_find(q.view(-1))
    stats = f.bulk_find_stats()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        deepen(f, e)
        with pytest.raises(cc.CCError) as ex:
            f.bulk_find_stats()
        assert ex.value.status == cc.CC_ERR_CUDA
        f.bulk_query(q, out)
    g.replay()
    torch.cuda.synchronize()
    assert out.all() and f.bulk_find_stats() == stats


@pytest.mark.parametrize("updates", [1, 2, 3])
def test_two_pass_update_replayed(cc, updates):
    """The list counter a replay appends through starts at zero each time."""
    import oracle
    r = np.random.default_rng(updates)
    st = torch.cuda.Stream()
    n, k = 20_000, 5_000
    e = [torch.empty((k, 2), dtype=torch.int32, device="cuda") for _ in range(updates)]
    f = cc.Forest(n, stream=st, update_variant=4, compress_every=0)
    ref = oracle.OracleUF(n)

    def fill():
        for x in e:
            p = r.integers(0, n, size=(k, 2)).astype(np.int32)
            ref.bulk_update(p)
            x.copy_(torch.from_numpy(p))
        torch.cuda.synchronize()

    fill()
    for x in e:
        f.bulk_update(x)            # the list is made here
    torch.cuda.synchronize()
    g = record(st, lambda: [f.bulk_update(x) for x in e])
    for eager in (False, False, True, False):
        fill()
        if eager:
            for x in e:
                f.bulk_update(x)
        else:
            g.replay()
        torch.cuda.synchronize()
    assert np.array_equal(f.labels().cpu().numpy(), ref.labels())
    f.sync()


@pytest.mark.parametrize("opts", [{"update_variant": 4}, {"edge_order": 6}, {"update_variant": 4, "edge_order": 9}])
def test_replay_after_a_larger_call_has_outgrown_the_scratch(cc, opts):
    import oracle
    r = np.random.default_rng(3)
    st = torch.cuda.Stream()
    n, k = 50_000, 6_000
    small = torch.empty((k, 2), dtype=torch.int32, device="cuda")
    large = torch.empty((5 * k, 2), dtype=torch.int32, device="cuda")
    f = cc.Forest(n, stream=st, **opts)
    ref = oracle.OracleUF(n)

    def fill(x):
        p = r.integers(0, n, size=x.shape).astype(np.int32)
        ref.bulk_update(p)
        x.copy_(torch.from_numpy(p))
        torch.cuda.synchronize()

    fill(small)
    f.bulk_update(small)
    torch.cuda.synchronize()
    g = record(st, lambda: f.bulk_update(small))
    if "edge_order" in opts:
        f.set_option("edge_order", 9)       # more buckets: the counters are outgrown too
    fill(large)
    f.bulk_update(large)
    for _ in range(2):
        fill(small)
        g.replay()
        torch.cuda.synchronize()
    assert np.array_equal(f.labels().cpu().numpy(), ref.labels())
    f.sync()
