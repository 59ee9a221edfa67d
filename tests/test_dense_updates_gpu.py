"""Bulk-Updates with two edges per vertex of the graph and more, where the first
parents are read again before a link, and just below that."""
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


@pytest.mark.parametrize("variant", range(6))
@pytest.mark.parametrize("n,k", [(2, 70_000), (16, 300_000), (9000, 17_999), (9000, 18_000), (9000, 300_000)])
def test_dense_minibatches(cc, variant, n, k):
    import oracle
    r = np.random.default_rng(n + k)
    batches = [r.integers(0, n, size=(k, 2)).astype(np.int32) for _ in range(3)]
    batches[0][:, 1] = np.minimum(batches[0][:, 0] + r.integers(0, 3, size=k), n - 1)   # a path first: deep
    ref = oracle.OracleUF(n)
    want = []
    for b in batches:
        ref.bulk_update(b)
        want.append(ref.labels())
    dev = [torch.from_numpy(b).cuda() for b in batches]
    for opts in ({}, {"hook": 1}, {"hook": 2, "compress_every": 0}, {"hook": 1, "hook_warp": 1, "compress_every": 0},
                 {"hook_warp": 1, "edges_per_thread": 4}, {"edges_per_thread": 1, "compress_scope": 1}):
        f = cc.Forest(n, update_variant=variant, **opts)
        for d, w in zip(dev, want):
            f.bulk_update(d)
            if opts.get("compress_every") != 0:
                assert np.array_equal(f.labels().cpu().numpy(), w), opts
        assert np.array_equal(f.labels().cpu().numpy(), want[-1]), opts
        assert f.components() == len(np.unique(want[-1])), opts
        f.sync()
        f.close()
