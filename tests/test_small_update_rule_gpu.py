"""The one-CTA Bulk-Update at the ends of its range, with and without a compression due."""
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


@pytest.mark.parametrize("every", [0, 1, 2])
@pytest.mark.parametrize("k", [2048, 2049, 4096, 4097])
@pytest.mark.parametrize("n", [8192, 8193])
def test_both_sides_of_the_rule(cc, n, k, every):
    import oracle
    r = np.random.default_rng(n + k + every)
    f = cc.Forest(n, compress_every=every)
    ref = oracle.OracleUF(n)
    for step in range(5):
        x = np.sort(r.choice(n, size=k + 1, replace=False)).astype(np.int32)     # a path: deep trees
        p = np.stack([x[1:], x[:-1]], axis=1) if step % 2 == 0 else r.integers(0, n, size=(k, 2)).astype(np.int32)
        q = r.integers(0, n, size=(3000, 2)).astype(np.int32)
        f.bulk_update(torch.from_numpy(p).cuda())
        ref.bulk_update(p)
        assert np.array_equal(f.bulk_query(torch.from_numpy(q).cuda()).cpu().numpy(), ref.bulk_query(q))
        if every == 1 or (n == 8192 and k <= 2048):
            assert f.depth()[0] <= 1
    assert np.array_equal(f.labels().cpu().numpy(), ref.labels())
    f.sync()
