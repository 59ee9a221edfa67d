"""The batched kernel in each of its shapes: pairs in registers or in a ring of two
to four chunks, with more operations than are staged at a time."""
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


@pytest.mark.parametrize("block,ept,cap", [
    (512, 1, 65536), (128, 1, 2048),                       # no ring
    (64, 2, 65536), (1024, 2, 65536), (1024, 4, 65536),    # one CTA per SM: the largest ring that fits
    (256, 2, 32768), (512, 4, 32768), (64, 4, 1024), (1024, 2, 300),
])
def test_many_short_operations(cc, block, ept, cap):
    import oracle
    r = np.random.default_rng(block * ept + cap)
    sizes = [1, 7, 300, min(cap, 5000), min(cap, 40_000)]
    f = cc.Forest.segmented(sizes, seg_block=block, seg_edges_per_thread=ept, seg_smem_cap=cap)
    refs = [oracle.OracleUF(n) for n in sizes]
    buf = torch.empty(4 << 20, dtype=torch.int32, device="cuda")
    host = np.zeros(4 << 20, dtype=np.int32)
    ops, want, at = [], [], 0
    for i in range(700):                                   # more than are staged at a time
        for g, n in enumerate(sizes):
            if i >= 40 and g != i % len(sizes):
                continue
            k = int(r.integers(0, 3)) * block * ept + int(r.integers(0, 90)) if i % 50 == 0 else int(r.integers(0, 60))
            p = r.integers(0, n, size=(k, 2)).astype(np.int32)
            host[at:at + 2 * k] = p.ravel()
            data = buf[at:at + 2 * k].view(k, 2)
            at += 2 * k + int(r.integers(0, 4))            # any 4-byte alignment
            if i % 2:
                out = torch.full((k,), 9, dtype=torch.uint8, device="cuda")
                ops.append((g, cc.OP_QUERY, data, out))
                want.append((out, refs[g].bulk_query(p)))
            else:
                ops.append((g, cc.OP_UPDATE, data, None))
                refs[g].bulk_update(p)
    assert at <= host.size
    buf.copy_(torch.from_numpy(host))
    torch.cuda.synchronize()
    f.submit(ops)
    f.sync()
    for out, exp in want:
        assert np.array_equal(out.cpu().numpy(), exp)
    lab = f.labels().cpu().numpy()
    for g, ref in enumerate(refs):
        a, b = f.offsets[g], f.offsets[g + 1]
        assert np.array_equal(lab[a:b] - a, ref.labels())
    f.sync()
