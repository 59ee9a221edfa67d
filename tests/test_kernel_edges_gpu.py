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
    assert np.array_equal(f.labels().cpu().numpy(), lab)
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
