"""Bulk-Query on both sides of its size rule: both nodes of a pair moved up, or
the larger one alone (large forests)."""
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


def roots_of(par):
    r = par.copy()
    while not np.array_equal(r[r], r):
        r = r[r]
    return r


@pytest.mark.parametrize("shape", ["flat", "random", "chains"])
@pytest.mark.parametrize("n", [(1 << 22) - 1, 1 << 22])
def test_answers_on_both_sides_of_the_rule(cc, n, shape):
    r = np.random.default_rng(n)
    par = np.arange(n, dtype=np.int32)
    if shape == "flat":
        par[1:] = np.where(r.random(n - 1) < 0.6, r.integers(0, 3, n - 1), par[1:])
        par[:3] = 0, 1, 2
    elif shape == "random":
        par[1:] = np.where(r.random(n - 1) < 0.95, (r.random(n - 1) * np.arange(1, n)).astype(np.int32), par[1:])
    else:
        par[20_000:] = np.arange(n - 20_000)
    root = roots_of(par)
    for k in ((1 << 17) - 1, (1 << 17) + 3):
        q = r.integers(0, n, size=(k, 2)).astype(np.int32)
        q[::7, 1] = q[::7, 0]
        q[1::5, 1] = root[q[1::5, 0]]
        q[2::5, 1] = par[par[q[2::5, 0]]]
        q[3::5] = q[3::5, ::-1]
        want = (root[q[:, 0]] == root[q[:, 1]]).astype(np.uint8)
        d = torch.from_numpy(q).cuda()
        for opts in ({}, {"query_halving": 1}, {"query_pairs_per_thread": 4, "query_variant": 1},
                     {"query_pairs_per_thread": 1, "query_halving": 1}):
            f = cc.Forest(n, **opts)
            p = torch.from_numpy(root if shape == "flat" else par).cuda()
            (f.load_labels if shape == "flat" else f.load_forest)(p)
            assert np.array_equal(f.bulk_query(d).cpu().numpy(), want), (k, opts)
            got = f.parent().cpu().numpy()
            assert (got <= par).all() and np.array_equal(roots_of(got), root)
            f.sync()
            f.close()
