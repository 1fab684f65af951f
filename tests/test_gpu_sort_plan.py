"""Sorts that leave low digits out and order the runs that remain by counting:
whatever the plan picks, orders equal the oracle's, and so do the positions
that queries find in the sorted prefixes."""
import numpy as np
import pytest

import oracle as O
import synthdata as S

pytestmark = pytest.mark.gpu


def _data(kind, n, d, seed):
    g = np.random.default_rng(seed)
    if kind == "scattered":
        return S.unit_gaussian(n, d, seed=seed)
    if kind == "clusters":  # a few hundred tight groups: long runs of equal top bits
        c = g.standard_normal((n // 200 + 1, d)).astype(np.float32)
        return c[g.integers(0, len(c), n)] + 1e-2 * g.standard_normal((n, d)).astype(np.float32)
    if kind == "one tight cluster":  # equal first words for all but the corners
        x = 1e-3 * g.standard_normal((n, d)).astype(np.float32)
        x[:4] = (S.unit_gaussian(4, d, seed=seed) * 5)[:n]
        return x
    return g.integers(0, 3, (n, d)).astype(np.float32)  # few distinct rows


@pytest.mark.parametrize("kind", ["scattered", "clusters", "one tight cluster", "few values"])
@pytest.mark.parametrize("n,d,bits,opts", [
    (30000, 16, 8, None),             # the prefix is the whole key
    (20000, 384, 8, None),            # top level only
    (20000, 64, 8, "prefix_words=1"),
    (9000, 6, 8, None),               # one word holds the key
    (9000, 40, 5, "sort_batch=2"),    # batches of 2 and 1 trees
    (4097, 100, 8, "prefix_words=3"), # three words: every pass runs
    (5, 20, 8, None), (2, 3, 2, None),
])
def test_orders_and_positions(kind, n, d, bits, opts):
    import torch
    import paper_2508_21682_gb300 as hf
    x = _data(kind, n, d, 3 * n + d).astype(np.float32)
    F = O.Forest(x, T=3, bits=bits, seed=5)
    q = x[:: max(1, n // 40)] + np.float32(1e-3)
    qc = O.query_codes(F, q)
    with hf.Forest(torch.from_numpy(x).cuda(), T=3, bits=bits, seed=5, options=opts) as G:
        for t in range(3):
            assert np.array_equal(G.order(t).astype(np.int64), F.sigma[t]), t
            assert np.array_equal(G.locate(t, torch.from_numpy(q).cuda()), O.locate(F, t, qc)), t


@pytest.mark.parametrize("kind", ["scattered", "clusters"])
def test_large_sample(kind):
    """From 2^18 points on the plan samples 4096 of them; the order is checked
    by its own property: full keys ascend, equal keys in index order."""
    import torch
    import paper_2508_21682_gb300 as hf
    n, d = (1 << 18) + 3, 16
    x = _data(kind, n, d, 5)
    with hf.build(torch.from_numpy(x).cuda(), T=2, bits=8, seed=5) as G:
        for t in range(2):
            k, o = G.keys(t), G.order(t).astype(np.int64)
            assert np.array_equal(np.sort(o), np.arange(n))
            assert np.array_equal(o, np.lexsort((np.arange(n), k[:, 1], k[:, 0])))
