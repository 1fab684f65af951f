"""Runs of equal key prefixes: the fix-up's three sources of the next key word,
run lengths around its caps, and near-duplicate groups that tie further down.
Orders are whole numbers, so they equal the oracle's exactly."""
import numpy as np
import pytest

import oracle as O
import synthdata as S

pytestmark = pytest.mark.gpu


def _points(d, seed):
    """Groups of rows that share their coarse codes (long prefix ties) and
    groups of exact copies, between scattered rows."""
    g = np.random.default_rng(seed)
    parts = [S.unit_gaussian(700, d, seed=seed)]
    for size in (2, 3, 31, 33, 256, 257, 1000):
        parts.append(np.repeat(g.standard_normal((1, d)) * 0.2, size, 0) + 2e-3 * g.standard_normal((size, d)))
    for size in (2, 3, 255, 256, 257):
        parts.append(np.repeat(g.standard_normal((1, d)) * 0.2, size, 0))
    x = np.concatenate(parts).astype(np.float32)
    return x[g.permutation(len(x))]


@pytest.mark.parametrize("d,bits,opts", [
    (128, 8, "prefix_words=1"),   # next word in the top level: ballots
    (64, 8, "prefix_words=1"),    # two levels: transform of the listed points
    (33, 8, None),                # six levels
    (100, 8, None),               # the key kernel's own extra word
    (16, 8, "prefix_words=1"),    # the next word completes the key
    (70, 1, "prefix_words=1"),    # one level only, a partial last word
])
def test_runs_of_equal_prefixes(d, bits, opts):
    import torch
    import paper_2508_21682_gb300 as hf
    x = _points(d, 11 + d)
    F = O.Forest(x, T=3, bits=bits, seed=5)
    with hf.Forest(torch.from_numpy(x).cuda(), T=3, bits=bits, seed=5, options=opts) as G:
        for t in range(3):
            assert np.array_equal(G.order(t).astype(np.int64), F.sigma[t]), t


@pytest.mark.parametrize("size", [8191, 8192, 8193])
def test_run_at_the_cap(size):
    """One run of `size` equal prefixes, next to short ones."""
    import torch
    import paper_2508_21682_gb300 as hf
    g = np.random.default_rng(size)
    x = np.concatenate([S.unit_gaussian(500, 33, seed=3) * 4,
                        0.1 + 1e-2 * g.standard_normal((size, 33)).astype(np.float32)]).astype(np.float32)
    F = O.Forest(x, T=2, bits=8, seed=6)
    with hf.Forest(torch.from_numpy(x).cuda(), T=2, bits=8, seed=6, options="prefix_words=1") as G:
        for t in range(2):
            assert np.array_equal(G.order(t).astype(np.int64), F.sigma[t]), t
