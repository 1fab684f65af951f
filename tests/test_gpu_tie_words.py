"""Near-duplicates in many dimensions: members that tie on the words the fix-up
has at hand, told apart by later words of the top bit level or by the full key,
in groups around a warp's and a block's share. Orders are whole numbers, so
they equal the oracle's exactly."""
import numpy as np
import pytest

import oracle as O
import synthdata as S

pytestmark = pytest.mark.gpu


def _points(d, n_loose, seed):
    """Scattered rows, groups that differ in the signs of few coordinates (the
    centres' coordinates are far from the axes' middles beside the noise),
    groups that differ in low bits only, and groups of copies."""
    g = np.random.default_rng(seed)
    parts = [S.unit_gaussian(n_loose, d, seed=seed)]
    for noise in (0.05, 0.004, 0.0):
        for size in (2, 3, 4, 5, 15, 16, 17, 31, 32, 33, 70):
            c = g.standard_normal((1, d)) * d ** -0.5
            parts.append(c + noise * d ** -0.5 * g.standard_normal((size, d)))
    x = np.concatenate(parts).astype(np.float32)
    return x[g.permutation(len(x))]


@pytest.mark.parametrize("d,bits,opts", [
    (256, 8, None),               # one word past word K in the top level
    (383, 8, None),               # two
    (384, 8, None),               # three
    (384, 8, "prefix_words=1"),
    (200, 8, None),               # none: full keys at once
    (384, 1, None),               # the top level is the whole key
    (330, 1, None),               # a partial last word after it
    (768, 4, None),               # rows of half a block
    (1100, 8, None),              # more than 128 key words
    (4096, 8, None),              # four rows a warp
])
def test_near_duplicates(d, bits, opts):
    import torch
    import paper_2508_21682_gb300 as hf
    x = _points(d, 300, 17 + d + bits)
    T = 2 if d < 2000 else 1
    F = O.Forest(x, T=T, bits=bits, seed=5)
    with hf.Forest(torch.from_numpy(x).cuda(), T=T, bits=bits, seed=5, options=opts) as G:
        for t in range(T):
            assert np.array_equal(G.order(t).astype(np.int64), F.sigma[t]), t


@pytest.mark.parametrize("d,noise", [(256, 0.02), (384, 0.02), (384, 0.004), (768, 0.0)])
def test_groups_at_the_cap(d, noise):
    """Groups of 255 to 257 members: the largest that a block orders, and the
    smallest that the host settles."""
    import torch
    import paper_2508_21682_gb300 as hf
    g = np.random.default_rng(d)
    parts = [S.unit_gaussian(200, d, seed=3)]
    for size in (100, 255, 256, 257, 300):
        parts.append(g.standard_normal((1, d)) * d ** -0.5 + noise * d ** -0.5 * g.standard_normal((size, d)))
    x = np.concatenate(parts).astype(np.float32)
    x = x[g.permutation(len(x))]
    F = O.Forest(x, T=2, bits=8, seed=6)
    with hf.Forest(torch.from_numpy(x).cuda(), T=2, bits=8, seed=6) as G:
        for t in range(2):
            assert np.array_equal(G.order(t).astype(np.int64), F.sigma[t]), t
