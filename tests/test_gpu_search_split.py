"""Small query batches share a query among several warps (trees, then window
chunks) and merge the parts' lists. hf_search_static never splits, so its lists
are the general path's: both must agree element by element."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,T,w,k,d,n", [
    (1, 40, 100, 10, 64, 5000),    # every tree and four chunks of a window apart
    (5, 32, 32, 32, 384, 3000),
    (3, 1, 40, 33, 100, 2000),     # one tree: chunks only; two list slots per lane
    (60, 40, 20, 1, 33, 1500),     # rows not float4-aligned; a tree per warp
    (1216, 3, 50, 50, 16, 900),    # the largest batch that splits
    (1217, 3, 50, 50, 16, 900),    # the first that does not
    (2, 3, 700, 64, 24, 300),      # windows wider than the set: unfilled tails, repeats in every tree
])
def test_split_search_equals_unsplit(nq, T, w, k, d, n):
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.gaussian_mixture(n, d, n_components=20, seed=3)).cuda()
    q = torch.from_numpy(S.mixture_queries(nq, d, n_components=20, data_seed=3, seed=4)).cuda()
    with hf.build(x, T=T, bits=8, seed=5) as G:
        ri, rd = G.search(q, k, w)
        si, sd = G.search_static(q, k, w)
        assert torch.equal(ri, si) and torch.equal(rd, sd)


@pytest.mark.parametrize("d,T,w,k,n,shift,scale", [
    (384, 8, 50, 30, 4000, 0.0, 1.0),
    (64, 5, 40, 33, 3000, 0.0, 1.0),      # two list slots per lane
    (100, 5, 64, 10, 3000, 30.0, 1.0),    # copies farther from their points than the points from each other
    (68, 4, 40, 10, 2000, 0.0, 3e18),     # squares near the top of the range, some beyond it
    (128, 4, 40, 10, 2000, 0.0, 1e-20),   # squares below it
    (128, 4, 300, 50, 200, 0.0, 1.0),     # windows wider than the set, unfilled tails
])
def test_half_width_screen_keeps_the_lists(d, T, w, k, n, shift, scale):
    """Large batches screen candidates against a BF16 copy; hf_search_static
    reads the float32 rows only. Repeated points make ties."""
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.gaussian_mixture(n, d, n_components=20, seed=3)
    x[n // 2: n // 2 + 40] = x[:40]
    q = S.mixture_queries(2000, d, n_components=20, data_seed=3, seed=4)
    q[:50] = x[:50]
    x, q = (x * np.float32(scale) + np.float32(shift)), (q * np.float32(scale) + np.float32(shift))
    xd, qd = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
    with hf.build(xd, T=T, bits=8, seed=5) as G:
        ri, rd = G.search(qd, k, w)
        si, sd = G.search_static(qd, k, w)
        assert torch.equal(ri, si) and torch.equal(rd, sd)
        ri, rd = G.search(qd, k, w)  # the copy is there now
        assert torch.equal(ri, si) and torch.equal(rd, sd)
