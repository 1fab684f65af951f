"""Large query batches: positions located in a launch of their own, candidates
screened, survivors scored several at a time. hf_search_static takes neither, so
both must agree element by element."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq,T,w,k,d,n,launches", [
    (1500, 40, 40, 64, 384, 4000, 3),   # two list slots per lane: quantize, locate, search
    (1500, 30, 64, 33, 128, 3000, 3),
    (2000, 24, 60, 50, 768, 2000, 3),
    (1024, 40, 40, 64, 384, 4000, 4),   # parts and their merge
    (1216, 16, 50, 10, 64, 3000, 4),
    (2100, 4096, 8, 10, 64, 300, 5),    # located in two slices
    (1300, 5, 300, 1, 68, 400, 3),      # windows wider than the set
    (2000, 8, 32, 64, 128, 1000, 2),    # few rows per slot of a long list: not screened
    (2000, 8, 32, 30, 128, 1000, 3),
])
def test_screened_search_equals_plain(nq, T, w, k, d, n, launches):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.gaussian_mixture(n, d, n_components=20, seed=3)
    x[n // 2: n // 2 + 60] = x[:60]  # ties, and equal keys inside a prefix
    q = S.mixture_queries(nq, d, n_components=20, data_seed=3, seed=4)
    q[:60] = x[:60]
    xd, qd = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
    with hf.build(xd, T=T, bits=8, seed=5) as G:
        si, sd = G.search_static(qd, k, w)
        for _ in range(2):  # the first makes the copy
            n0 = hf.launch_count()
            ri, rd = G.search(qd, k, w)
            n1 = hf.launch_count()
            assert torch.equal(ri, si) and torch.equal(rd, sd)
        assert n1 - n0 == launches


def test_screened_lists_of_far_apart_values():
    """Rows whose squares overflow next to ordinary ones, lists that stay short."""
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.gaussian_mixture(60, 64, n_components=5, seed=3)
    x[::7] *= np.float32(1e19)
    q = np.repeat(x, 20, 0)[:1100]
    xd, qd = torch.from_numpy(x).cuda(), torch.from_numpy(q).cuda()
    with hf.build(xd, T=16, bits=8, seed=5) as G:
        si, sd = G.search_static(qd, 32, 9)
        ri, rd = G.search(qd, 32, 9)
        assert torch.equal(ri, si) and torch.equal(rd, sd)
