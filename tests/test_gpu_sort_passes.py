"""What a build reports of its sort passes."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


def test_reported_passes():
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.unit_gaussian(20_000, 64, seed=3)
    spread, copies = torch.from_numpy(x).cuda(), torch.from_numpy(np.repeat(x[:5], 4000, 0)).cuda()
    with hf.build(spread, T=4, bits=8, seed=5) as G:
        assert 4 <= G.timings()["sort_passes"] < 16  # almost no two points share 32 bits
    with hf.build(copies, T=2, bits=8, seed=5) as G:
        assert G.timings()["sort_passes"] == 16
    with hf.build(spread, T=2, bits=8, seed=5, options="prefix_words=3") as G:
        assert G.timings()["sort_passes"] == 24
    with hf.build(spread[:, :8].contiguous(), T=2, bits=8, seed=5) as G:
        assert G.timings()["sort_passes"] <= 8  # a key of one word
