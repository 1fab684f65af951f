"""What a build reports of its own launches and sort passes."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,bits,opts,slice_plane", [
    (384, 8, None, True),                 # words of the top level
    (64, 8, None, False),                 # tie_words
    (100, 8, None, False),                # the key kernel's own third word
    (20, 8, "prefix_words=2", False),     # the third word completes the key
    (3, 8, None, False),                  # the prefix is the whole key
    (384, 8, "prefix_words=3", True),     # three words are always sorted in full
    (64, 8, "sort_batch=2", False),
])
def test_reported_launches(d, bits, opts, slice_plane):
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.unit_gaussian(5000, d, seed=3)).cuda()
    n0 = hf.launch_count()
    with hf.build(x, T=4, bits=bits, seed=5, options=opts) as G:
        launched = hf.launch_count() - n0
        assert launched == G.timings()["build_launches"] + 3 + slice_plane  # range, quantization, plane 0


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
