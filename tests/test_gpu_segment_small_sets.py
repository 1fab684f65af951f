"""Per-set ranges of many small sets, and of sets at the edges of a block's row
share beside them."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,d", [
    ([2] * 256, 16),
    ([3] * 100 + [256, 255, 257, 2, 511, 512, 513, 2], 16),   # 256 rows a block
    ([64, 63, 65, 2, 127, 128, 129] * 8, 64),                 # 64 rows a block
    ([1024, 1023, 1025, 2, 5000, 2, 2], 4),                   # 1,024 rows a block
    ([2] * 100 + [40_000] + [2] * 100, 33),                   # one lane per column, many chunks of one set
])
def test_ranges_of_small_sets(sizes, d):
    """Codes of a segmented matrix equal those of each set built alone."""
    import torch
    import paper_2508_21682_gb300 as hf
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = S.unit_gaussian(int(off[-1]), d, seed=9)
    for i in range(len(sizes)):
        x[off[i]:off[i + 1]] = x[off[i]:off[i + 1]] * (1 + i % 7) - np.float32(0.25) * (i % 5)
    xd = torch.from_numpy(x).cuda()
    with hf.build_segmented(xd, off, T=1, bits=8, seed=5) as G:
        got = G.codes()
    for i in range(len(sizes)):
        with hf.build(xd[off[i]:off[i + 1]].clone(), T=1, bits=8, seed=5) as H:
            assert np.array_equal(got[off[i]:off[i + 1]], H.codes()), i


@pytest.mark.parametrize("row", [0, 2, 200, 255, 256, 700, 1023])
def test_non_finite_rows_are_found(row):
    import torch
    import paper_2508_21682_gb300 as hf
    off = np.concatenate([[0], np.cumsum([2] * 100 + [600, 224])]).astype(np.int64)
    x = S.unit_gaussian(1024, 16, seed=9)
    x[row, 5] = np.nan
    with pytest.raises(hf.HFError):
        hf.build_segmented(torch.from_numpy(x).cuda(), off, T=1, bits=8, seed=5)
