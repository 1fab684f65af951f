"""Per-set ranges of a segmented matrix at the edges of the kernel's row and
column chunks."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,d", [
    ([2, 2, 3, 700, 2, 4096, 33], 64),
    ([5, 300, 2], 33),             # one column per lane
    ([20000, 2, 9000], 4),         # eight rows per warp
    ([40, 41], 1),
    ([257, 1000], 200),            # a last column chunk that is not full
])
def test_segment_ranges(sizes, d):
    """Codes of a segmented matrix equal those of each set built alone."""
    import torch
    import paper_2508_21682_gb300 as hf
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = S.unit_gaussian(int(off[-1]), d, seed=9)
    for i, s in enumerate(sizes):
        x[off[i]:off[i + 1]] = x[off[i]:off[i + 1]] * (1 + i) - 0.25 * i
    xd = torch.from_numpy(x).cuda()
    with hf.build_segmented(xd, off, T=1, bits=8, seed=5) as G:
        got = G.codes()
    for i in range(len(sizes)):
        with hf.build(xd[off[i]:off[i + 1]].clone(), T=1, bits=8, seed=5) as H:
            assert np.array_equal(got[off[i]:off[i + 1]], H.codes()), i
