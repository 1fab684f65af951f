"""Plain windows of small matrices whose rows are not 16-byte aligned: they take
other tiles than aligned rows, with the same pairs, sums and lists."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,w", [
    (2, 16, 3), (200, 16, 2), (255, 16, 16), (257, 16, 17), (3000, 32, 33), (3000, 16, 80), (3000, 16, 130),
    (152 * 256, 8, 5), (152 * 256 + 1, 8, 5),          # the last size of the rule at w < 64, and the next
    (76 * 256, 8, 70), (76 * 256 + 1, 8, 70),          # at w < 128
])
def test_unaligned_rows_equal_aligned_rows(n, d, w):
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.unit_gaussian(n, d, seed=n + w)).cuda()
    buf = torch.empty(n * d + 1, device="cuda")
    y = buf[1:].view(n, d)
    y.copy_(x)
    assert x.data_ptr() % 16 == 0 and y.data_ptr() % 16 == 4
    k = min(12, n)
    with hf.build(x, T=2, bits=8, seed=5) as F, hf.build(y, T=2, bits=8, seed=5) as G:
        ai, ad = F.knn_graph(k, w)
        bi, bd = G.knn_graph(k, w)
    # the lists come from the same sums; the re-rank adds unaligned rows' lanes in another order
    assert torch.equal(ai, bi)
    a, b = ad.cpu().numpy().astype(np.float64), bd.cpu().numpy().astype(np.float64)
    ok = np.isfinite(a)
    assert np.array_equal(ok, np.isfinite(b))
    assert np.all(np.abs(a[ok] - b[ok]) <= 2 * (4 + 7 + d / 32) * 2.0 ** -24 * a[ok])
