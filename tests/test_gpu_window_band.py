"""The plain and sketch forms' pair band: offset tiles of 64, 32 and 16 and
their remainders, row chunks of a band that does not fit its scratch at once,
set boundaries, and lists of 16, 32 and 64 slots while they fill.

Integer-valued points: every squared distance is exact in float32, so the lists
equal a brute force over the orders' windows element by element."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


def _brute(x, orders, rows, w, k, bounds):
    """Top k by (distance, index) of the window candidates of `rows`."""
    n = len(x)
    pos = [np.argsort(o, kind="stable") for o in orders]
    xi = x.astype(np.int64)
    out_i, out_d = np.full((len(rows), k), -1, np.int64), np.full((len(rows), k), np.inf)
    for a, r in enumerate(rows):
        cand = set()
        for o, p in zip(orders, pos):
            q = int(p[r])
            lo, hi = bounds(r, n)
            cand.update(o[max(lo, q - w):min(hi, q + w + 1)].tolist())
        cand.discard(int(r))
        c = np.array(sorted(cand), np.int64)
        d = ((xi[c] - xi[r]) ** 2).sum(1)
        s = np.lexsort((c, d))[:k]
        out_i[a, :len(s)], out_d[a, :len(s)] = c[s], d[s]
    return out_i, out_d


@pytest.mark.parametrize("n,d,T,w,k", [
    (3000, 8, 3, 1, 1),
    (3000, 17, 3, 15, 16), (3000, 16, 3, 16, 17), (3000, 20, 2, 17, 10), (3000, 8, 2, 33, 32),
    (3000, 8, 3, 48, 33), (3000, 9, 2, 49, 10), (3000, 8, 2, 64, 64), (3000, 8, 2, 65, 20),
    (3000, 8, 2, 112, 50), (3000, 8, 2, 704, 40),
    (511, 8, 2, 300, 10), (20, 8, 2, 64, 30),
    (200_000, 4, 2, 704, 12),  # several row chunks
])
def test_window_lists_equal_brute_force(n, d, T, w, k):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.small_integer_points(n, d, seed=n + w)
    with hf.build(torch.from_numpy(x).cuda(), T=T, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(T)]
        gi, gd = G.knn_graph(k, w)
        gi, gd = gi.cpu().numpy(), gd.cpu().numpy()
    rows = np.arange(n) if n <= 3000 else np.unique(np.concatenate(
        [orders[0][::997], *[orders[0][a:b] for a, b in ((0, 8), (n - 8, n))]]))
    rows = rows[::max(1, len(rows) // 600)]
    oi, od = _brute(x, orders, rows, w, k, lambda r, m: (0, m))
    assert np.array_equal(gi[rows], oi) and np.array_equal(gd[rows].astype(np.float64), od)


def test_window_stays_within_sets():
    import torch
    import paper_2508_21682_gb300 as hf
    sizes = [2, 700, 3, 64, 1500]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    x = S.small_integer_points(int(off[-1]), 8, seed=2)
    with hf.build_segmented(torch.from_numpy(x).cuda(), off, T=2, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(2)]
        gi, gd = G.knn_graph(12, 80)
    seg = np.searchsorted(off, np.arange(len(x)), side="right") - 1
    oi, od = _brute(x, orders, np.arange(len(x)), 80, 12, lambda r, m: (off[seg[r]], off[seg[r] + 1]))
    assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gd.cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("threads", [0, 256, 512])
def test_planned_window_equals_direct(threads):
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.gaussian_mixture(5000, 40, n_components=20, seed=3)).cuda()
    with hf.build(x, T=3, bits=8, seed=5) as G:
        ri, rd = G.knn_graph(10, 100)
        oi, od = torch.empty_like(ri), torch.empty_like(rd)
        G.graph_plan(10, 100, threads)
        G.knn_graph_enqueue(oi, od)
        G.status()
        assert torch.equal(ri, oi) and torch.equal(rd, od)
