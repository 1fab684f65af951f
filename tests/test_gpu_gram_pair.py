"""Wide windows of the tensor forms (two CTAs per tile of 256 positions) at the
edges of tiles, units and sets.

Integer-valued points: BF16 rounding, inner products and squared distances are
exact in float32, so the lists equal a brute force over the orders' windows
element by element. FP8 rounds such points, so its lists are checked for what
must hold of every pick and for the share of the true neighbours found."""
import numpy as np
import pytest

import oracle as O
import synthdata as S
from _helpers import check_tensor_lists

pytestmark = pytest.mark.gpu


def _brute(x, orders, rows, k, span):
    """Top k by (distance, index); span(row, position, tree) -> [lo, hi)."""
    pos = [np.argsort(o, kind="stable") for o in orders]
    xi = x.astype(np.int64)
    out_i, out_d = np.full((len(rows), k), -1, np.int64), np.full((len(rows), k), np.inf)
    for a, r in enumerate(rows):
        cand = set()
        for t, (o, p) in enumerate(zip(orders, pos)):
            lo, hi = span(int(r), int(p[r]), t)
            cand.update(o[lo:hi].tolist())
        cand.discard(int(r))
        c = np.array(sorted(cand), np.int64)
        d = ((xi[c] - xi[r]) ** 2).sum(1)
        s = np.lexsort((c, d))[:k]
        out_i[a, :len(s)], out_d[a, :len(s)] = c[s], d[s]
    return out_i, out_d


@pytest.mark.parametrize("n,d,w,k", [
    (127, 8, 128, 10), (129, 8, 128, 10), (255, 64, 200, 15), (257, 70, 128, 15), (385, 8, 1000, 20),
    (2500, 100, 129, 10), (2500, 64, 256, 15), (3000, 384, 300, 15), (2500, 512, 400, 31), (40000, 16, 1024, 15),
])
def test_pair_tiles_equal_brute_force(n, d, w, k):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.small_integer_points(n, d, seed=n + d)
    with hf.build(torch.from_numpy(x).cuda(), T=2, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(2)]
        G.set_option("mode", 1)
        gi, gd = G.knn_graph(k, w)
        assert G.timings()["graph_form"] == 1.0
        gi, gd = gi.cpu().numpy(), gd.cpu().numpy()
    rows = np.arange(n) if n <= 3000 else np.unique(np.concatenate([orders[0][::211], orders[0][:3], orders[0][-3:]]))
    oi, od = _brute(x, orders, rows, k, lambda r, p, t: (max(0, p - w), min(n, p + w + 1)))
    assert np.array_equal(gi[rows], oi) and np.array_equal(gd[rows].astype(np.float64), od)


@pytest.mark.parametrize("n,d,w,k", [(9001, 8, 4097, 10), (9001, 300, 9000, 15), (18000, 8, 8200, 20)])
def test_windows_wider_than_the_bounds_pass(n, d, w, k):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.small_integer_points(n, d, seed=n + d)
    x[n // 2:n // 2 + 40] = x[:40]  # equal points far apart by index
    with hf.build(torch.from_numpy(x).cuda(), T=2, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(2)]
        G.set_option("mode", 1)
        gi, gd = G.knn_graph(k, w)
        assert G.timings()["graph_form"] == 1.0
        wp = torch.from_numpy(np.random.default_rng(1).integers(1, w + 1, n).astype(np.int32)).cuda()
        bi, bd = G.knn_graph_budget(k, wp, torch.full((n,), 2, dtype=torch.int32, device="cuda"))
        wp = wp.cpu().numpy()
    rows = np.unique(np.concatenate([np.arange(0, n, 151), orders[0][:3], orders[0][-3:]]))
    oi, od = _brute(x, orders, rows, k, lambda r, p, t: (max(0, p - w), min(n, p + w + 1)))
    assert np.array_equal(gi.cpu().numpy()[rows], oi) and np.array_equal(gd.cpu().numpy()[rows].astype(np.float64), od)
    oi, od = _brute(x, orders, rows, k, lambda r, p, t: (max(0, p - wp[r]), min(n, p + wp[r] + 1)))
    bi, bd = bi.cpu().numpy()[rows], bd.cpu().numpy()[rows].astype(np.float64)
    assert np.array_equal(bi, oi) and np.array_equal(bd, od)


def test_pair_tiles_within_sets_and_budgets():
    import torch
    import paper_2508_21682_gb300 as hf
    sizes = [2, 700, 3, 130, 1500, 255]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(off[-1])
    x = S.small_integer_points(n, 24, seed=2)
    xd = torch.from_numpy(x).cuda()
    seg = np.searchsorted(off, np.arange(n), side="right") - 1
    with hf.build_segmented(xd, off, T=2, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(2)]
        G.set_option("mode", 1)
        gi, gd = G.knn_graph(12, 200)
    oi, od = _brute(x, orders, np.arange(n), 12,
                    lambda r, p, t: (max(off[seg[r]], p - 200), min(off[seg[r] + 1], p + 201)))
    assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gd.cpu().numpy().astype(np.float64), od)
    g = np.random.default_rng(3)
    wp = g.integers(0, 400, n).astype(np.int32)
    wp[g.random(n) < 0.3] = 0
    tp = g.integers(0, 3, n).astype(np.int32)
    with hf.build(xd, T=2, bits=8, seed=5) as G:
        orders = [G.order(t).astype(np.int64) for t in range(2)]
        wp[orders[0][512:1024]] = 0  # whole tiles without a window
        G.set_option("mode", 1)
        gi, gd = G.knn_graph_budget(12, torch.from_numpy(wp).cuda(), torch.from_numpy(tp).cuda())

    def span(r, p, t):
        return (max(0, p - wp[r]), min(n, p + wp[r] + 1)) if t < tp[r] and wp[r] > 0 else (p, p + 1)
    oi, od = _brute(x, orders, np.arange(n), 12, span)
    assert np.array_equal(gi.cpu().numpy(), oi) and np.array_equal(gd.cpu().numpy().astype(np.float64), od)


@pytest.mark.parametrize("n,d,w", [(2500, 100, 129), (3001, 768, 300), (1500, 896, 128)])
def test_pair_tiles_fp8(n, d, w):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.gaussian_mixture(n, d, n_components=20, seed=3)
    F = O.Forest(x, T=2, bits=8, seed=5)
    with hf.build(torch.from_numpy(x).cuda(), T=2, bits=8, seed=5) as G:
        G.set_option("mode", 2)
        G.set_option("tensor_slack", 17)
        gi, gd = G.knn_graph(15, w)
        assert G.timings()["graph_form"] == 2.0
    oi, _ = O.knn_graph(F, 15, w)
    check_tensor_lists(x, gi.cpu().numpy(), gd.cpu().numpy(), oi, np.arange(n), min_hit=0.93)


@pytest.mark.parametrize("mode,d,w", [(0, 40, 100), (1, 384, 40), (1, 384, 300), (2, 768, 300)])
def test_captured_plan_equals_direct(mode, d, w):
    """Pairs, the bound pass, single tiles and the plain band, replayed from a
    captured graph after the direct call left other values in the outputs."""
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.gaussian_mixture(6000, d, n_components=20, seed=4)).cuda()
    with hf.build(x, T=3, bits=8, seed=5) as G:
        G.set_option("mode", mode)
        ri, rd = G.knn_graph(10, w)
        assert G.timings()["graph_form"] == mode
        G.graph_plan(10, w)
        oi, od = torch.full_like(ri, -7), torch.full_like(rd, -7.0)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        graph = hf.CudaGraph(side.cuda_stream)
        with graph:
            G.knn_graph_enqueue(oi, od, side.cuda_stream)
        for _ in range(2):
            graph.launch()
            G.status(side.cuda_stream)
            assert torch.equal(oi, ri) and torch.equal(od, rd)
            with torch.cuda.stream(side):
                oi.fill_(-7)
                od.fill_(-7.0)
        graph.close()
