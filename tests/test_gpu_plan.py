"""Graph plans of the plain form: what a later plan leaves of an earlier one."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


def _capture(hf, G, oi, od, side):
    graph = hf.CudaGraph(side.cuda_stream)
    with graph:
        G.knn_graph_enqueue(oi, od, side.cuda_stream)
    return graph


@pytest.mark.parametrize("n,later", [(5000, [200]), (5000, [8, 704, 33]), (150_000, [40, 300]), (5000, None)])
def test_replay_after_another_plan(n, later):
    """A captured graph stays right, and writes nothing of another owner's,
    when the forest is planned again for other windows (None: by the tuner)
    and other forests have taken memory meanwhile."""
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.gaussian_mixture(n, 20, n_components=20, seed=3)).cuda()
    side = torch.cuda.Stream()
    with hf.build(x, T=3, bits=8, seed=5) as G:
        windows = [32] + (later or [])
        ref = {w: G.knn_graph(10, w) for w in windows}
        oi, od = torch.empty_like(ref[32][0]), torch.empty_like(ref[32][1])
        side.wait_stream(torch.cuda.current_stream())
        graphs = []
        for w in windows:
            G.graph_plan(10, w, 0, side.cuda_stream)
            graphs.append((w, _capture(hf, G, oi, od, side)))
        if later is None:
            G.autotune(10, 0.99, sample=64, w_max=704, forms=1)
        # forests of many sizes take whatever memory was given back
        others = [hf.build(x[:m].clone(), T=t, bits=8, seed=7) for m in (300, 1000, 2500, n) for t in (1, 4, 16)]
        before = [[o.order(t) for t in range(o.T)] for o in others]
        for _ in range(2):
            for w, graph in graphs:
                with torch.cuda.stream(side):
                    oi.fill_(-7)
                    od.fill_(-7.0)
                graph.launch()
                G.status(side.cuda_stream)
                assert torch.equal(oi, ref[w][0]) and torch.equal(od, ref[w][1]), w
        for o, orders in zip(others, before):
            for t, a in enumerate(orders):
                assert np.array_equal(o.order(t), a)
            o.close()
        for _, graph in graphs:
            graph.close()


@pytest.mark.parametrize("w", [480, 481, 520, 704])
@pytest.mark.parametrize("threads", [0, 256, 512])
def test_block_sizes_at_wide_windows(threads, w):
    """Every block size that a plan accepts runs at every window of the form."""
    import torch
    import paper_2508_21682_gb300 as hf
    x = torch.from_numpy(S.gaussian_mixture(3000, 24, n_components=20, seed=3)).cuda()
    with hf.build(x, T=2, bits=8, seed=5) as G:
        ri, rd = G.knn_graph(10, w)
        oi, od = torch.empty_like(ri), torch.empty_like(rd)
        G.graph_plan(10, w, threads)
        G.knn_graph_enqueue(oi, od)
        G.status()
        assert torch.equal(ri, oi) and torch.equal(rd, od)
