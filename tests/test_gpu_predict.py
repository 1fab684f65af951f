"""Predictions at the edges of the row tiles and input chunks, against the
float64 network with the same BF16 storage."""
import numpy as np
import pytest

from oracle import budget as OB
import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(1, 64), (127, 100), (129, 33), (300, 1), (513, 65), (40000, 384), (130, 1000)])
def test_predict_edges(n, d):
    import torch
    import paper_2508_21682_gb300 as hf
    x = S.unit_gaussian(n, d, seed=7)
    m = hf.Mlp(d, seed=3)
    p = m.get_params()
    g = np.random.default_rng(d)
    p = (p + 0.02 * g.standard_normal(p.shape)).astype(np.float32)  # biases too
    m.set_params(p)
    xd = torch.from_numpy(x).cuda()
    y = m.predict(xd).cpu().numpy()
    host = np.empty((n, 2), np.float32)
    m.predict(xd, out=host)
    assert np.array_equal(host, y)
    rows = np.unique(np.concatenate([np.arange(min(n, 200)), np.arange(max(0, n - 200), n)]))
    ref, _ = OB.mlp_forward(p, x[rows])
    assert np.max(np.abs(y[rows] - ref)) <= 1e-2 * max(1.0, np.max(np.abs(ref)))
    m.close()
