"""The prediction kernel against the training step's forward pass."""
import numpy as np
import pytest

import synthdata as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(128, 1), (128, 64), (256, 33), (384, 100), (1024, 384), (8192, 65)])
def test_predictions_are_the_training_forward(n, d):
    """With a batch's own predictions as its targets every error y - t of the
    training step is exactly zero, so loss and gradients are, if and only if
    both passes give the same bits."""
    import torch
    import paper_2508_21682_gb300 as hf
    m = hf.Mlp(d, seed=3)
    p = m.get_params()
    p = (p + 0.05 * np.random.default_rng(d).standard_normal(p.shape)).astype(np.float32)  # biases too
    m.set_params(p)
    x = torch.from_numpy(S.unit_gaussian(n, d, seed=7)).cuda()
    y = m.predict(x)
    assert float(y.abs().max()) > 1e-3
    loss, grads = m.grads(x, y)
    assert loss == 0.0 and not np.any(grads)
    loss, _ = m.grads(x, y + 0.5)
    assert loss > 0.0
    m.close()
