"""The gradient kernel of the guess network at the edges of its chunks of 64 samples and of its 256 blocks, against the
FP64 reference (oracle/mlp_ref.py).

Tolerance: each entry is a sum of n products in FP32 whose factors carry a few roundings of the 64-term layers, so its
error is below 2e-4 of the entry plus 1% of the layer's largest entry: the bound of the full-batch gradient test."""
import numpy as np
import pytest

from oracle import mlp_ref as M
from paper_1802_04449_gb300 import clv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 63, 64, 65, 127, 256 * 64, 256 * 64 + 1])
def test_gradient_at_chunk_edges(n):
    import torch
    rng = np.random.default_rng(n)
    p = (M.init_params(2) + 0.05 * rng.normal(size=M.NPARAM)).astype(np.float32)
    X, Y = rng.normal(size=(n, M.NIN)).astype(np.float32), rng.normal(size=(n, M.NOUT)).astype(np.float32)
    loss_ref, g_ref = M.loss_and_grad(p.astype(np.float64), X.astype(np.float64), Y.astype(np.float64))
    loss, g = clv.mlp_loss_grad(*(torch.tensor(a, device="cuda") for a in (p, X, Y)))
    g = g.cpu().numpy().astype(np.float64)
    assert float(loss.item()) == pytest.approx(loss_ref, rel=2e-5)
    o = 0
    for name, shape in M.SHAPES:
        k = int(np.prod(shape))
        gr, gg = g_ref[o:o + k], g[o:o + k]
        bound = 2e-4 * (np.abs(gr) + 1e-2 * np.abs(gr).max())
        assert np.all(np.abs(gg - gr) <= bound), (name, float(np.max(np.abs(gg - gr) / bound)))
        o += k


@pytest.mark.parametrize("batch", [1, 100, 256 * 64 + 100])
def test_one_training_step_is_adam_on_the_mean_gradient(batch):
    """One step on n = 1 sample drawn `batch` times is the Adam step on that sample's gradient."""
    import torch
    rng = np.random.default_rng(batch)
    p = M.init_params(3).astype(np.float32)
    X, Y = rng.normal(size=(1, M.NIN)).astype(np.float32), rng.normal(size=(1, M.NOUT)).astype(np.float32)
    loss_ref, g = M.loss_and_grad(p.astype(np.float64), X.astype(np.float64), Y.astype(np.float64))
    d = {k: torch.tensor(a, device="cuda") for k, a in (("p", p), ("X", X), ("Y", Y))}
    work = torch.zeros(clv.MLP_TRAIN_WORK_FLOATS, device="cuda")
    loss = clv.mlp_train(d["p"], work, d["X"], d["Y"], 1, batch, 1e-3, 7)
    assert float(loss[0].item()) == pytest.approx(loss_ref, rel=2e-5)
    m = work[:clv.MLP_NPARAM].cpu().numpy()
    assert np.all(np.abs(m - 0.1 * g) <= 0.1 * 2e-4 * (np.abs(g) + 1e-2 * np.abs(g).max()))
