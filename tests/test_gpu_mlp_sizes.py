"""The warm-start network's loss and gradients at the edges of its tiles (16 rows, 8 and 32
columns, 8 steps of 16): one sample, one input, one output, widths just past a tile.
Tolerances as for the full-size network: BF16 operands against an oracle that rounds at the
same places (loss 1e-3, gradients 5e-3 of their largest component)."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2311_01242_gb300.mlp import WarmStartMLP, init_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_in,hidden,n_out", [(1, 1, 16, 1), (16, 16, 16, 8), (17, 17, 48, 33), (129, 4, 144, 40),
                                                 (256, 33, 256, 512), (9, 16, 128, 97)])
def test_loss_and_gradient(B, n_in, hidden, n_out):
    rng = np.random.default_rng(B)
    p = init_params(n_in, hidden, n_out, seed=1)
    x = rng.normal(size=(B, n_in)).astype(np.float32)
    t = rng.normal(size=(B, n_out)).astype(np.float32)
    net = WarmStartMLP(n_in, hidden, n_out, params=p)
    loss = float(net.loss_grad(torch.as_tensor(x).cuda(), torch.as_tensor(t).cuda())[0])
    g = net.grads.cpu().numpy()
    loss_o, g_o = omlp.loss_grad(p.astype(np.float64), x.astype(np.float64), t.astype(np.float64), n_in, hidden, n_out)
    assert abs(loss - loss_o) <= 1e-3 * abs(loss_o)
    for name, (o, shp) in omlp.layout(n_in, hidden, n_out)[0].items():
        n = int(np.prod(shp))
        a, b = g[o:o + n].astype(np.float64), g_o[o:o + n]
        assert np.abs(a - b).max() <= 5e-3 * max(np.abs(b).max(), 1e-300), name
    y = net.forward(x).cpu().numpy()
    y_o, _ = omlp.forward(p.astype(np.float64), x.astype(np.float64), n_in, hidden, n_out)
    assert np.abs(y - y_o).max() <= 1e-3 * np.abs(y_o).max()
