"""The packed FP32 gradient kernel at the edges of its tiles: 64 chains, 64 data
rows, features in steps of 4 up to the padded width, and the row ranges.  Bars of
the FP32 form: gradients within 1e-5 of max|g| per chain, log p within 2e-6."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,M", [(1, 2, 1), (63, 3, 63), (64, 4, 64), (65, 5, 65), (128, 63, 2), (129, 64, 129),
                                   (200, 65, 64), (999, 124, 130), (1000, 125, 7), (5000, 128, 200),
                                   # grids of more blocks than SMs, where the packed kernel runs
                                   (1000, 125, 641), (65, 64, 4990), (130, 3, 3300), (2, 2, 9800), (999, 128, 700),
                                   (64, 65, 9729), (190, 63, 3265)])
def test_gradient_at_tile_edges(ora, n, d, M):
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=max(n, 2), n_feat=d - 1, M=M, data_seed=n + d)
    X, y = pr.X[:n], pr.y[:n]
    tg = laps.Target(laps.LOGREG, d, X=X, y=y)
    lp, g = tg.logp_grad(torch.tensor(pr.x0, dtype=torch.float32, device="cuda"))
    lp_o, g_o = ora.OracleTarget(ora.LOGREG, d, X=X, y=y, prior_var=1.0).logp_grad(pr.x0)
    g = g.double().cpu().numpy()
    assert (np.abs(g - g_o).max(axis=1) <= 1e-5 * np.abs(g_o).max(axis=1)).all()
    np.testing.assert_allclose(lp.double().cpu().numpy(), lp_o, rtol=2e-6)
