"""The tensor-core gradients at the edges of their tiles: 128 chains, 64- and
128-row data chunks, K steps and N in 16 features; and labels other than 0 and 1,
which the BF16 form does not fold into its data.  Bars: BF16 form 4e-3 of max|g|
and 2e-5 of log p against the oracle on the rounded data (one BF16 rounding of each
residual); three-term form 1e-5 and 2e-6 against the data as given."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(1, 2, 1), (127, 15, 127), (128, 16, 128), (129, 17, 129), (63, 63, 5), (64, 64, 64), (65, 65, 2),
          (1000, 112, 130), (257, 113, 40), (2000, 128, 300)]


@pytest.mark.parametrize("labels", ["binary", "fractions"])
@pytest.mark.parametrize("n,d,M", SHAPES)
def test_gradient_at_tile_edges(ora, n, d, M, labels):
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=max(n, 2), n_feat=d - 1, M=M, data_seed=n + d)
    X, y = pr.X[:n], pr.y[:n]
    if labels == "fractions":
        y = np.asarray(np.random.default_rng(n).random(n), dtype=np.float32).astype(np.float64)
    tg = laps.Target(laps.LOGREG, d, X=X, y=y)
    x = torch.tensor(pr.x0, dtype=torch.float32, device="cuda")
    Xb = torch.from_numpy(np.asarray(X, dtype=np.float32)).to(torch.bfloat16).double().numpy()
    for precision, data, g_bar, lp_bar in ((laps.MIXED, Xb, 4e-3, 2e-5), (laps.BF16X3, X, 1e-5, 2e-6)):
        lp, g = tg.logp_grad(x, precision=precision)
        tg.check()
        lp_o, g_o = ora.OracleTarget(ora.LOGREG, d, X=data, y=y, prior_var=1.0).logp_grad(pr.x0)
        g = g.double().cpu().numpy()
        assert (np.abs(g - g_o).max(axis=1) <= g_bar * np.abs(g_o).max(axis=1)).all(), precision
        np.testing.assert_allclose(lp.double().cpu().numpy(), lp_o, rtol=lp_bar)
