"""The streamed path's chain updates in both forms (inputs loaded a chain ahead while the
blocks fit two to an SM, at their use beyond), with one, two and more partial gradients a
chain, and with fewer chains than warps: fixed-step runs against the oracle."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# FP32 partials: ranges of 64 rows, so n = 64 gives one, n = 128 two while they fill no further wave of blocks
@pytest.mark.parametrize("precision", [0, 2])
@pytest.mark.parametrize("n,d,M", [(64, 20, 5), (64, 5, 2500), (128, 20, 1201), (128, 100, 2500), (700, 20, 3000), (128, 20, 9728),
                                   (128, 20, 9729), (300, 65, 10001)])
def test_fixed_steps(ora, n, d, M, precision):
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=n, n_feat=d - 1, M=M, n_steps=50)
    s = laps.Sampler(laps.Target.from_problem(pr), M, n_total_steps=50, fixed_eps=0.01, precision=precision)
    s.init(torch.tensor(pr.x0, dtype=torch.float32, device="cuda"), seed=1)
    r = ora.OracleLAPS(ora.OracleTarget(pr.kind, pr.d, X=pr.X, y=pr.y, prior_var=pr.prior_var), pr.x0, seed=1,
                       n_total_steps=50, fixed_eps=0.01)
    for _ in range(3):
        s.step(1)
        r.iterate(1)
        x, xr = s.sample().double().cpu().numpy(), r.x()
        assert (np.linalg.norm(x - xr, axis=1) / np.linalg.norm(xr, axis=1)).max() <= 1e-5
