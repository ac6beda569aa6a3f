"""The sampler's form of the packed FP32 gradient kernel, which runs when the grid
exceeds the SM count: bit for bit the plain kernel's gradient and log p (a sampler
of few chains runs that one), at the edges of its tiles and on logits near 0, where
the sigmoid's reciprocal is nearest a tie; and its steps against the oracle."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _init(laps, tg, x0, **cfg):
    s = laps.Sampler(tg, x0.shape[0], n_total_steps=50, **cfg)
    s.init(torch.tensor(x0, dtype=torch.float32, device="cuda"), seed=1)
    return s


def _near_ties(M, d):
    """Points whose logit is their last coordinate (the data's intercept), the multiples of 2^-26 up to 2^-21 either
    side of 0 in turn: there 1 + e^-|z| takes the values just below 2."""
    z = np.arange(-32, 33)[np.arange(M) % 65] * 2.0 ** -26
    return np.concatenate([np.zeros((M, d - 1)), z[:, None]], axis=1)


# one range of data rows (n <= 64) whatever the grid: 64 chains a block, more blocks than any GPU here has SMs
@pytest.mark.parametrize("points", ["normal", "ties"])
@pytest.mark.parametrize("n,d,M", [(64, 64, 64 * 200), (63, 65, 64 * 170 + 1), (1, 2, 64 * 190 - 1), (33, 128, 64 * 165 + 63),
                                   (50, 101, 64 * 200 + 17), (17, 30, 64 * 200)])
def test_packed_and_plain_kernels_agree(n, d, M, points):
    from paper_2601_16696_gb300 import laps
    assert (M + 63) // 64 > torch.cuda.get_device_properties(0).multi_processor_count
    pr = W.logreg(n_data=64, n_feat=d - 1, M=M, data_seed=n + d)
    x0 = pr.x0 if points == "normal" else _near_ties(M, d)
    tg = laps.Target(laps.LOGREG, d, X=pr.X[:n], y=pr.y[:n])
    big = _init(laps, tg, x0).state()
    for sl in (slice(0, 131), slice(M - 70, M)):
        small = _init(laps, tg, x0[sl]).state()
        for k in (2, 3):  # g and log p
            assert torch.equal(big[k][sl], small[k]), k


@pytest.mark.parametrize("n,d,M", [(1000, 101, 1500), (130, 60, 5000), (700, 128, 2111)])
def test_steps_of_a_large_grid(ora, n, d, M):
    """Grids of more blocks than SMs with several ranges of rows: fixed-step runs against the oracle, 1e-5."""
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=n, n_feat=d - 1, M=M, n_steps=50)
    s = _init(laps, laps.Target.from_problem(pr), pr.x0, fixed_eps=0.01)
    r = ora.OracleLAPS(ora.OracleTarget(pr.kind, pr.d, X=pr.X, y=pr.y, prior_var=pr.prior_var), pr.x0, seed=1,
                       n_total_steps=50, fixed_eps=0.01)
    for _ in range(3):
        s.step(1)
        r.iterate(1)
        x, xr = s.sample().double().cpu().numpy(), r.x()
        assert (np.linalg.norm(x - xr, axis=1) / np.linalg.norm(xr, axis=1)).max() <= 1e-5
