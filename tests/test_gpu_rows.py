"""Kernels that move rows between the caller's arrays and the padded ones: short rows
(several to a warp), long ones (in pieces), few and many; and that few long rows, or few
points with many partial gradients, do not wait on one warp."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _batch(laps, d, M, seed=0):
    x0 = np.random.default_rng(seed).standard_normal((M, d)).astype(np.float32)
    b = laps.Batch([W.Problem("p", W.GAUSS_DIAG, d, M, 10, x0, prec=np.ones(d))], n_total_steps=10)
    b.init(seed=1)
    return b, x0


@pytest.mark.parametrize("d,M", [(2, 2), (2, 70000), (3, 513), (4, 33), (5, 65536), (15, 1000), (16, 1001), (17, 100),
                                 (31, 9000), (32, 9), (33, 4095), (33, 4097), (127, 50), (128, 4096), (129, 3), (129, 2049),
                                 (1000, 511), (1000, 513), (10240, 2), (10240, 60)])
def test_samples_are_the_initial_positions(d, M):
    from paper_2601_16696_gb300 import laps
    b, x0 = _batch(laps, d, M)
    out = torch.full((M + 1, d), 7.0, device="cuda")  # the row after the last stays as it is
    b.sample(0, out[:M])
    np.testing.assert_array_equal(out[:M].cpu().numpy(), x0)
    assert (out[M] == 7.0).all()


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,d,M", [(2000, 2, 3), (2000, 3, 4200), (700, 31, 40), (700, 33, 4097), (1500, 127, 5),
                                   (1500, 128, 2100)])
def test_gradient_of_rows_alone_and_among_others(n, d, M, precision):
    """A point's gradient does not depend on where its row lies: the first, a middle and the last row of the call
    repeat in another order (the same data split: equal M)."""
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=n, n_feat=d - 1, M=M, data_seed=d)
    tg = laps.Target(laps.LOGREG, d, X=pr.X, y=pr.y)
    x = torch.tensor(pr.x0, dtype=torch.float32, device="cuda")
    perm = torch.randperm(M, generator=torch.Generator().manual_seed(1)).cuda()
    lp, g = tg.logp_grad(x, precision=precision)
    lp2, g2 = tg.logp_grad(x[perm], precision=precision)
    assert torch.equal(lp[perm], lp2) and torch.equal(g[perm], g2)
    z = pr.x0 @ pr.X.T
    g64 = (pr.y - 1.0 / (1.0 + np.exp(-z))) @ pr.X - pr.x0
    bar = {0: 1e-5, 1: 2e-2, 2: 1e-5}[precision]  # mixed: the data and residuals are rounded to BF16
    assert (np.abs(g.double().cpu().numpy() - g64).max(1) <= bar * np.abs(g64).max(1)).all()


def _us(fn, n=40):
    """Median of five blocks of n calls, microseconds a call."""
    for _ in range(3):
        fn()
    ts = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            fn()
        b.record()
        torch.cuda.synchronize()
        ts.append(1e3 * a.elapsed_time(b) / n)
    return sorted(ts)[2]


def test_few_long_rows_are_spread():
    """Two rows of 10000 take no longer than three times 200 rows of 100 (they took 4.8 times with a warp a row)."""
    from paper_2601_16696_gb300 import laps
    long, short = _batch(laps, 10000, 2)[0], _batch(laps, 100, 200)[0]
    o = torch.empty(2, 10000, device="cuda")
    p = torch.empty(200, 100, device="cuda")
    assert _us(lambda: long.sample(0, o)) <= 3.0 * _us(lambda: short.sample(0, p))


def test_few_points_are_spread():
    """Eight points of a three-term gradient with 157 partials take less than 1000 points (as long, 93 us, with a
    warp adding a row; about 40 against 63 us of launches otherwise)."""
    from paper_2601_16696_gb300 import laps
    pr = W.logreg(n_data=10000, n_feat=100, M=1)
    tg = laps.Target(laps.LOGREG, 101, X=pr.X, y=pr.y)
    x = torch.randn(1000, 101, device="cuda")
    few = x[:8].contiguous()
    assert _us(lambda: tg.logp_grad(few, precision=2)) <= 0.85 * _us(lambda: tg.logp_grad(x, precision=2))
