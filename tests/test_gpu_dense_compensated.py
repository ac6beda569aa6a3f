"""The dense-precision Gaussian's gradient is the compensated dot product (Ogita,
Rump and Oishi, 2005) of every column, each component as accurate as one in twice
binary32: bit for bit the binary32 operations below, whatever the scales of the
rows of P, the size of a component next to its chain's largest, or the neighbours
of a chain."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu
F = np.float32


def _rotated(rng, d, cond):
    R, _ = np.linalg.qr(rng.standard_normal((d, d)))
    P = (R * np.logspace(0, np.log10(cond), d)) @ R.T
    return 0.5 * (P + P.T), R


def _problem(kind, d, M, seed):
    """(P, x): binary32 values in binary64, P symmetric."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((M, d))
    if kind == "scales":  # two blocks of condition 1e5, twenty decades apart
        P = np.zeros((d, d))
        h = d // 2
        P[:h, :h] = 1e20 * _rotated(rng, h, 1e5)[0]
        P[h:, h:] = _rotated(rng, d - h, 1e5)[0]
    elif kind == "tiny":  # rows whose squares underflow beside ordinary ones
        P, _ = _rotated(rng, d, 1e5)
        s = np.where(np.arange(d) < d // 2, 1e-12, 1.0)
        P = P * s[:, None] * s
    elif kind == "large":  # products near the top of the range
        P = np.diag(np.where(np.arange(d) % 2 == 0, 1e19, 1.0))
        x = np.where(rng.random((M, d)) < 0.5, -1e19, 1e19) * rng.uniform(0.5, 1.0, (M, d))
    else:  # equilibrium draws of a rotated spectrum: every component cancels
        cond = float(kind)
        P, R = _rotated(rng, d, cond)
        x = (x / np.sqrt(np.logspace(0, np.log10(cond), d))) @ R.T
        x[0] = 0.0 if M > 3 else x[0]
    return np.asarray(P, dtype=F).astype(np.float64), np.asarray(x, dtype=F).astype(np.float64)


def _compensated(P, x, device="cuda"):
    """-P x: x p = pr + er exactly, (hi, e) = TwoSum(hi, pr), lo += e + er, hi + lo at the end
    (separate binary32 operations, products exact in binary64)."""
    P, x = torch.tensor(P, device=device), torch.tensor(x, device=device)
    hi = torch.zeros(x.shape, dtype=torch.float32, device=device)
    lo = torch.zeros_like(hi)
    for j in range(x.shape[1]):
        prod = x[:, j:j + 1] * P[j]
        pr = prod.float()
        er = (prod - pr.double()).float()
        s = hi + pr
        bp = s - hi
        e = (hi - (s - bp)) + (pr - bp)
        hi, lo = s, lo + (e + er)
    return -(hi + lo).cpu().numpy()


KINDS = ["1e5", "1e8", "scales", "tiny", "large"]


# the ensemble's sizes reach one, two and four chains a warp and several waves of them on 152 SMs
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("d,M", [(2, 3), (7, 5), (33, 160), (61, 2500), (100, 64), (100, 5000), (129, 2433), (256, 5200),
                                 (300, 50), (320, 2600), (511, 40), (512, 2)])
def test_target_gradient_bits(kind, d, M):
    from paper_2601_16696_gb300 import laps
    P, x = _problem(kind, d, M, d + M)
    tg = laps.Target(laps.GAUSS_DENSE, d, prec=P)
    lp, g = tg.logp_grad(torch.tensor(x, dtype=torch.float32, device="cuda"))
    ref = _compensated(P, x)
    np.testing.assert_array_equal(g.cpu().numpy(), ref)
    # log p sums x_i r_i the same way: binary32's unit of the result and of the terms' absolute sum, twice binary32
    if kind != "large":
        t = 0.5 * x * ref.astype(np.float64)
        bar = 2.0 ** -23 * np.abs(t.sum(1)) + 2.0 ** -44 * d * np.abs(t).sum(1)
        assert (np.abs(lp.double().cpu().numpy() - t.sum(1)) <= bar).all()


@pytest.mark.parametrize("kind", KINDS[:4])
@pytest.mark.parametrize("d,M", [(2, 3), (7, 5), (33, 160), (61, 100), (100, 64), (100, 1000), (100, 4096), (128, 31)])
def test_resident_gradient_bits(kind, d, M):
    """The gradient the register-resident kernel keeps after initialisation (sigma = 1)."""
    from paper_2601_16696_gb300 import laps
    P, x = _problem(kind, d, M, d + M)
    x[0] = 1.0  # x = 0 has no direction
    s = laps.Sampler(laps.Target(laps.GAUSS_DENSE, d, prec=P), M, n_total_steps=50)
    s.init(torch.tensor(x, dtype=torch.float32, device="cuda"), seed=1)
    assert s.launch_info()["resident"] == 1
    np.testing.assert_array_equal(s.state()[2].cpu().numpy(), _compensated(P, x))
