"""The dense-precision Gaussian's gradient where -P x cancels heavily.

The sums of P x run in a biased form that is repeated compensated for a chain
whose result is small against its bias.  Here every third chain sits in the
softest direction of a matrix of condition number 1e7 (those repeat), the
others do not, so warps with and without such chains, and mixed ones, occur.
Bar: the compensated dot product's bound u |r| + (d u)^2 |P| |x| (Ogita, Rump
and Oishi, 2005; u = 2^-24), twice it for the sums' own rounding."""
import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2601_16696_gb300 import laps
    laps.lib()
    return laps


def _problem(d, M, seed):
    rng = np.random.default_rng(seed)
    R, _ = np.linalg.qr(rng.standard_normal((d, d)))
    lam = np.logspace(-7, 0, d)
    P = (R / lam) @ R.T
    P = np.asarray(0.5 * (P + P.T), dtype=np.float32).astype(np.float64)
    soft = np.linalg.eigh(P)[1][:, 0]
    x = rng.standard_normal((M, d))
    x[::3] = soft * rng.uniform(0.5, 2.0, (len(x[::3]), 1))
    x[1] = 0.0
    x = np.asarray(x, dtype=np.float32).astype(np.float64)
    return W.Problem("soft_d%d" % d, W.GAUSS_DENSE, d, M, 50, x, prec=P)


def _check(pr, g):
    u = 2.0 ** -24
    ref = -pr.x0 @ pr.prec
    bar = 2.0 * (u * np.abs(ref) + (pr.d * u) ** 2 * (np.abs(pr.x0) @ np.abs(pr.prec)))
    # unflagged chains: the biased sums' share, 2^-25 of the largest result of the chain
    bar += 2.0 ** -25 * np.abs(ref).max(axis=1, keepdims=True)
    assert (np.abs(g.double().cpu().numpy() - ref) <= bar).all()


@pytest.mark.parametrize("d,M", [(7, 5), (32, 33), (61, 100), (100, 64), (128, 31), (300, 50), (511, 40), (512, 2)])
def test_target_gradient(L, d, M):
    pr = _problem(d, M, d + M)
    _, g = L.Target.from_problem(pr).logp_grad(torch.tensor(pr.x0, dtype=torch.float32, device="cuda"))
    _check(pr, g)


@pytest.mark.parametrize("d,M", [(7, 5), (32, 33), (61, 100), (100, 64), (100, 1000), (128, 31)])
def test_resident_gradient(L, d, M):
    """The gradient the register-resident kernel keeps after initialisation (x = 0 has no direction: left out)."""
    pr = _problem(d, M, d + M)
    pr.x0[1] = 1.0
    s = L.Sampler(L.Target.from_problem(pr), pr.M, n_total_steps=pr.n_steps)
    s.init(torch.tensor(pr.x0, dtype=torch.float32, device="cuda"), seed=1)
    assert s.launch_info()["resident"] == 1
    _check(pr, s.state()[2])
