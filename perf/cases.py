"""Performance cases of the LAPS library: what its users have it do, through the public binding.

A user evaluates a target (its log density and gradient, alone or under autograd), runs one
ensemble (a register-resident target, the dense-precision Gaussian, or the streamed logistic
regression), or runs a batch of uneven problems in one launch.  The sizes are those of the
repository's workloads (``workloads.py``) and ragged ones around them.

The sampler cases hold the step size fixed (the configuration of the fixed-step ablation).  The
kernels and the work per iteration are those of an adaptive run; but the adaptive controller's
first update divides by an energy error near 1e-8, so that two correct binary32 runs leave each
other by 1e-4 within a few steps and their outputs could not be compared.
"""
import math

import numpy as np
import torch

from paper_2601_16696_gb300 import laps, workloads
from paper_2601_16696_gb300.autograd import target_logp

DEV = "cuda"
KINDS = {"gauss": laps.GAUSS_DIAG, "banana": laps.BANANA, "funnel": laps.FUNNEL, "dense": laps.GAUSS_DENSE,
         "logreg": laps.LOGREG}
PRECISIONS = {"fp32": laps.FP32, "mixed": laps.MIXED, "bf16x3": laps.BF16X3}
# step sizes of the targets' fixed-step runs (positions drawn as below), for d = 100
FIXED_EPS = {"gauss": 0.0625, "banana": 0.0625, "funnel": 0.0625, "dense": 0.001953125, "logreg": 0.0078125}
BATCH_EPS = 0.0625
# an adjusted case begins its bisection below the target acceptance's step: a chain whose test falls within
# rounding of its uniform is then rare, and outputs of correct runs stay comparable
ADJUSTED_EPS = 0.25


def listed():
    return [
        # log p of a handful of points with its gradient through torch.autograd: a user's own optimiser or
        # diagnostic around a built-in target; the smallest call, launches and host work
        {"name": "autograd_funnel_M256", "family": "autograd", "kind": "funnel", "d": 101, "M": 256},
        # the plain ensemble of the first workload (256 chains), a whole unadjusted run: every iteration is
        # latency, not work
        {"name": "gauss_M256_run", "family": "run", "kind": "gauss", "d": 100, "M": 256, "phase": "unadjusted",
         "steps": 1000, "K": 0},
        # the banana ensemble (4096 chains), unadjusted steps: the phase every run begins with
        {"name": "banana_M4096_unadjusted", "family": "run", "kind": "banana", "d": 100, "M": 4096,
         "phase": "unadjusted", "steps": 64, "K": 0},
        # the same ensemble in the Metropolis-adjusted phase (15-step proposals): most gradients of a run are here
        {"name": "banana_M4096_adjusted", "family": "run", "kind": "banana", "d": 100, "M": 4096,
         "phase": "adjusted", "steps": 4, "K": 0},
        # the rotated ill-conditioned Gaussian, register-resident: the dense precision matrix in shared memory
        {"name": "dense_d100_M4096", "family": "run", "kind": "dense", "d": 100, "M": 4096, "phase": "unadjusted",
         "steps": 16, "K": 0},
        # the same target beyond the resident kernel's dimension, a ragged size on the streamed path
        {"name": "dense_d300_M1500", "family": "run", "kind": "dense", "d": 300, "M": 1500, "phase": "unadjusted",
         "steps": 8, "K": 0},
        # the logistic regression's ensemble gradient in each arithmetic: the contraction a user's evaluation
        # (and each step of a run) consists of
        {"name": "logreg_grad_fp32", "family": "gradient", "n": 10000, "d": 101, "M": 8192, "precision": "fp32"},
        {"name": "logreg_grad_mixed", "family": "gradient", "n": 10000, "d": 101, "M": 8192, "precision": "mixed"},
        {"name": "logreg_grad_bf16x3", "family": "gradient", "n": 10000, "d": 101, "M": 8192, "precision": "bf16x3"},
        # a run of the logistic regression, mixed precision: gradient, chain updates and finalise per step
        {"name": "logreg_run_mixed", "family": "run", "kind": "logreg", "n": 10000, "d": 101, "M": 8192,
         "precision": "mixed", "phase": "unadjusted", "steps": 32, "K": 0},
        # many problems of uneven size and one of d = 10^4 in one launch: the batched workload, unadjusted steps
        {"name": "batch_uneven_unadjusted", "family": "batch", "shapes": 0, "n_small": 24, "big_d": 10000,
         "big_M": 4096, "phase": "unadjusted", "steps": 8},
        # a small batch in the adjusted phase (second- and fourth-order integrators side by side)
        {"name": "batch_small_adjusted", "family": "batch", "shapes": 1, "n_small": 8, "big_d": 0, "big_M": 0,
         "phase": "adjusted", "steps": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["autograd", "resident", "resident", "dense", "gradient", "gradient", "logreg", "batch"])
    if family == "autograd":
        kind = rng.choice(["gauss", "banana", "funnel"])
        d = _log_int(rng, 2, 400)
        return {"family": "autograd", "kind": kind, "d": d + d % 2 if kind == "banana" else d,
                "M": _log_int(rng, 1, 32768)}
    if family == "resident":
        kind = rng.choice(["gauss", "banana", "funnel"])
        d = _log_int(rng, 8, 400)
        d = d + d % 2 if kind == "banana" else d
        M = _log_int(rng, 32, 2000 if d > 128 else 4096)
        adjusted = rng.random() < 0.4
        K = rng.choice([0, 0, 0, 20]) if not adjusted and d <= 128 and M <= 2048 else 0
        return {"family": "run", "kind": kind, "d": d, "M": M, "phase": "adjusted" if adjusted else "unadjusted",
                "steps": rng.randint(2, 4) if adjusted else rng.randint(16, 64), "K": K}
    if family == "dense":
        d = _log_int(rng, 16, 400)
        return {"family": "run", "kind": "dense", "d": d, "M": _log_int(rng, 32, 4000 if d <= 128 else 1500),
                "phase": "unadjusted", "steps": rng.randint(4, 12), "K": 0}
    if family == "gradient":
        precision = rng.choice(["fp32", "mixed", "bf16x3"])
        return {"family": "gradient", "n": _log_int(rng, 64, 10000),
                "d": _log_int(rng, 4, 200 if precision == "fp32" else 128), "M": _log_int(rng, 16, 8192),
                "precision": precision}
    if family == "logreg":
        return {"family": "run", "kind": "logreg", "n": _log_int(rng, 200, 10000), "d": _log_int(rng, 8, 128),
                "M": _log_int(rng, 64, 8192), "precision": rng.choice(["fp32", "mixed", "bf16x3"]),
                "phase": "unadjusted", "steps": rng.randint(4, 16), "K": 0}
    adjusted = rng.random() < 0.4
    big = not adjusted and rng.random() < 0.5
    return {"family": "batch", "shapes": rng.randint(2, 9999), "n_small": rng.randint(2, 8 if adjusted else 24),
            "big_d": _log_int(rng, 2000, 10000) if big else 0, "big_M": _log_int(rng, 64, 4096) if big else 0,
            "phase": "adjusted" if adjusted else "unadjusted", "steps": rng.randint(2, 3) if adjusted else rng.randint(2, 8)}


# ---------------------------------------------------------------- inputs
def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + 17)


def _target_data(case, seed):
    """The target's parameters: {"prec"} or {"X", "y"} (numpy, binary32 values)."""
    if case["family"] == "gradient" or case["kind"] == "logreg":
        pr = workloads.logreg(n_data=case["n"], n_feat=case["d"] - 1, M=1, data_seed=seed)
        return {"X": pr.X, "y": pr.y}
    if case["kind"] == "dense":
        return {"prec": workloads.icg(d=case["d"], M=1, seed=seed).prec}
    if case["kind"] == "gauss":
        # variances log-spaced over 1e-2 .. 1e2, in another order for each seed
        pr = workloads.gauss_diag(d=case["d"], M=1)
        return {"prec": np.random.default_rng(seed).permutation(pr.prec)}
    return {}


def _positions(case, seed, data):
    """Initial positions N(0, I), or the cold start 3 N(0, I) of the diagonal Gaussian.  The adjusted phase
    begins near equilibrium (the unadjusted phase precedes it): exact draws of the target."""
    z = torch.randn(case["M"], case["d"], generator=_rng(seed), device=DEV)
    if case.get("phase") != "adjusted":
        return 3.0 * z if case.get("kind") == "gauss" else z
    if case["kind"] == "gauss":
        return z / torch.tensor(data["prec"], device=DEV).sqrt().float()
    if case["kind"] == "banana":
        z[:, 1::2] = z[:, 0::2] ** 2 + 0.1 * z[:, 1::2]
        return z
    z[:, 0] *= 3.0  # the funnel: v ~ N(0, 9), x_i | v ~ N(0, e^v)
    z[:, 1:] *= torch.exp(0.5 * z[:, :1])
    return z


def _eps(case):
    """The fixed step size: |u| = 1, so a step moves a coordinate by about eps / sqrt(d)."""
    e = FIXED_EPS[case["kind"]] * math.sqrt(case["d"] / 100.0)
    return float(np.float32(e * ADJUSTED_EPS if case["phase"] == "adjusted" else e))


def _batch_problems(case, seed):
    """[(d, M, prec)]: shapes of the batched workload, each problem's variances in a seeded order.  The library
    draws the initial positions, or (adjusted phase, as above) the caller passes draws of each target."""
    out = []
    rng = np.random.default_rng(seed)
    shapes = [(d, k, M) for d, k, M in workloads.batch64_shapes(case["shapes"], case["n_small"])]
    if case["phase"] == "adjusted":
        # a proposal is 15 steps of two or five gradients: fewer chains for about the same work
        shapes = [(d, k, min(M, 512)) for d, k, M in shapes]
    if case["big_d"]:
        shapes.append((case["big_d"], 1e4, case["big_M"]))
    for d, kappa, M in shapes:
        var = kappa ** (np.arange(d) / max(d - 1, 1) - 0.5)
        out.append((d, M, rng.permutation((1.0 / var).astype(np.float32).astype(np.float64))))
    return out


def _batch_eps(case):
    return BATCH_EPS * ADJUSTED_EPS if case["phase"] == "adjusted" else BATCH_EPS


def _batch_positions(case, seed):
    """The problems' initial positions, adjusted phase (None: the library draws them)."""
    if case["phase"] != "adjusted":
        return None
    rng = _rng(seed)
    return [torch.randn(M, d, generator=rng, device=DEV) / torch.tensor(prec, device=DEV).sqrt().float()
            for d, M, prec in _batch_problems(case, seed)]


def prepare(case, seed):
    family = case["family"]
    state = {"family": family, "seed": int(seed)}
    if family == "batch":
        x0 = _batch_positions(case, seed)
        probs = [workloads.Problem("p%d" % k, laps.GAUSS_DIAG, d, M, 2000, x0[k] if x0 else None, prec=prec)
                 for k, (d, M, prec) in enumerate(_batch_problems(case, seed))]
        state["batch"] = laps.Batch(probs, use_x0=x0 is not None, n_total_steps=2000, fixed_eps=_batch_eps(case),
                                    force_switch_at=1 if case["phase"] == "adjusted" else 0)
        state["steps"] = case["steps"]
        return state
    kind = "logreg" if family == "gradient" else case["kind"]
    data = _target_data(case, seed)
    state["target"] = laps.Target(KINDS[kind], case["d"], **data)
    x0 = _positions(case, seed, data)
    if family == "autograd":
        state["x"] = x0.requires_grad_(True)
        return state
    state["x"] = x0
    if family == "gradient":
        state["precision"] = PRECISIONS[case["precision"]]
        return state
    more = {"precision": PRECISIONS[case["precision"]]} if kind == "logreg" else {}
    state["sampler"] = laps.Sampler(state["target"], case["M"], n_total_steps=2000, fixed_eps=_eps(case),
                                    force_switch_at=1 if case["phase"] == "adjusted" else 0, dtilde_K=case["K"], **more)
    state["steps"] = case["steps"]
    return state


def run(state):
    family = state["family"]
    if family == "autograd":
        logp = target_logp(state["x"], state["target"])
        (grad,) = torch.autograd.grad(logp.sum(), state["x"])
        return [logp.detach(), grad]
    if family == "gradient":
        return list(state["target"].logp_grad(state["x"], precision=state["precision"]))
    if family == "batch":
        b = state["batch"]
        b.init(seed=state["seed"])
        b.step(state["steps"])
        return [b.sample(k) for k in range(b.n)]
    s = state["sampler"]
    s.init(state["x"], seed=state["seed"])
    s.step(state["steps"])
    return list(s.state())


# ---------------------------------------------------------------- work
STEP_OPS = {"unadjusted": 113, "mn2": 122, "mn4": 155}  # arithmetic operations per coordinate and step: the noise of
# two O maps, the B and A maps with a diagonal target, the ensemble's sums


def _grads(case, d):
    """(steps, gradients) one pass takes per chain."""
    if case["phase"] == "unadjusted":
        return case["steps"], case["steps"] + 1
    n = 15 * (case["steps"] - 1)
    return 1 + n, 2 + n * (5 if d > 200 else 2)


def _steps_flops(case, M, d):
    steps, _ = _grads(case, d)
    if case["phase"] == "unadjusted":
        return STEP_OPS["unadjusted"] * M * d * steps
    return M * d * (STEP_OPS["unadjusted"] + (steps - 1) * STEP_OPS["mn4" if d > 200 else "mn2"])


def work(case):
    family = case["family"]
    if family == "batch":
        flops = nbytes = 0
        for d, M, _ in _batch_problems(case, 0):
            flops += _steps_flops(case, M, d)
            nbytes += 4 * d + 4 * M * d * (2 if case["phase"] == "adjusted" else 1)
        return {"bytes": nbytes, "flops": flops}
    M, d = case["M"], case["d"]
    if family == "autograd":
        return {"bytes": 4 * M * (2 * d + 1), "flops": 6 * M * d}
    if family == "gradient":
        n = case["n"]
        return {"bytes": 4 * (n * d + n + 2 * M * d + M), "flops": 4 * M * n * d + 12 * M * n}
    _, grads = _grads(case, d)
    flops = _steps_flops(case, M, d)
    data = 0
    if case["kind"] == "logreg":
        flops += grads * (4 * M * case["n"] * d + 12 * M * case["n"])
        data = 4 * case["n"] * (d + 1)
    elif case["kind"] == "dense":
        flops += grads * 2 * M * d * d
        data = 4 * d * d
    elif case["K"]:
        flops += case["steps"] * 4 * M * d * case["K"]
    return {"bytes": data + 4 * M * d * 4 + 8 * M + 4 * d, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
M32 = 0xFFFFFFFF


def _philox(j, m, t, tag, seed):
    """Philox4x32-10 (Salmon et al., 2011) on broadcast int64 tensors, counter (j, m, t, tag)."""
    c = [v.to(torch.int64) if isinstance(v, torch.Tensor) else torch.full((), v, dtype=torch.int64, device=DEV)
         for v in (j, m, t, tag)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c


def _uniform(r):
    return ((r >> 9).double() + 0.5) * 2.0 ** -23


def _normals(M, d, t, tag, pid, seed):
    """Box-Muller normals of coordinates 4j .. 4j + 3 from one counter, chains 0 .. M - 1."""
    nblk = (d + 3) // 4
    j = torch.arange(nblk, device=DEV)[None, :]
    m = torch.arange(M, device=DEV)[:, None]
    r = [v.expand(M, nblk) for v in _philox(j, m, t, tag | (pid << 8), seed)]
    z = torch.empty(M, nblk, 4, dtype=torch.float64, device=DEV)
    for h in range(2):
        rad = torch.sqrt(-2.0 * torch.log(_uniform(r[2 * h])))
        ang = 2.0 * math.pi * _uniform(r[2 * h + 1])
        z[:, :, 2 * h], z[:, :, 2 * h + 1] = rad * torch.cos(ang), rad * torch.sin(ang)
    return z.view(M, 4 * nblk)[:, :d]


def _logp_grad64(kind, x, data):
    if kind == "gauss":
        g = -data["prec"] * x
        return 0.5 * (g * x).sum(1), g
    if kind == "dense":
        g = -(x @ data["prec"])
        return 0.5 * (g * x).sum(1), g
    if kind == "banana":
        a, b = x[:, 0::2], x[:, 1::2]
        r = (b - a * a) / 0.01
        g = torch.empty_like(x)
        g[:, 0::2], g[:, 1::2] = 2.0 * a * r - a, -r
        return (-0.5 * a * a - 0.5 * (b - a * a) * r).sum(1), g
    if kind == "funnel":
        v, w = x[:, :1], x[:, 1:]
        n, ev, ss = x.shape[1] - 1, torch.exp(-v), (w * w).sum(1, keepdim=True)
        lp = -0.5 * v * v / 9.0 - 0.5 * n * v - 0.5 * ev * ss
        return lp[:, 0], torch.cat([-v / 9.0 - 0.5 * n + 0.5 * ev * ss, -w * ev], 1)
    X, y = data["X"], data["y"]
    lp = -0.5 * (x * x).sum(1)
    g = -x
    for a in range(0, x.shape[0], 1024):
        z = x[a:a + 1024] @ X.T
        lp[a:a + 1024] += (y * z - torch.nn.functional.softplus(z, threshold=700.0)).sum(1)
        g[a:a + 1024] += (y - torch.sigmoid(z)) @ X
    return lp, g


TABLES = {"lf": ([0.5, 0.5], [1.0]),
          "mn2": ([0.1931833275, 1.0 - 2 * 0.1931833275, 0.1931833275], [0.5, 0.5])}
_B1, _B2, _A1, _A2 = 0.0839831526, 0.6822365335, 0.2539785108, -0.032302867
_B3, _A3 = 0.5 - _B1 - _B2, 1.0 - 2 * (_A1 + _A2)
TABLES["mn4"] = ([_B1, _B2, _B3, _B3, _B2, _B1], [_A1, _A2, _A3, _A2, _A1])


class _Run64:
    """The fixed-step LAPS run of one problem in binary64 (Algorithm 1 of the paper)."""

    def __init__(self, kind, data, x0, eps, seed, pid, switch):
        self.kind, self.data, self.seed, self.pid, self.switch = kind, data, seed, pid, switch
        self.M, self.d = x0.shape
        self.sigma = torch.ones(self.d, dtype=torch.float64, device=DEV)
        self.y, self.eps, self.t, self.p, self.phase = x0, eps, 0, 0, 0
        self.lp, self.g = self._target(self.y)
        self.u = self.g / self.g.norm(dim=1, keepdim=True)
        self.L = 2.0 * torch.sqrt(self.y.var(0, unbiased=False).sum()).item()
        self.lo = self.hi = 0.0
        self.adapting = True

    def _target(self, y):
        lp, g = _logp_grad64(self.kind, y * self.sigma, self.data)
        return lp, g * self.sigma

    def _noise(self, t, tag):
        return _normals(self.M, self.d, t, tag, self.pid, self.seed)

    def _o(self, u, t, tag):
        c1 = math.exp(-0.5 * self.eps / self.L)
        u = c1 * u + math.sqrt(1.0 - c1 * c1) / math.sqrt(self.d) * self._noise(t, tag)
        return u / u.norm(dim=1, keepdim=True)

    def _b(self, u, g, be):
        gn = g.norm(dim=1, keepdim=True)
        e = g / gn
        eu = (e * u).sum(1, keepdim=True)
        dl = be * gn / (self.d - 1)
        ze = torch.exp(-dl)
        den = (1 + ze * ze) + eu * (1 - ze * ze)
        kin = (self.d - 1) * (dl + torch.log(0.5 * den))
        return (2 * ze * u + (1 - ze) * ((1 + ze) + eu * (1 - ze)) * e) / den, kin[:, 0]

    def _steps(self, y, u, g, lp, table, n, t0):
        b, a = TABLES[table]
        delta = torch.zeros(self.M, dtype=torch.float64, device=DEV)
        for k in range(n):
            u = self._o(u, t0 + k, 1)
            for s, bs in enumerate(b):
                u, kin = self._b(u, g, bs * self.eps)
                delta += kin
                if s < len(a):
                    y = y + a[s] * self.eps * u
                    old = lp
                    lp, g = self._target(y)
                    delta += old - lp
            u = self._o(u, t0 + k, 2)
        return y, u, g, lp, delta

    def step(self):
        if self.phase == 0:
            self.y, self.u, self.g, self.lp, _ = self._steps(self.y, self.u, self.g, self.lp, "lf", 1, self.t)
            self.t += 1
            var = self.y.var(0, unbiased=False)
            self.L = 2.0 * torch.sqrt(var.sum()).item()
            if self.switch and self.t >= self.switch:
                self.phase, self.sigma = 1, torch.sqrt(var)
                self.eps *= math.sqrt(self.d / var.sum().item())
                self.L = 1.25 * 15 * self.eps
                self.y, self.g = self.y / self.sigma, self.g * self.sigma
            return
        z = self._noise(self.p, 3)
        table, target = ("mn4", 0.9) if self.d > 200 else ("mn2", 0.7)
        y, u, g, lp, delta = self._steps(self.y, z / z.norm(dim=1, keepdim=True), self.g, self.lp, table, 15, self.t)
        r = _philox(0, torch.arange(self.M, device=DEV), self.p, 4 | (self.pid << 8), self.seed)[0]
        keep = (delta + torch.log(_uniform(r)) < 0)[:, None]
        self.y, self.u, self.g = (torch.where(keep, n, o) for n, o in ((y, self.y), (u, self.u), (g, self.g)))
        self.lp = torch.where(keep[:, 0], lp, self.lp)
        acc = torch.exp(-delta.clamp(min=0)).mean().item()
        self.adapting = self.adapting and abs(acc - target) > 0.03
        if self.adapting and acc > target:
            self.lo, self.eps = self.eps, 0.5 * (self.eps + self.hi) if self.hi > 0 else 2.0 * self.eps
        elif self.adapting:
            self.hi, self.eps = self.eps, 0.5 * (self.eps + self.lo) if self.lo > 0 else 0.5 * self.eps
        self.L = 1.25 * 15 * self.eps
        self.t, self.p = self.t + 15, self.p + 1


def exact(case, seed):
    family, seed = case["family"], int(seed)
    switch = 1 if case.get("phase") == "adjusted" else 0
    if family == "batch":
        out, x0 = [], _batch_positions(case, seed)
        for k, (d, M, prec) in enumerate(_batch_problems(case, seed)):
            r = _Run64("gauss", {"prec": torch.tensor(prec, device=DEV)},
                       x0[k].double() if x0 else _normals(M, d, 0, 0, k, seed).clone(), _batch_eps(case), seed, k, switch)
            for _ in range(case["steps"]):
                r.step()
            out.append(r.y * r.sigma)
        return out
    data = _target_data(case, seed)
    x = _positions(case, seed, data).double()
    data = {k: torch.tensor(v, dtype=torch.float64, device=DEV) for k, v in data.items()}
    if family in ("autograd", "gradient"):
        return list(_logp_grad64("logreg" if family == "gradient" else case["kind"], x, data))
    r = _Run64(case["kind"], data, x, _eps(case), seed, 0, switch)
    for _ in range(case["steps"]):
        r.step()
    return [r.y, r.u, r.g, r.lp, r.sigma]
