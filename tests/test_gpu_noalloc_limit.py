"""laps_run_noalloc at the limit of its fixed scratch array: what fits with the fewest
blocks is run, also where the columns of the faster, spread launch shape (twice the blocks)
would not fit; what fits neither way is refused with the size it needs."""
import re

import numpy as np
import pytest
import torch

from paper_2601_16696_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SCRATCH = 16 << 20


def _columns(d_pad, G):
    return (4 * d_pad + 5) * 8 * G


def test_the_widest_window_that_fits_the_fewest_blocks_runs():
    from paper_2601_16696_gb300 import laps
    d, M = 400, 1000
    tg = laps.Target(laps.GAUSS_DIAG, d, prec=np.ones(d))
    shape = laps.Sampler(tg, M, n_total_steps=10).launch_info()
    few = dict(chains_per_block=512 // shape["lanes_per_chain"])  # the shape of the fewest blocks, asked for
    wide = laps.Sampler(tg, M, n_total_steps=10, **few).launch_info()
    assert shape["threads"] == 256 and wide["threads"] == 512 and shape["blocks"] == 2 * wide["blocks"] - 1
    extra = _columns(d, shape["blocks"]) - _columns(d, wide["blocks"])
    prec = torch.ones(d, device="cuda")
    x0 = torch.randn(M, d, generator=torch.Generator().manual_seed(1)).cuda()
    out = torch.empty(M, d, device="cuda")

    def run(T, **cfg):
        out.fill_(float("nan"))
        return laps.run_noalloc(laps.GAUSS_DIAG, d, M, x0, 3, out, prec=prec, n_total_steps=T, window_frac=1.0,
                                fixed_eps=0.05, **cfg)

    with pytest.raises(laps.LapsError) as e:  # far too large: the message states the need of this T
        run(20000, **few)
    need = int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))
    per_T = 8 * d
    T_wide = 20000 - (need - SCRATCH + per_T - 1) // per_T  # the largest T that fits with the fewest blocks
    assert extra > 20 * per_T
    for T in (T_wide - 1, T_wide):
        st = run(T)
        assert abs(st["t"] - T) < 15 and torch.isfinite(out).all()
    ref = laps.Sampler(tg, M, n_total_steps=T, window_frac=1.0, fixed_eps=0.05, **few)
    ref.init(x0, seed=3)
    ref.run()
    assert torch.equal(ref.sample(), out)
    with pytest.raises(laps.LapsError):
        run(T_wide + 2)
