"""dd_fp64_fma_rate is a ceiling: the force kernel, bound by the same pipes, does not issue FP64 instructions faster."""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d

pytestmark = pytest.mark.gpu


def test_force_kernel_stays_below_the_probe():
    torch = pytest.importorskip("torch")
    L, nf = (24,) * 4, 12
    ctx = dd4d.Context(L, 0.13)
    ctx.gauge_random(0.4, 2)
    info = ctx.set_geometry([[(0, 6), (8, 14), (16, 22)]] * 4)
    chi = torch.ones((nf, info["n_dpi"], 24), dtype=torch.float64, device="cuda")
    F = torch.zeros(24 ** 4 * 32, dtype=torch.float64, device="cuda")
    best = 0.0
    for _ in range(3):
        ctx.timing_enable(True)
        ctx.mb_force(np.full(nf, 0.3 + 0.2j), chi, F, dd4d.params(1e-10, inner_prec="f32"))
        ms, launches, flops = ctx.timing_get(3)
        assert launches == 1 and flops == 576.0 * nf * 4 * 81 * 6 * 7 ** 3     # active links of 81 cores of 7^4
        best = max(best, flops / 576 * 336 / (ms * 1e-3))       # 288 FMAs and 48 additions per link and field
    rate = dd4d.fp64_fma_rate() * 1e12 / 2
    # event times of a kernel of 4.5 ms and clocks a moment apart: 2 %
    assert best <= 1.02 * rate, (best, rate)
    assert best >= 0.5 * rate
    ctx.close()
