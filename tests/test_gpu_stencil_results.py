"""One answer of dd_apply_D_block: by the launch form a fresh batch takes, by a chosen one, after a tuned solve."""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d, synth
from oracle.geometry import uniform_cores

from gpu_common import make_case

pytestmark = pytest.mark.gpu


def _bf16(a):
    """a rounded to the nearest BF16 number, ties to even."""
    bits = a.astype(np.float32).view(np.uint32)
    return ((bits + 0x7fff + (bits >> 16 & 1)) & 0xffff0000).astype(np.uint32).view(np.float32).astype(np.float64)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_stencil_before_and_after_a_tuned_solve(prec, nrhs):
    """Framed blocks of 5^4 and 4^4 sites: items of 128 sites and remainders."""
    L = (8, 8, 8, 8)
    _, ctx, info, _ = make_case(L, 0.13, 0.4, 3, [[(0, 2), (4, 6)]] * 3 + [[(0, 2), (4, 5)]])
    ids = list(range(info["nblocks"]))
    n = sum(len(ctx.geom_sites(dd4d.SET_OMEGA, k)) for k in ids)
    psi = synth.complex_gaussian(5, synth.TAG_RHS, (n * nrhs, 12))
    fresh, chosen, tuned, x = (np.zeros_like(psi) for _ in range(4))
    ctx.apply_D_block("omega", ids, nrhs, psi, fresh, prec)
    ctx.set_hop_variant(prec, 0)
    ctx.apply_D_block("omega", ids, nrhs, psi, chosen, prec)
    ctx.set_hop_variant(prec, -1)
    ctx.solve_blocks("omega", ids, nrhs, psi, x, dd4d.params(1e-8, inner_prec=prec, inner_tol=1e-3, autotune=True))
    ctx.apply_D_block("omega", ids, nrhs, psi, tuned, prec)
    v = fresh.view(np.float64)
    if prec == "bf16":
        # the FP32 sums, not rounded to BF16; by a chosen variant they are
        assert np.array_equal(v, v.astype(np.float32)) and not np.array_equal(v, _bf16(v))
        assert np.array_equal(tuned, fresh) and np.array_equal(chosen.view(np.float64), _bf16(v))
    else:
        # the tuned variant may add the eight directions in another order: sums of 24 products and 17 terms
        assert np.array_equal(fresh, chosen)
        u = {"f64": 2.0 ** -53, "f32": 2.0 ** -24}[prec]
        assert np.abs(tuned - fresh).max() <= 64 * u * np.abs(fresh).max()
    ctx.close()


@pytest.mark.parametrize("nrhs,starts", [(5, "k_hop<"), (6, "k_hop_lb"), (7, "k_hop<"), (8, "k_hop_lb"), (9, "k_hop<"),
                                         (12, "k_hop_lb"), (13, "k_hop<"), (17, "k_hop<"), (18, "k_hop<")])
def test_default_form_of_large_batches(nrhs, starts):
    """Bundle CTAs have a warp per rhs; with 7 or 9 they leave much of an SM idle and the plain form is taken."""
    torch = pytest.importorskip("torch")
    ctx = dd4d.Context((24,) * 4, 0.12)
    ctx.gauge_random(0.4, 2)
    info = ctx.set_geometry([[(0, 6), (8, 14), (16, 22)]] * 4)
    ids = list(range(info["nblocks"]))
    gen = torch.Generator(device="cuda")
    gen.manual_seed(nrhs)
    b = torch.randn((len(ids), nrhs, info["max_omega"], 24), generator=gen, device="cuda", dtype=torch.float64)
    x = torch.zeros_like(b)
    st = ctx.solve_blocks("omega", ids, nrhs, b, x, dd4d.params(1e-6, inner_prec="f32", inner_tol=1e-3))
    assert st["status"] == 0 and st["max_relres"] <= 1e-6
    assert dd4d.hop_variant_name("f32", st["hop_variant"]).startswith(starts)
    ctx.close()
