"""Memory of the link copies and clover bundles: what is freed when the links or the term change, and allocations that
fail on the host (the test hook makes one act as if the device were out of memory)."""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d, synth
from oracle.geometry import uniform_cores

from gpu_common import make_case

pytestmark = pytest.mark.gpu

L = (8, 8, 8, 8)
CORES = uniform_cores(L, 3, 1)


def _free():
    torch = pytest.importorskip("torch")
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _blocks(ctx, info, nrhs=1):
    ids = list(range(info["nblocks"]))
    return ids, synth.complex_gaussian(3, synth.TAG_RHS, (len(ids), nrhs, info["max_omega"], 12))


def test_copies_that_are_not_used_any_more_are_freed():
    """FP64 and BF16 copies of 16 framed blocks of 9^4 sites go when the links have changed twice without their use."""
    big = (16, 16, 16, 16)
    U, ctx, info, _ = make_case(big, 0.13, 0.3, 1, uniform_cores(big, 7, 1))
    ids, psi = _blocks(ctx, info)
    out = np.zeros_like(psi)
    for prec in ("f64", "bf16", "f32"):
        ctx.apply_D_block("omega", ids, 1, psi, out, prec)
    held = _free()
    for _ in range(2):
        ctx.gauge_upload(U)
        ctx.apply_D_block("omega", ids, 1, psi, out, "f32")
    sites = 16 * 9 ** 4
    assert _free() - held >= 0.9 * 40 * sites * (16 + 4)       # 40 complex numbers a site in each
    ctx.close()


def test_clover_bundles_are_freed_with_the_term():
    big = (16, 16, 16, 16)
    U, ctx, info, _ = make_case(big, 0.13, 0.3, 1, uniform_cores(big, 7, 1))
    ids, b = _blocks(ctx, info)
    x = np.zeros_like(b)
    ctx.set_clover(1.0)
    ctx.solve_blocks("omega", ids, 1, b, x, dd4d.params(1e-10, inner_prec="f32"))
    held = _free()
    ctx.set_clover(0.0)
    assert _free() - held >= 0.9 * 16 * 9 ** 4 * 288
    with_term = x.copy()
    ctx.set_clover(1.0)
    ctx.solve_blocks("omega", ids, 1, b, x, dd4d.params(1e-10, inner_prec="f32"))
    assert np.array_equal(x, with_term)
    ctx.close()


def _results(ctx, ids, b, csw):
    out = []
    for prec in ("f64",) if csw else ("f64", "f32", "bf16"):
        out.append(np.zeros_like(b))
        ctx.apply_D_block("omega", ids, 2, b, out[-1], prec)
    for inner in ("f32", "bf16"):
        out.append(np.zeros_like(b))
        ctx.solve_blocks("omega", ids, 2, b, out[-1], dd4d.params(1e-10, inner_prec=inner, inner_tol=1e-3))
    return out


@pytest.mark.parametrize("csw", [0.0, 1.0])
def test_failed_allocations_free_stale_copies(csw):
    """After new links, each of the first allocations of a solve fails once in turn: the stale copies go, the
    allocation is tried again, and every result equals that of a context that never held others."""
    U1, old, info, _ = make_case(L, 0.13, 0.3, 1, CORES)
    U2, new, _, _ = make_case(L, 0.13, 0.3, 2, CORES)
    ids, b = _blocks(old, info, 2)
    x = np.zeros_like(b)
    for ctx in (old, new):
        ctx.set_clover(csw)
    want = _results(new, ids, b, csw)
    lam = synth.complex_gaussian(4, synth.TAG_RHS, (1, 1, info["n_lambda1"], 12))
    for k in range(1, 9):
        old.gauge_upload(U1)
        first = _results(old, ids, b, csw)
        old.gauge_upload(U2)
        old.debug_alloc_fault(k)
        # the frame's copies are not there yet the first time, later its workspaces are: allocations in any case
        old.solve_blocks("lambda1", None, 1, lam, np.zeros_like(lam), dd4d.params(1e-10, inner_prec="f32"))
        got = _results(old, ids, b, csw)
        old.debug_alloc_fault(0)
        for g, w, f in zip(got, want, first):
            assert np.array_equal(g, w) and not np.array_equal(g, f)
    old.close()
    new.close()


def test_failed_allocation_without_stale_copies_is_reported():
    U, ctx, info, _ = make_case(L, 0.13, 0.3, 1, CORES)
    ids, b = _blocks(ctx, info)
    x = np.zeros_like(b)
    ctx.debug_alloc_fault(3)
    with pytest.raises(dd4d.DDError) as e:
        ctx.solve_blocks("omega", ids, 1, b, x, dd4d.params(1e-10, inner_prec="f32"))
    assert e.value.status == dd4d.DD_ENOMEM
    st = ctx.solve_blocks("omega", ids, 1, b, x, dd4d.params(1e-10, inner_prec="f32"))
    assert st["status"] == 0 and st["max_relres"] <= 1e-10
    ctx.close()
