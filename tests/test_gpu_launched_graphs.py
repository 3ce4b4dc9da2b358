"""The graphs of the launched inner solves at FP32 and BF16: captured iterations, the device-side loop, the whole solve.

Small batches solve their inner systems in one launch, unless a launch variant is chosen.  Here one is, on a batch of
uneven blocks, so that the graphs hold the launched iterations that every larger batch runs; the launch count shows it
(nine kernels an iteration).
"""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d, synth

from gpu_common import make_case

pytestmark = pytest.mark.gpu


def _case(inner):
    L = (12, 8, 8, 10)
    cores = [[(0, 3), (6, 8)], [(1, 2), (5, 6)], [(0, 4), (6, 6)], [(0, 2), (4, 7)]]
    _, ctx, info, _ = make_case(L, 0.12, 0.5, 7, cores)
    ctx.set_hop_variant(inner, 0)
    ids = list(range(info["nblocks"]))
    tot = sum(len(ctx.geom_sites(dd4d.SET_OMEGA, b)) for b in ids)
    return ctx, ids, synth.complex_gaussian(13, synth.TAG_RHS, (2 * tot, 12))


def _solve(ctx, ids, b, inner, itol, launched=True, **flags):
    x = np.zeros_like(b)
    n0 = dd4d.launch_count()
    st = ctx.solve_blocks("omega", ids, 2, b, x, dd4d.params(1e-10, inner_prec=inner, inner_tol=itol, **flags))
    n = dd4d.launch_count() - n0
    assert st["status"] == 0 and st["max_relres"] <= 1e-10
    assert (n >= 9 * st["max_iters"]) == launched, (n, st["max_iters"])
    return x, st


@pytest.mark.parametrize("flag", ["graph", "graph_loop", "graph_solve"])
@pytest.mark.parametrize("inner,itol", [("f32", 3e-6), ("f32", 1e-3), ("f32", 3e-3), ("bf16", 1e-3)])
def test_graphs_of_launched_inner_solves_are_bit_identical(flag, inner, itol):
    """The second solve replays the graph; the tolerances reach the updated residual and its verification."""
    ctx, ids, b = _case(inner)
    x0, s0 = _solve(ctx, ids, b, inner, itol)
    x1, s1 = _solve(ctx, ids, b, inner, itol, **{flag: True})
    x2, s2 = _solve(ctx, ids, b, inner, itol, **{flag: True})
    assert np.array_equal(x0, x1) and np.array_equal(x1, x2)
    assert s0["outer_cycles"] == s1["outer_cycles"] == s2["outer_cycles"]
    assert s0["max_iters"] == s1["max_iters"] == s2["max_iters"]
    ctx.close()


@pytest.mark.parametrize("inner", ["f32", "bf16"])
def test_without_a_chosen_variant_the_batch_takes_one_launch(inner):
    ctx, ids, b = _case(inner)
    x0, s0 = _solve(ctx, ids, b, inner, 1e-3)
    ctx.set_hop_variant(inner, -1)
    x1, s1 = _solve(ctx, ids, b, inner, 1e-3, launched=False)
    # both within cond(D) * tol of the solution; cond(D) < 100 at this kappa
    assert np.linalg.norm(x1 - x0) <= 2 * 100 * 1e-10 * np.linalg.norm(x0)
    ctx.close()


@pytest.mark.parametrize("cell,nrhs,kind,inner,one", [
    (4, 12, "omega", "f32", True), (8, 4, "omega", "f32", True), (6, 12, "lambda1", "f32", True), (10, 2, "omega", "f32", True),
    (10, 1, "omega", "f32", False), (10, 1, "omega", "bf16", False), (12, 1, "omega", "f32", False),
    (12, 1, "omega", "bf16", False), (9, 1, "omega", "bf16", False),
])
def test_form_of_small_batches(cell, nrhs, kind, inner, one):
    """Where the one launch was measured faster, with a margin, it is taken; where the launched form was, that is."""
    ctx = dd4d.Context((2 * cell,) * 4, 0.125)
    ctx.gauge_random(0.5, 2)
    info = ctx.set_geometry([[(0, cell - 2), (cell, 2 * cell - 2)]] * 4)
    ids = list(range(info["nblocks"])) if kind == "omega" else None
    n = info["nblocks"] * info["max_omega"] if ids else info["n_lambda1"]
    b = synth.complex_gaussian(3, synth.TAG_RHS, (n * nrhs, 12))
    x = np.zeros_like(b)
    for call in range(2):                            # the first also gathers the links
        n0 = dd4d.launch_count()
        st = ctx.solve_blocks(kind, ids, nrhs, b, x, dd4d.params(1e-8, inner_prec=inner, inner_tol=1e-3))
        n1 = dd4d.launch_count()
    assert st["status"] == 0 and (n1 - n0 < 9 * st["max_iters"]) == one, (n1 - n0, st["max_iters"])
    ctx.close()
