"""Inner solves of small batches (one launch of thread-block clusters), the sums over many work items, and link copies
that are filled again for new links.

A solve is right when every system's true residual, taken with the oracle's restricted operator (or the FP64 stencil,
which the oracle pins elsewhere) is at most the tolerance asked for: |b - D x| <= 1e-10 |b|, with 1e-7 of slack for the
rounding of the comparison itself.
"""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d, synth
from oracle.geometry import uniform_cores
from oracle.lattice import apply_D_restricted

from gpu_common import make_case, relerr, to_field

pytestmark = pytest.mark.gpu

TOL = 1e-10
CASES = {
    # framed blocks of 3^4: 41 and 40 sites per parity, so the second 32-site chunk is a remainder
    "4x4": ((4, 4, 4, 4), uniform_cores((4, 4, 4, 4), 1, 1)),
    # uneven blocks, one direction undecomposed
    "uneven": ((8, 6, 4, 4), [[(0, 2), (4, 6)], [(0, 1), (3, 4)], [(0, 0), (2, 2)], []]),
    "8x4": ((8, 8, 8, 8), uniform_cores((8, 8, 8, 8), 3, 1)),
}


@pytest.mark.parametrize("name,kind,nrhs,inner", [
    ("4x4", "omega", 1, "f32"), ("4x4", "omega", 3, "bf16"), ("4x4", "omega", 5, "f32"), ("4x4", "lambda1", 4, "f32"),
    ("uneven", "omega", 1, "f32"), ("uneven", "omega", 4, "bf16"), ("uneven", "omega", 7, "f32"),
    ("uneven", "lambda1", 3, "f32"), ("8x4", "omega", 13, "f32"), ("8x4", "lambda1", 2, "bf16"),
])
def test_one_launch_inner_solves(name, kind, nrhs, inner):
    L, cores = CASES[name]
    U, ctx, info, geo = make_case(L, 0.13, 0.4, 5, cores)
    ids = list(range(info["nblocks"])) if kind == "omega" else None
    sites = ([ctx.geom_sites(dd4d.SET_OMEGA, b) for b in ids] if ids is not None
             else [ctx.geom_sites(dd4d.SET_LAMBDA1)])
    masks = geo.omega_mask if ids is not None else [geo.Lambda1]
    sizes = [len(s) for s in sites]
    b = synth.complex_gaussian(7, synth.TAG_RHS, (sum(sizes) * nrhs * 12,))
    if nrhs > 2:
        b[12 * sizes[0]:24 * sizes[0]] = 0           # one system of the first block has nothing to solve
    x = np.zeros_like(b)
    prm = dd4d.params(TOL, inner_prec=inner, inner_tol=1e-3 if inner == "bf16" else 1e-5)
    st = ctx.solve_blocks(kind, ids, nrhs, b, x, prm)
    assert st["status"] == dd4d.DD_OK and st["max_relres"] <= TOL, st
    at = 0
    for k, n in enumerate(sizes):
        for r in range(nrhs):
            f, xf = to_field(L, sites[k], b[at:at + 12 * n]), to_field(L, sites[k], x[at:at + 12 * n])
            at += 12 * n
            res = f - apply_D_restricted(U, xf, 0.13, masks[k])
            assert np.linalg.norm(res) <= TOL * np.linalg.norm(f) * 1.0000001
    # the launched form on the same systems (a chosen launch variant takes it) agrees on the iterations to one or two
    y = np.zeros_like(b)
    ctx.set_hop_variant(inner, 0)
    s2 = ctx.solve_blocks(kind, ids, nrhs, b, y, prm)
    assert s2["status"] == dd4d.DD_OK and abs(s2["max_iters"] - st["max_iters"]) <= max(2, st["max_iters"] // 5)
    # both are within |D^-1| tol |b| of the solution; cond(D) < 100 here
    assert relerr(x, y) < 2 * 100 * TOL
    ctx.close()


@pytest.mark.parametrize("inner", ["f64", "f32"])
def test_sums_over_many_items(inner):
    """A frame of more than 32 work items of 128 sites (the sums run 32 items at a time)."""
    L = (12, 12, 12, 12)
    cores = uniform_cores(L, 4, 2)
    U, ctx, info, geo = make_case(L, 0.125, 0.4, 6, cores)
    n = len(ctx.geom_sites(dd4d.SET_LAMBDA1))
    assert n > 2 * 33 * 128
    b = synth.complex_gaussian(8, synth.TAG_RHS, (1, 2, n, 12))
    x, d = np.zeros_like(b), np.zeros_like(b)
    ctx.set_hop_variant("f32", 0)                    # the launched form
    st = ctx.solve_blocks("lambda1", None, 2, b, x, dd4d.params(TOL, inner_prec=inner))
    assert st["status"] == dd4d.DD_OK and st["max_relres"] <= TOL
    ctx.apply_D_block("lambda1", None, 2, x, d, "f64")
    for r in range(2):
        assert np.linalg.norm(b[0, r] - d[0, r]) <= TOL * np.linalg.norm(b[0, r]) * 1.0000001
    ctx.close()


def test_new_links_refill_every_copy():
    """Link copies keep their memory when the links change: results equal those of a context that never held others."""
    L = (4, 4, 4, 4)
    cores = uniform_cores(L, 1, 1)
    U1, old, info, _ = make_case(L, 0.13, 0.3, 1, cores)
    U2, new, _, _ = make_case(L, 0.13, 0.3, 2, cores)
    ids = list(range(info["nblocks"]))
    b = synth.complex_gaussian(3, synth.TAG_RHS, (len(ids), 2, len(old.geom_sites(dd4d.SET_OMEGA, 0)), 12))

    def results(ctx):
        out = []
        for prec in ("f64", "f32", "bf16"):
            d, x = np.zeros_like(b), np.zeros_like(b)
            ctx.apply_D_block("omega", ids, 2, b, d, prec)
            st = ctx.solve_blocks("omega", ids, 2, b, x, dd4d.params(TOL, inner_prec=prec, inner_tol=1e-3))
            assert st["status"] == dd4d.DD_OK
            out += [d, x]
        return out

    first = results(old)
    old.gauge_upload(U2)
    for a, c, f in zip(results(old), results(new), first):
        assert np.array_equal(a, c) and not np.array_equal(a, f)
    old.close()
    new.close()
