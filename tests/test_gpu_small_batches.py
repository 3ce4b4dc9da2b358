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


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_stencil_of_many_units_equals_one_rhs_at_a_time(prec):
    """Whole items per CTA (more than 16 units per SM) and 32 sites per CTA do the same arithmetic on every site."""
    L = (4, 4, 4, 4)
    U, ctx, info, _ = make_case(L, 0.13, 0.4, 9, uniform_cores(L, 1, 1))
    ids, R = list(range(info["nblocks"])), 176       # 16 blocks x 176 rhs of one item per parity
    n = len(ctx.geom_sites(dd4d.SET_OMEGA, 0))
    psi = synth.complex_gaussian(11, synth.TAG_RHS, (len(ids), R, n, 12))
    out = np.zeros_like(psi)
    ctx.apply_D_block("omega", ids, R, psi, out, prec)
    for r in (0, 1, 87, R - 1):
        one, d = np.ascontiguousarray(psi[:, r:r + 1]), np.zeros((len(ids), 1, n, 12), dtype=np.complex128)
        ctx.apply_D_block("omega", ids, 1, one, d, prec)
        assert np.array_equal(d[:, 0], out[:, r])
    ctx.close()


def test_fp32_stencil_converts_as_the_host_does():
    """At kappa = 0 the FP32 stencil returns its input rounded to FP32 and widened again: ties, denormals, both ends."""
    L = (4, 4, 4, 4)
    U, ctx, info, _ = make_case(L, 0.0, 0.3, 1, uniform_cores(L, 1, 1))
    n = len(ctx.geom_sites(dd4d.SET_OMEGA, 0))
    rng = np.random.default_rng(5)
    v = rng.standard_normal(24 * n) * 10.0 ** rng.uniform(-44, 35, 24 * n)
    v[:9] = 0.0, -0.0, 1 + 2.0 ** -24, 1 + 3 * 2.0 ** -24, 2 - 2.0 ** -25, 2.0 ** -149, 2.0 ** -126, 1e38, -2.0 ** -140
    psi = v.view(np.complex128).reshape(1, 1, n, 12)
    out = np.zeros_like(psi)
    ctx.apply_D_block("omega", [0], 1, psi, out, "f32")
    assert np.array_equal(out.view(np.float64), psi.view(np.float64).astype(np.float32).astype(np.float64))
    ctx.close()


@pytest.mark.parametrize("inner", ["f32", "bf16"])
def test_nothing_to_solve_after_a_solve(inner):
    """b = 0 gives x = 0 whatever the work vectors hold from the solve before."""
    L = (4, 4, 4, 4)
    U, ctx, info, _ = make_case(L, 0.13, 0.3, 1, uniform_cores(L, 1, 1))
    ids, n = list(range(info["nblocks"])), len(ctx.geom_sites(dd4d.SET_OMEGA, 0))
    b = synth.complex_gaussian(4, synth.TAG_RHS, (len(ids), 2, n, 12))
    x = np.zeros_like(b)
    assert ctx.solve_blocks("omega", ids, 2, b, x, dd4d.params(TOL, inner_prec=inner))["status"] == dd4d.DD_OK
    b[:, 1] = 0                                      # every second system
    ctx.solve_blocks("omega", ids, 2, b, x, dd4d.params(TOL, inner_prec=inner))
    assert np.all(x[:, 1] == 0) and np.all(np.abs(x[:, 0]).max(axis=(1, 2)) > 0)
    x[:] = 1
    st = ctx.solve_blocks("omega", ids, 2, np.zeros_like(b), x, dd4d.params(TOL, inner_prec=inner))
    assert st["status"] == dd4d.DD_OK and np.all(x == 0)
    ctx.close()
