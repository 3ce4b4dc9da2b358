"""Rounding of the inner solver's products on systems of many 32-site chunks.

A lane adds at most 24 numbers in FP32, a warp 32 lanes in five more additions, and everything above is FP64, in the
launched form and in the one-launch form of small batches.  At kappa = 0 the Schur complement is the identity: the
inner solve's right-hand side is b on the even sites, and (r^, M p) = (r^, r).  The right-hand sides hold numbers of two
sizes, so that a longer FP32 sum would lose all the small ones behind its first.
"""

import numpy as np
import pytest

from paper_2211_06902_gb300 import dd4d, synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24                       # unit roundoff of FP32
RHS = 16                             # on the frame of 16^4 with 7^4 cores: 424 chunks of its even sites
CHUNKS = 424


def _mix32(x):
    x = x.astype(np.uint32)
    x ^= x >> np.uint32(16)
    x = (x * np.uint32(0x7feb352d)).astype(np.uint32)
    x ^= x >> np.uint32(15)
    x = (x * np.uint32(0x846ca68b)).astype(np.uint32)
    return x ^ (x >> np.uint32(16))


def _shadow(system, n, comps):
    """The generated shadow vector of one system on even sites 0 .. n - 1 (spinor.cuh), first `comps` components."""
    h = _mix32(_mix32(np.array([0x2211 + system])) + np.arange(n, dtype=np.uint32))
    m = np.arange(2 * comps, dtype=np.uint32) * np.uint32(0x9e3779b9)
    r = (h[:, None] + m[None, :]).view(np.int32).astype(np.float32).astype(np.float64) * 2.0 ** -31
    return r[:, 0::2] + 1j * r[:, 1::2]


@pytest.fixture(scope="module")
def case():
    L = (16,) * 4
    ctx = dd4d.Context(L, 0.0)
    ctx.gauge_random(0.3, 1)
    ctx.set_geometry([[(0, 6), (8, 14)]] * 4)
    sites = ctx.geom_sites(dd4d.SET_LAMBDA1)
    even = np.flatnonzero(sum(np.unravel_index(sites, L)) % 2 == 0)
    assert (len(even) + 31) // 32 == CHUNKS
    yield ctx, len(sites), even
    ctx.close()


def _solve(ctx, form, b):
    ctx.set_hop_variant("f32", 0 if form == "launched" else -1)
    x = np.zeros_like(b)
    c0 = dd4d.launch_count()
    st = ctx.solve_blocks("lambda1", None, RHS, b, x,
                          dd4d.params(1e-5, inner_prec="f32", inner_tol=0.5, maxiter=1, max_outer=1))
    launches = dd4d.launch_count() - c0
    assert st["status"] == dd4d.DD_OK and st["max_iters"] == 1
    return launches, ctx.debug_inner_sums(RHS)


@pytest.mark.parametrize("groups", [2, 4, 8, 16])    # chunks go to 2 groups of warps per CTA of a cluster of 1 .. 8
@pytest.mark.parametrize("form", ["one launch", "launched"])
def test_norms_of_long_vectors(case, form, groups):
    ctx, n, even = case
    run = -(-CHUNKS // groups)
    first = np.arange(len(even)) // 32 % run == 0
    # four numbers 1 in a lane's first chunk and pair, then numbers below half an ulp of their sum
    v = np.where(first, 1.0, float(np.float32(np.sqrt(0.9 * 2.0 ** -22))))
    b = np.zeros((1, RHS, n, 12), dtype=np.complex128)
    b[0, :, even] = (v * (1 + 1j))[:, None, None]
    _, (target, _) = _solve(ctx, form, b)
    exact = 0.25 * 24.0 * np.sum(v ** 2)
    # 24 additions in a lane and 5 in a warp, each off by at most U of the sum of positive numbers so far
    assert np.all(np.abs(target / exact - 1) <= 30 * U), np.abs(target / exact - 1).max() / U


@pytest.mark.parametrize("groups", [2, 4, 8, 16])
@pytest.mark.parametrize("form", ["one launch", "launched"])
def test_products_of_long_vectors(case, form, groups):
    ctx, n, even = case
    run = -(-CHUNKS // groups)
    first = np.arange(len(even)) // 32 % run == 0
    t = np.where(first, 1.0625, 0.9 * 2.0 ** -23)    # real part of conj(r^) b per component; the imaginary part is 0
    b = np.zeros((1, RHS, n, 12), dtype=np.complex128)
    for s in range(RHS):
        h = _shadow(s, len(even), 2)
        b[0, s, even, :2] = (t[:, None] * h / np.abs(h) ** 2).astype(np.complex64)
    _, (_, alpha) = _solve(ctx, form, b)
    # (r^, r) and (r^, M p) hold the same products in different order.  Of a lane's 24 numbers the two large components
    # are four, 2.125 together, and the other twenty ten small components: they lose at most 10 * 1.8 U / 2.125 = 8.5 U.
    # The roundings of the large ones (4) and of the warp's sum (5) are at most U each: 17.5 U down or 9 U up on
    # either side
    assert np.all(np.abs(alpha - 1) <= 27 * U), np.abs(alpha - 1).max() / U


def test_both_forms_run(case):
    """Start (2 launches), one iteration (9) and the last check against one launch."""
    ctx, n, even = case
    b = np.zeros((1, RHS, n, 12), dtype=np.complex128)
    b[0, :, even] = 1
    assert _solve(ctx, "launched", b)[0] - _solve(ctx, "one launch", b)[0] == 11
