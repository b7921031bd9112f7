"""Refinement of short lists (a thread per point and element) against the thread-per-point path: the same points
alone, in lists around a unit of eight, and in one long list, with 1, 9 and 121 copies (tiles of 32 and 8 elements),
give the same bits, and 121 copies agree with the FP64 path.

Tolerance (derived before the first run): 1e-11 of the sum of the magnitudes at level 2, the level's
own estimate, and 1e-9 at level 1."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tol", [1e-8, 1e-13])  # level 1 (nearly) alone, both levels
@pytest.mark.parametrize("half", [0, 1, 5])
def test_short_lists(half, tol):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    g = I.cube(n_per_edge=3)
    gen = np.random.default_rng(half)
    size = np.abs(g.elements["v"]).max()
    ctx = N.Context(mixed_point_tol=tol)
    lattice = np.array([20 * size, 0, 0, 0, 20 * size, 0]) if half else None
    N.nebem_set_geometry(ctx.h, g.elements, lattice, -half, half)
    ctx.n = g.elements.size
    ctx.set_sigma(gen.uniform(0.5, 1.5, ctx.n) * 1e-9)
    # all points flagged after the FP32 pass; level 1's own estimate (1e-9 B) decides on level 2
    N.nebem_set_error_model(ctx.h, 0.0, 1e3, 0.0)
    leaves = -(-ctx.n // 32)
    many = 8 * (32 * 5 * 160 // leaves + 1)
    pts = gen.uniform(-4 * size, 4 * size, (many, 3))
    phi, E = ctx.eval(pts, N.NEBEM_MIXED)
    st = N.nebem_eval_stats(ctx.h)
    assert st.refined_level1 == many and (tol > 1e-9 or st.refined_level2 == many)
    for a, b in ((0, 1), (3, 10), (11, 19), (100, 133), (5, 505)):
        p, e = ctx.eval(pts[a:b], N.NEBEM_MIXED)
        assert np.array_equal(p, phi[a:b]) and np.array_equal(e, E[a:b])
    rp, rE = ctx.eval(pts[:505], N.NEBEM_FP64)
    ctx.close()
    scale = 1e-9 if tol > 1e-9 else 1e-11
    assert (np.abs(phi[:505] - rp) <= scale * np.abs(rp)).all()  # one sign: the sum is its magnitudes'
    # |E|: the magnitudes' sum is at most phi's over the distance, 0.05 size
    assert (np.linalg.norm(E[:505] - rE, axis=1) <= scale * np.abs(rp) / (0.05 * size)).all()


@pytest.mark.parametrize("half", [0, 1, 5])
@pytest.mark.parametrize("per_edge", [3, 7])
def test_short_lists_fp32_pass(half, per_edge):
    """The FP32 pass of few points (a thread per point and element) and of many: the same bits, estimates included;
    tiles of 16 and 4 elements with whole and partial groups, a last leaf of 22 and of 6 elements."""
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    g = I.cube(n_per_edge=per_edge)
    gen = np.random.default_rng(half)
    size = np.abs(g.elements["v"]).max()
    ctx = N.Context(mixed_point_tol=0.0)
    lattice = np.array([6 * size, 0, 0, 0, 6 * size, 0]) if half else None
    N.nebem_set_geometry(ctx.h, g.elements, lattice, -half, half)
    ctx.n = g.elements.size
    ctx.set_sigma(gen.normal(size=ctx.n) * 1e-9)
    pts = gen.uniform(-2.5 * size, 2.5 * size, (12000, 3))
    phi, E, err, _ = ctx.eval_err(pts)
    for a, b in ((0, 1), (3, 10), (11, 19), (100, 133), (5, 505)):
        p, e, r, _ = ctx.eval_err(pts[a:b])
        assert np.array_equal(p, phi[a:b]) and np.array_equal(e, E[a:b]) and np.array_equal(r, err[a:b])
    ctx.close()
