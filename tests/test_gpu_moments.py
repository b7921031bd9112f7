"""The refinement's first level: pairs from 28 radii on by the element's moments, nearer ones by Gauss
nodes, against the FP64 path; one element of each kind (of 20 um, and scaled by 1e-5 and 1e5), with 1, 9, 25 and 121 copies (an odd count
leaves half of the last packed step empty).

Tolerance (derived before the first run): the series ends at degree 4, and the terms left out are
at most 1.3e-9 (phi) and 7.8e-9 (E) of the pair at 28 radii (triangles), falling like r^-5; the FP32
terms add 2e-10 and 1e-9; the 6-point rule between 24 and 28 radii has 1.9e-9 and six times
that; all relative to the result, which one near pair dominates."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu

U = 2e-5
SHAPES = {
    "triangle": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [0.3 * U, 0.1 * U, 0.8 * U]]),
    "sliver": (I.KIND_TRI, [[0, 0, 0], [U, 0, 0], [0.1 * U, 0, 0.05 * U]]),
    "strip": (I.KIND_RECT, [[0, 0, 0], [U, 0, 0], [U, 0, 0.1 * U], [0, 0, 0.1 * U]]),
    "quad": (I.KIND_QUAD, [[0, 0, 0], [U, 0, 0], [0.8 * U, 0, 0.9 * U], [0.1 * U, 0, 0.6 * U]]),
}


@pytest.mark.parametrize("half, scale", [(0, 1.0), (1, 1.0), (2, 1.0), (5, 1.0), (1, 1e-5), (1, 1e5)])
@pytest.mark.parametrize("name", list(SHAPES))
def test_level1_against_fp64(name, half, scale):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    kind, verts = SHAPES[name][0], scale * np.array(SHAPES[name][1], float)
    el = np.zeros(1, dtype=I.ELEMENT_DTYPE)
    el["kind"], el["eps_a"], el["eps_b"] = kind, 1.0, 1.0
    v = np.zeros((4, 3))
    v[: len(verts)] = verts
    el["v"] = v
    c = np.mean(verts, axis=0)
    rho = max(np.linalg.norm(np.subtract(p, c)) for p in verts)
    gen = np.random.default_rng(half)
    d = gen.normal(size=(240, 3))
    d[:40, 1] = 0.0
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    r = np.repeat([24.5, 27.9, 28.1, 40.0, 64.0, 300.0], 40) * rho
    pts = c + r[:, None] * d
    # level 1 for every point: an estimate above the tolerance after the FP32 pass, below it after level 1
    ctx = N.Context(mixed_point_tol=1e-6)
    lattice = scale * np.array([2000.0 * U, 0, 0, 0, 2000.0 * U, 0]) if half else None
    N.nebem_set_geometry(ctx.h, el, lattice, -half, half)
    ctx.n = 1
    ctx.set_sigma(np.array([1e-6]))
    N.nebem_set_error_model(ctx.h, 0.0, 1e3, 0.0)
    phi, E = ctx.eval(pts, N.NEBEM_MIXED)
    st = N.nebem_eval_stats(ctx.h)
    assert st.refined_level1 == pts.shape[0] and st.refined_level2 == 0
    rphi, rE = ctx.eval(pts, N.NEBEM_FP64)
    ctx.close()
    x = (28 * rho / r) ** 5
    x[r < 28 * rho] = 1.5
    assert (np.abs(phi - rphi) <= (1.6e-9 * x + 2e-10) * np.abs(rphi)).all()
    size = np.linalg.norm(rE, axis=1)
    # the copies are 2000 U apart: E is within a few per cent of the nearest pair's, nothing cancels
    assert (np.linalg.norm(E - rE, axis=1) <= (1e-8 * x + 1e-9) * size).all()
