"""The error scales of refinement level 1 are FP64 sums.  On a charged conductor every density and every Phi' is
positive, so B_phi is the potential itself, summed over the same values in the same order, and the
returned estimate is 1e-9 phi whatever the values' own errors are.

Tolerance (derived before the first run): 2 n u of the sum of 384 positive terms, 1e-13; a sum in FP32 is
off by about 1e-8."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("points", [9, 257, 20011])  # lanes; lanes; a thread per point
def test_estimate_is_the_potential(points):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    g = I.cube(n_per_edge=8)
    ctx = N.Context(mixed_point_tol=1e-7).set_geometry(g)
    sigma, _, _ = ctx.solve(N.NEBEM_FP64)
    assert (sigma > 0).all()
    gen = np.random.default_rng(points)
    d = gen.normal(size=(points, 3))
    # outside the cube of edge 0.01, beyond 3 radii (2.7e-3) of every element: no pair in FP64
    pts = d / np.linalg.norm(d, axis=1)[:, None] * gen.uniform(0.0125, 0.03, (points, 1))
    phi, _, err, _ = ctx.eval_err(pts)
    assert np.abs(err[:, 0] / (1e-9 * phi) - 1).max() <= 1e-13
