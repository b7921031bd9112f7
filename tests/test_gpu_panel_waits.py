"""The grid barrier of the cooperative LU panel running out (a poll limit of 1 through wait_polls) in both
precisions: systems of more rows than one cluster takes, FP64 with panels ahead of the trailing update too.
nebem_solve returns NEBEM_TIMEOUT from the factorisation (nothing is written, where a sweep that gives up
writes NaN), and the same context solves once the limit is back at its default.

Tolerance of the solution: ten times the mixed solve's last correction (ir_tol, 1e-8)."""
import ctypes as C

import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MESHES = {1812: (dict(n_phi=36, n_r=4, n_zc=1, n_zf=8), 5),   # FP64: cooperative panels
          2388: (dict(n_phi=36, n_r=6, n_zc=1, n_zf=8), 5),   # and the next one beside the update
          4632: (dict(n_phi=60, n_r=7, n_zc=2, n_zf=10), 6)}  # FP32: cooperative panels


@pytest.mark.parametrize("n,precision", [(1812, "fp64"), (2388, "fp64"), (4632, "mixed")])
def test_panel_gives_up_then_solves(n, precision):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    spec, plane = MESHES[n]
    g = I.thgem(I.PlateSpec(**spec), n_plane=plane)
    assert g.n == n
    prec = {"fp64": N.NEBEM_FP64, "mixed": N.NEBEM_MIXED}[precision]
    ctx = N.Context(wait_polls=1).set_geometry(g)
    sigma = np.full(g.n, 7.0)
    rc = N.load().nebem_solve(ctx.h, prec, sigma.ctypes.data_as(C.POINTER(C.c_double)), None)
    assert rc == N.NEBEM_TIMEOUT, (rc, N.load().nebem_last_error())
    assert (sigma == 7.0).all() and b"factorisation" in N.load().nebem_last_error()
    N.nebem_set_wait_polls(ctx.h, 0)
    got, _, _ = ctx.solve(prec)
    ctx.close()
    other = N.Context().set_geometry(g)
    want, _, _ = other.solve(N.NEBEM_MIXED if precision == "fp64" else N.NEBEM_FP64)
    other.close()
    assert np.abs(got - want).max() <= 1e-7 * np.abs(want).max()
