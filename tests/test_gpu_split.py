"""A point's bits do not depend on how a launch deals the work: whole point groups, element
chunks or element leaves (chosen by the number of points), FP64 and mixed."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_same_bits_for_every_split(prec):
    import torch
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    p = N.NEBEM_FP64 if prec == "fp64" else N.NEBEM_MIXED
    g = I.thgem(I.PlateSpec(n_phi=24, n_r=3, n_zc=1, n_zf=4), n_plane=3)  # 828 elements: 4 chunks, 26 leaves
    ctx = N.Context().set_geometry(g)
    ctx.solve(N.NEBEM_MIXED)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # 2 rounds of resident blocks (3 or 6 per SM, 128 points each) and a bit: whole groups too
    most = 2 * (3 if prec == "fp64" else 6) * sms * 128 + 641
    pts = I.cell_points(g, most, I.rng(0, 77))
    ref = ctx.eval(pts, p)
    for n in (1, 127, 129, 1000, 30000, most - 700):
        phi, E = ctx.eval(pts[:n], p)
        assert np.array_equal(phi, ref[0][:n]) and np.array_equal(E, ref[1][:n]), n
    ctx.close()
