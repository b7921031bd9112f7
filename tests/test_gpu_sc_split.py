"""Mixed space-charge sums: source runs shared by the blocks of a cluster or not, one or two pairs of targets
per thread, against sums in FP64; counts around the tile, unit and dispatch edges, with a softening
whose square is subnormal in FP32 (which selects the root) and an ordinary one.

Tolerance (derived before the first run): a pair's FP32 operations and its sum over 32 sources stay within
40 roundings of 6e-8 of the pair, so a sum within 2.4e-6 of the sum of the pairs' magnitudes."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("soft", [3e-20, 1e-6])
@pytest.mark.parametrize("nsrc, ntgt", [(1, 1), (33, 129), (1023, 257), (1024, 513), (1025, 1), (1153, 4863),
                                        (2049, 4865), (300, 38913), (1024, 0), (4865, 0), (1000, 0)])
def test_split_sums(nsrc, ntgt, soft):
    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    gen = np.random.default_rng(nsrc + ntgt)
    src = gen.uniform(-1e-3, 1e-3, (nsrc, 3))
    q = gen.choice([-1.0, 1.0, 2.5], nsrc) * 1.602e-19
    own = ntgt == 0  # the carriers themselves, each without its own term
    if own:
        soft = max(soft, 1e-18)  # below 5e-20 the excluded pair's 1 / s^2 is infinite in FP32
    tgt = src if own else gen.uniform(-1e-3, 1e-3, (ntgt, 3))
    ctx = N.Context().set_geometry(I.cube(n_per_edge=1))
    N.nebem_space_charge(ctx.h, src, q, soft)
    phi, E = N.nebem_space_charge_eval(ctx.h, tgt, N.NEBEM_MIXED, exclude_self=own)
    ctx.close()
    ke = 1.0 / (4 * np.pi * 8.8541878128e-12)
    for a in range(0, len(tgt), 2048):
        d = tgt[a : a + 2048, None] - src[None]
        r2 = (d**2).sum(-1) + soft**2
        if own:
            r2[np.arange(len(r2)), a + np.arange(len(r2))] = np.inf
        w = ke * q / np.sqrt(r2)
        assert (np.abs(phi[a : a + 2048] - w.sum(1)) <= 2.4e-6 * np.abs(w).sum(1)).all()
        f = w / r2
        size = np.abs(f[..., None] * d).sum(1)
        assert (np.abs(E[a : a + 2048] - (f[..., None] * d).sum(1)) <= 2.4e-6 * size).all()
