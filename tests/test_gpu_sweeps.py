"""Triangular sweeps whose CTAs pass values through memory: sizes around a block, a warp and the four column
groups, against LAPACK; a right-hand side with NaN (of the pattern that marks a value as not yet passed)
ends with NaN and no timeout.

Tolerance (derived before the first run): backward error of elimination with partial pivoting, n eps times
the size of the solution for matrices with a dominant diagonal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 15, 31, 32, 33, 63, 64, 65, 95, 97, 128, 143, 700])
def test_sweep_sizes(n):
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    gen = np.random.default_rng(n)
    A = gen.normal(size=(n, n)) / np.sqrt(n) + 4.0 * np.eye(n)[gen.permutation(n)]
    b = gen.normal(size=n)
    dA = torch.tensor(A.T.copy(), device="cuda")  # column major
    piv = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx = N.Context()
    N.nebem_lu_factor_device(ctx.h, dA.data_ptr(), n, piv.data_ptr())
    x = torch.tensor(b, device="cuda")
    N.nebem_lu_solve_device(ctx.h, dA.data_ptr(), n, piv.data_ptr(), x.data_ptr())
    ref = np.linalg.solve(A, b)
    assert np.abs(x.cpu().numpy() - ref).max() <= 64 * n * 2.2e-16 * np.abs(ref).max()
    bad = b.copy()
    bad.view(np.uint64)[n // 2] = 0xFFFFFFFFFFFFFFFF
    y = torch.tensor(bad, device="cuda")
    N.nebem_lu_solve_device(ctx.h, dA.data_ptr(), n, piv.data_ptr(), y.data_ptr())
    assert np.isnan(y.cpu().numpy()).any()
    ctx.close()
