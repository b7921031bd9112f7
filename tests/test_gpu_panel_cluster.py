"""LU panels in one thread-block cluster: systems around its edges (fewer rows than CTAs, whole and partial
panels, the largest FP64 panel of 16 x 96 rows and one more), P A = L U.

Tolerance (derived before the first run): elimination's backward error n u |L||U|, four times it for the
tensor-core update's digits; pivots never smaller than another entry of their column (|L| <= 1, with
one rounding of the scaled column)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 5, 16, 17, 63, 65, 130, 400, 1535, 1537])
@pytest.mark.parametrize("single", [False, True])
def test_factors(n, single):
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    dt = np.float32 if single else np.float64
    A = np.random.default_rng(n).normal(size=(n, n)).astype(dt)
    dA = torch.tensor(A.T.copy(), device="cuda")  # column major
    piv = torch.empty(n, dtype=torch.int32, device="cuda")
    ctx = N.Context()
    (N.nebem_lu_factor_device_f32 if single else N.nebem_lu_factor_device)(ctx.h, dA.data_ptr(), n, piv.data_ptr())
    torch.cuda.synchronize()
    ctx.close()
    lu = dA.cpu().numpy().T.astype(np.float64)
    L, U = np.tril(lu, -1) + np.eye(n), np.triu(lu)
    perm = np.arange(n)
    for k, p in enumerate(piv.cpu().numpy()):
        perm[[k, p]] = perm[[p, k]]
    u = np.finfo(dt).eps / 2
    assert np.abs(L).max() <= 1 + 4 * u
    bound = 4 * max(n, 8) * u * (np.abs(L) @ np.abs(U))
    assert (np.abs(A[perm].astype(np.float64) - L @ U) <= bound).all()


@pytest.mark.parametrize("n", [2111, 2112, 2240, 3001])
def test_panels_ahead(n):
    """Sizes where the first panels are taken beside the trailing update: the first whole step, one row less,
    and a partial last panel; backward error 4 n u of |A| |x|."""
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    gen = np.random.default_rng(n)
    A = gen.normal(size=(n, n)) + 8 * np.sqrt(n) * np.eye(n)[gen.permutation(n)]
    b = gen.normal(size=n)
    dA = torch.tensor(A.T.copy(), device="cuda")
    piv = torch.empty(n, dtype=torch.int32, device="cuda")
    x = torch.tensor(b, device="cuda")
    ctx = N.Context()
    N.nebem_lu_factor_device(ctx.h, dA.data_ptr(), n, piv.data_ptr())
    N.nebem_lu_solve_device(ctx.h, dA.data_ptr(), n, piv.data_ptr(), x.data_ptr())
    torch.cuda.synchronize()
    ctx.close()
    x = x.cpu().numpy()
    assert (np.abs(A @ x - b) <= 4 * n * 1.2e-16 * (np.abs(A) @ np.abs(x) + np.abs(b))).all()
