"""FP64 LU with the digit-product trailing update (lu_tc64.cu) at the edges of its tiles (64 columns,
128 rows), with rows and columns scaled by powers of ten, and with a NaN entry.

Tolerance (derived before the first run): the classical bound |P A - L U| <= n u |L| |U| with u =
2^-53, taken at the largest entry of |L| |U| of the unscaled matrix, times 8 for U12 through the
explicit inverse of the unit-lower block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    from paper_2606_24154_gb300 import build, nebem
    build.build()
    nebem.load()
    return nebem


def _factor(N, A, **opts):
    import torch
    n = A.shape[0]
    ctx = N.Context(**opts)
    d = torch.tensor(np.asfortranarray(A).ravel(order="F"), device="cuda")
    p = torch.empty(n, dtype=torch.int32, device="cuda")
    code = 0
    try:
        N.nebem_lu_factor_device(ctx.h, d.data_ptr(), n, p.data_ptr())
    except N.NebemError as e:
        code = e.code
    LU, piv = d.cpu().numpy().reshape(n, n, order="F"), p.cpu().numpy()
    perm = np.arange(n)
    for k, q in enumerate(piv):
        perm[[k, q]] = perm[[q, k]]
    ctx.close()
    return np.tril(LU, -1) + np.eye(n), np.triu(LU), perm, code


@pytest.mark.parametrize("block", [32, 64])
@pytest.mark.parametrize("n", [64, 65, 127, 129, 192, 193, 257, 450])
def test_factors_reconstruct_under_scaling(N, n, block):
    gen = np.random.default_rng(n)
    A = gen.normal(size=(n, n))
    rows, cols = 10.0 ** gen.integers(-9, 10, n), 10.0 ** gen.integers(-9, 10, n)
    for dr, dc in ((np.ones(n), np.ones(n)), (rows, np.ones(n)), (np.ones(n), cols)):
        S = A * dr[:, None] * dc[None, :]
        L, U, perm, code = _factor(N, S, lu_block=block)
        assert code == 0
        back = 1.0 / (dr[perm][:, None] * dc[None, :])
        err = np.abs(S[perm] - L @ U) * back
        big = (np.abs(L) @ np.abs(U)) * back
        # err's own evaluation in FP64 is bounded by the same n u |L| |U|
        assert err.max() <= (8 + 1) * n * 2.0 ** -53 * big.max(), (err.max(), big.max())


def test_nan_stays_in_its_row(N):
    n = 200
    A = np.random.default_rng(3).normal(size=(n, n)) + 20 * np.eye(n)
    B = A.copy()
    B[n - 1, 5] = np.nan  # never a pivot candidate before the last column
    L, U, perm, code = _factor(N, B)
    assert code == N.NEBEM_SINGULAR  # the last column's only candidate is NaN
    Lc, Uc, permc, _ = _factor(N, A)
    if permc[n - 1] == n - 1:
        assert np.array_equal(L[: n - 1], Lc[: n - 1]) and np.array_equal(U[: n - 1], Uc[: n - 1])
    assert np.isfinite(L[: n - 1]).all() and np.isfinite(U[: n - 1]).all()
    assert np.isnan(U[n - 1, n - 1])
