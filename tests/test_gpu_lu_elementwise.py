"""FP64 LU element by element: matrices whose elements differ in size in ways that scaling rows and columns
cannot undo, so that the digits of the trailing update (lu_tc64.cu) are too coarse for a part of the elements.

Tolerance (derived before the first run): elimination's bound |P A - L U| <= n u |L| |U| holds per element;
four times it, for U12 through the explicit inverse of the unit-lower block.  L U is formed in extended
precision.  The same factorisation with FP64 fmas throughout (nebem_lu_factor_device_noalloc) is held to the
same bound, and says which elements become infinite or NaN."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
U53 = 2.0 ** -53


@pytest.fixture(scope="module")
def N():
    from paper_2606_24154_gb300 import build, nebem
    build.build()
    nebem.load()
    return nebem


def factor(N, A, fmas=False, **opts):
    import torch
    n = A.shape[0]
    ctx = N.Context(**opts)
    d = torch.tensor(np.asfortranarray(A).ravel(order="F"), device="cuda")
    p = torch.empty(n, dtype=torch.int32, device="cuda")
    try:
        if fmas:
            N.nebem_lu_factor_device_noalloc(d.data_ptr(), n, p.data_ptr())
        else:
            N.nebem_lu_factor_device(ctx.h, d.data_ptr(), n, p.data_ptr())
    except N.NebemError as e:
        assert e.code == N.NEBEM_SINGULAR
    torch.cuda.synchronize()
    ctx.close()
    LU, perm = d.cpu().numpy().reshape(n, n, order="F"), np.arange(n)
    for k, q in enumerate(p.cpu().numpy()):
        perm[[k, q]] = perm[[q, k]]
    return LU, perm


def excess(A, LU, perm, tiny=0.0):
    """The largest |P A - L U| over its bound."""
    n = A.shape[0]
    L = (np.tril(LU, -1) + np.eye(n)).astype(np.longdouble)
    U = np.triu(LU).astype(np.longdouble)
    err, bound = np.abs(A[perm] - L @ U), 4 * n * U53 * (np.abs(L) @ np.abs(U)) + tiny
    return float((err / np.where(bound > 0, bound, 1)).max())


def groups(n, eps, member, seed):
    A = np.random.default_rng(seed).normal(size=(n, n))
    return np.where(member[:, None] == member[None], A, eps * A)


def coupled(n, eps):
    return groups(n, eps, np.arange(n) % 2, n)


def sparse_column(n, big):
    A = np.random.default_rng(n).normal(size=(n, n)) + 40 * np.eye(n)
    A[:, -1] = 0
    A[32, -1], A[-1, -1] = big, 1
    return A


@pytest.mark.parametrize("A", [pytest.param((coupled, n, e), id="coupled-%d-%g" % (n, e))
                               for n in (192, 333) for e in (1.0, 1e-4, 1e-8, 1e-14, 1e-20)] +
                         [pytest.param((sparse_column, 192, b), id="column-%g" % b) for b in (1e6, 1e8, 1e12, 1e16)])
def test_weak_coupling(N, A):
    A = A[0](*A[1:])
    assert excess(A, *factor(N, A)) <= 1
    assert excess(A, *factor(N, A, fmas=True)) <= 1


@pytest.mark.parametrize("block", [32, 64])
@pytest.mark.parametrize("rows", [1, 8, 9, 31])
def test_weakly_coupled_rows_of_a_warp(N, rows, block):
    """`rows` of every 32 in a group of their own: the single elements and the chains of the fma path."""
    n = 230
    A = groups(n, 1e-12, np.arange(n) % 32 < rows, rows) + 40 * np.eye(n)
    LU, perm = factor(N, A, lu_block=block)
    assert np.array_equal(perm, np.arange(n))
    assert excess(A, LU, perm) <= 1


@pytest.mark.parametrize("scale", [1e300, 1e-300])
def test_ends_of_the_exponent_range(N, scale):
    n = 200
    A = np.random.default_rng(5).normal(size=(n, n)) * scale
    assert excess(A, *factor(N, A), tiny=n * 2.0 ** -1074) <= 1


def test_zero_rows_and_columns(N):
    """Zeros in L21 (rows) and U12 (columns) of the first panels, and two blocks without coupling."""
    n = 250
    A = np.random.default_rng(6).normal(size=(n, n)) + 40 * np.eye(n)
    A[100:140, :90] = 0
    A[:90, 150:190] = 0
    A[:128, 200:] = A[200:, :128] = 0
    LU, perm = factor(N, A)
    assert excess(A, LU, perm) <= 1
    assert (LU[100:140, :90] == 0).all() and (LU[:90, 150:190] == 0).all()
    assert (LU[:128, 200:] == 0).all() and (LU[200:, :128] == 0).all()


@pytest.mark.parametrize("value,row,col", [(np.inf, 3, 199), (-np.inf, 3, 199), (np.nan, 3, 199), (np.nan, 199, 5)])
def test_not_finite(N, value, row, col):
    """One such value in U12's last column, or (NaN, which is never a pivot) in L21's last row: where the
    factors are not finite they are what fmas make of it, and the others keep their bound."""
    n = 200
    A = np.random.default_rng(3).normal(size=(n, n)) + 20 * np.eye(n)
    A[row, col] = value
    LU, perm = factor(N, A)
    ref, rperm = factor(N, A, fmas=True)
    assert np.array_equal(perm, np.arange(n)) and np.array_equal(rperm, perm)
    assert np.array_equal(np.isnan(LU), np.isnan(ref)) and np.array_equal(np.isinf(LU), np.isinf(ref))
    m = n - 1
    assert np.isfinite(LU[:m, :m]).all() and excess(A[:m, :m], LU[:m, :m], np.arange(m)) <= 1
