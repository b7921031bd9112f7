"""Calls on a device whose memory is nearly used up (a matrix or a caller's own data beside them): work space
that only makes a call faster is done without, and the results are the same bits (FP64 LU: P A = L U within
4 n u |L||U| per element)."""
import contextlib
import ctypes as C

import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.fixture(scope="module")
def N():
    from paper_2606_24154_gb300 import build, nebem
    build.build()
    nebem.load()
    return nebem


@contextlib.contextmanager
def room(megabytes):
    """All of the device's memory but this much taken (not touched), by the runtime's own allocator: torch's
    takes small requests in blocks of 20 MB."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    rt, taken = C.CDLL("libcudart.so.%s" % torch.version.cuda.split(".")[0]), []
    try:
        for block in (1 << 30, 32 * MB, 2 * MB):
            while torch.cuda.mem_get_info()[0] >= megabytes * MB + block:
                p = C.c_void_p()
                assert rt.cudaMalloc(C.byref(p), C.c_size_t(block)) == 0
                taken.append(p)
        yield
    finally:
        torch.cuda.synchronize()
        for p in taken:
            rt.cudaFree(p)


def cell():
    return I.thgem(I.PlateSpec(n_phi=24, n_r=3, n_zc=1, n_zf=4), n_plane=3)  # 828 elements


# partial sums of 125 MB and 42 MB
@pytest.mark.parametrize("precision,points,megabytes", [("mixed", 100000, 40), ("fp64", 50000, 16)])
def test_evaluation(N, precision, points, megabytes):
    import torch
    g = cell()
    prec = {"fp64": N.NEBEM_FP64, "mixed": N.NEBEM_MIXED}[precision]
    pts = torch.from_numpy(I.cell_points(g, points, I.rng(0, 9))).cuda()
    out = [[torch.empty(points, dtype=torch.float64, device="cuda"),
            torch.empty((points, 3), dtype=torch.float64, device="cuda")] for _ in range(2)]
    sigma = None
    for (phi, E), tight in zip(out, (False, True)):
        ctx = N.Context().set_geometry(g)
        sigma = ctx.solve(N.NEBEM_MIXED)[0] if sigma is None else sigma
        ctx.set_sigma(sigma)
        # the tables of the refinement are made by the first evaluation
        ctx.eval(pts[:100].cpu().numpy(), N.NEBEM_MIXED)
        with room(megabytes) if tight else contextlib.nullcontext():
            N.nebem_eval_device(ctx.h, pts.data_ptr(), points, phi.data_ptr(), E.data_ptr(), prec)
            torch.cuda.synchronize()
        ctx.close()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def test_server(N):
    g = cell()
    ctx = N.Context().set_geometry(g)
    ctx.solve(N.NEBEM_MIXED)
    pts = I.cell_points(g, 3000, I.rng(0, 10))
    want = ctx.eval(pts, N.NEBEM_MIXED)
    opt = N.nebem_server_default_options()
    opt.arena_points = 20000

    def served():
        srv, phi, E = N.nebem_server_create([ctx.h], opt), np.empty(3000), np.empty((3000, 3))
        N.nebem_server_wait(srv, N.nebem_server_submit(srv, 0, pts, phi, E, N.NEBEM_MIXED))
        N.nebem_server_destroy(srv)
        return phi, E

    for got in served(), None:
        if got is None:
            with room(24):  # its partial sums alone: 38 MB
                got = served()
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    ctx.close()


def test_factorisation(N):
    import torch
    n = 3000
    A = np.random.default_rng(n).normal(size=(n, n))
    lu, piv = torch.tensor(A.T.copy(), device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    ctx = N.Context()
    N.nebem_lu_factor_device(ctx.h, lu.clone().data_ptr(), n, piv.data_ptr())
    N.nebem_lu_factor_device_noalloc(torch.eye(64, dtype=torch.float64, device="cuda").data_ptr(), 64, piv.data_ptr())
    with room(5):  # 7.3 MB of work space; 1.6 MB without the digits
        N.nebem_lu_factor_device(ctx.h, lu.data_ptr(), n, piv.data_ptr())
        torch.cuda.synchronize()
    ctx.close()
    LU, perm = lu.cpu().numpy().T, np.arange(n)
    for k, q in enumerate(piv.cpu().numpy()):
        perm[[k, q]] = perm[[q, k]]
    L, U = np.tril(LU, -1) + np.eye(n), np.triu(LU)
    assert (np.abs(A[perm] - L @ U) <= 4 * n * 2.0 ** -53 * (np.abs(L) @ np.abs(U))).all()
