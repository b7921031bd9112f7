"""A block may touch the shared memory of another block of its cluster only once that block is known to run,
which takes a cluster barrier.  Whether one is missing does not show in results (the blocks of a cluster start
within less than the time that the kernels take to load their data), so the order is read from the source:
in every kernel body that maps another block's shared memory, a cluster barrier stands before the first use."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_24154_gb300", "csrc")
BARRIER = re.compile(r"(this_cluster\(\)|\bcl)\.(sync|barrier_wait)\(")
REMOTE = re.compile(r"map_shared_rank\(|mapa\.shared::cluster")


def bodies():
    """(file, first line, text) of every top-level function of the CUDA sources that reaches remote memory."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^__(?:device|global)__.*?^}", text, re.M | re.S):
            if REMOTE.search(m.group(0)):
                yield os.path.basename(path), text.count("\n", 0, m.start()) + 1, m.group(0)


FOUND = list(bodies())


def test_the_kernels_are_found():
    assert {f for f, _, _ in FOUND} >= {"lu.cu", "spacecharge.cu"}


@pytest.mark.parametrize("name,line,text", FOUND, ids=["%s:%d" % b[:2] for b in FOUND])
def test_barrier_before_remote_memory(name, line, text):
    barrier = BARRIER.search(text)
    assert barrier and barrier.start() < REMOTE.search(text).start(), (name, line)


@pytest.mark.gpu
@pytest.mark.parametrize("single", [False, True])
def test_panels_of_blocks_without_rows(single):
    """The smallest panels, most of whose 16 blocks hold no rows, beside work of another stream: P A = L U
    within elimination's n u |L||U| (four times it), the same factors every time."""
    import numpy as np
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    dt = np.float32 if single else np.float64
    factor = N.nebem_lu_factor_device_f32 if single else N.nebem_lu_factor_device
    ctx, other = N.Context(), torch.cuda.Stream()
    busy = torch.randn(2048, 2048, device="cuda")
    torch.cuda.synchronize()
    for n in (1, 2, 5, 17, 33):
        A = np.random.default_rng(n).normal(size=(n, n)).astype(dt)
        first = None
        for _ in range(40):
            with torch.cuda.stream(other):
                busy @ busy
            dA, piv = torch.tensor(A.T.copy(), device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
            factor(ctx.h, dA.data_ptr(), n, piv.data_ptr(), torch.cuda.current_stream().cuda_stream)
            got = dA.cpu().numpy().T
            first = got if first is None else first
            assert np.array_equal(got, first)
        L, U, perm = np.tril(first.astype(float), -1) + np.eye(n), np.triu(first.astype(float)), np.arange(n)
        for k, p in enumerate(piv.cpu().numpy()):
            perm[[k, p]] = perm[[p, k]]
        u = np.finfo(dt).eps / 2
        assert (np.abs(A[perm].astype(float) - L @ U) <= 4 * max(n, 8) * u * (np.abs(L) @ np.abs(U))).all()
    torch.cuda.synchronize()
    ctx.close()
