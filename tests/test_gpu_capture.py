"""A context's first FP64 evaluation captured into a graph, its scratch with it: the replays give the bits of a call
outside."""
import numpy as np
import pytest

from paper_2606_24154_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_first_fp64_evaluation_in_a_graph():
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    g = I.thgem(I.PlateSpec(n_phi=24, n_r=3, n_zc=1, n_zf=4), n_plane=3)
    ctx = N.Context().set_geometry(g)
    sigma, _, _ = ctx.solve(N.NEBEM_MIXED)
    pts = torch.from_numpy(I.cell_points(g, 500, I.rng(0, 11))).cuda()
    phi, E = torch.zeros(500, dtype=torch.float64, device="cuda"), torch.zeros((500, 3), dtype=torch.float64, device="cuda")
    other = N.Context().set_geometry(g)
    other.set_sigma(sigma)
    want = other.eval(pts.cpu().numpy(), N.NEBEM_FP64)  # loads the kernels; ctx has no pool yet
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        N.nebem_eval_device(ctx.h, pts.data_ptr(), 500, phi.data_ptr(), E.data_ptr(), N.NEBEM_FP64,
                            torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        phi.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(phi.cpu().numpy(), want[0]) and np.array_equal(E.cpu().numpy(), want[1])
    del graph
    ctx.close()
    other.close()
