"""Factorisations of different orders in two threads, a context each, at the same time: no call's launch settings
reach the other's, and the factors are those of the calls one after another, bit for bit."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("single", [False, True])
def test_two_orders_at_once(single):
    import torch

    from paper_2606_24154_gb300 import build, nebem as N
    build.build()
    factor = N.nebem_lu_factor_device_f32 if single else N.nebem_lu_factor_device
    dt = torch.float32 if single else torch.float64
    orders = (6000, 4200) if single else (7000, 1700)  # both beyond the one-cluster panel
    A = [torch.from_numpy(np.random.default_rng(n).normal(size=(n, n))).to("cuda", dt) for n in orders]

    def work(k, repeats):
        ctx, out = N.Context(), []
        for _ in range(repeats):
            lu, piv = A[k].clone(), torch.empty(orders[k], dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            factor(ctx.h, lu.data_ptr(), orders[k], piv.data_ptr())
            out.append((lu, piv))
        torch.cuda.synchronize()
        ctx.close()
        return out

    want = [work(k, 1)[0] for k in (0, 1)]
    got, wrong = [None, None], []

    def thread(k, repeats):
        try:
            got[k] = work(k, repeats)
        except Exception as e:  # reported by the test's own thread
            wrong.append(e)

    threads = [threading.Thread(target=thread, args=(0, 8)), threading.Thread(target=thread, args=(1, 24))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong
    for k in (0, 1):
        for lu, piv in got[k]:
            assert torch.equal(piv, want[k][1]) and torch.equal(lu, want[k][0])
