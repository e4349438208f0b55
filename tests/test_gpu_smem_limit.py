"""Kernels whose shared memory grows with the grid (the FFT passes, the filter passes): a
handle with a small grid, used from another thread or between two calls, must not lower
the kernel's limit under a larger one's launches and captured graphs."""
import threading

import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def make(jko, n, fft, prec, gamma):
    pb = inputs.porous_problem(n, seed=1, gamma=gamma, n_steps=2)
    pb.max_iter = 8
    return pb, jko.create_from_problem(pb, precision=prec, loop=2, **({"fft": 1} if fft else {}))


@pytest.mark.parametrize("fft,prec,large,small", [(True, "FP64", 512, 64), (True, "FP32", 700, 64),
                                                  (False, "FP64", 256, 160), (False, "FP32", 512, 200)])
def test_small_grids_leave_the_limit_of_large_ones(fft, prec, large, small):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    P = jko.Precision[prec]
    gamma = 4e-3
    pa, a = make(jko, large, fft, P, gamma)
    ps, s = make(jko, small, fft, P, gamma)
    qa = torch.tensor(pa.q0, dtype=a.dtype, device="cuda")
    qs = torch.tensor(ps.q0, dtype=s.dtype, device="cuda")
    torch.cuda.synchronize()
    ref = jko.jko_flow(a, qa, 2)[1].clone()
    errors = []

    def work(h, q, reps):
        try:
            g = torch.ones_like(q)
            for _ in range(reps):
                jko.jko_flow_record(h, q, 1)
                jko.jko_flow_backward(h, g, want_w=False)   # passes launched one by one, not from a graph
        except Exception as e:                     # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(a, qa, 40)),
               threading.Thread(target=work, args=(s, qs, 200))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    again = jko.jko_flow(a, qa, 2)[1]
    jko.jko_destroy(a)
    jko.jko_destroy(s)
    assert not errors, errors
    assert torch.equal(ref, again)
