"""A batch on strips enqueues the steps of a flow without host decisions; an invalid p0 is
still reported after the first steps, not after all of them."""
import time

import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_invalid_input_does_not_run_the_whole_flow():
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pbs = [inputs.porous_problem(33, seed=2, gamma=4e-3, ny=47), inputs.crowd_problem(64, ny=41, gamma=4e-3),
           inputs.porous_problem(129, seed=4, gamma=2e-3, ny=65)]
    b = jko.jko_batch_create(pbs, precision=jko.Precision.FP32)
    good = [torch.tensor(pb.q0, dtype=torch.float32, device="cuda") for pb in pbs]
    bad = [p.clone() for p in good]
    bad[2][7] = -1.0
    jko.jko_batch_flow(b, good, 300)
    t0 = time.perf_counter()
    jko.jko_batch_flow(b, good, 300)
    t1 = time.perf_counter()
    with pytest.raises(jko.JKOError) as e:
        jko.jko_batch_flow(b, bad, 300)
    t2 = time.perf_counter()
    print("valid", t1 - t0, "invalid", t2 - t1)
    assert "flow 2" in str(e.value)
    assert t2 - t1 < 0.25 * (t1 - t0)       # two steps of 300 and their set-up
    jko.jko_batch_destroy(b)
