"""A batch whose flows all run on strips (one graph per step, images copied in one
launch): an invalid p0 is reported for its flow with the outputs untouched and the
batch usable afterwards; more steps than a call before; flows that share the SMs
unevenly (one large, several small, odd sizes and an image whose bytes are no
multiple of 16) equal the flows alone, bit for bit."""
import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def problems():
    return [inputs.crowd_problem(300, gamma=1e-3, tol=1e-6, n_steps=2),
            inputs.porous_problem(33, seed=2, gamma=4e-3, ny=47),
            inputs.crowd_problem(64, ny=41, gamma=4e-3),
            inputs.porous_problem(129, seed=4, gamma=2e-3, ny=65)]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
def test_uneven_flows_equal_the_flows_alone(prec):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pbs = problems()
    P = jko.Precision[prec]
    b = jko.jko_batch_create(pbs, precision=P)
    dt = torch.float32 if prec == "FP32" else torch.float64
    p0s = [torch.tensor(pb.q0, dtype=dt, device="cuda") for pb in pbs]
    for steps in (1, 18, 3):
        finals, table = jko.jko_batch_flow(b, p0s, steps)
    for f, pb in enumerate(pbs):
        h = jko.create_from_problem(pb, precision=P)
        pf, _, infos = jko.jko_flow(h, p0s[f], 3)
        assert torch.equal(pf, finals[f]), f
        assert [i["iters"] for i in infos] == [table[t][f]["iters"] for t in range(3)]
        jko.jko_destroy(h)
    jko.jko_batch_destroy(b)


def test_invalid_input_leaves_outputs_untouched():
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pbs = problems()[1:]
    b = jko.jko_batch_create(pbs, precision=jko.Precision.FP32)
    good = [torch.tensor(pb.q0, dtype=torch.float32, device="cuda") for pb in pbs]
    ref, _ = jko.jko_batch_flow(b, good, 1)
    for bad_value in (float("nan"), -1.0):
        bad = [p.clone() for p in good]
        bad[1][5] = bad_value
        outs = [torch.full_like(p, 7.0) for p in good]
        with pytest.raises(jko.JKOError) as e:
            jko.jko_batch_step(b, bad, outs)
        assert "flow 1" in str(e.value)
        assert all(bool((o == 7.0).all()) for o in outs)
    again, _ = jko.jko_batch_flow(b, good, 1)
    assert all(torch.equal(x, y) for x, y in zip(ref, again))
    jko.jko_batch_destroy(b)
