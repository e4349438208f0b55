"""The heat kernel's persistent form with grid barriers (heat.cu), whose blocks walk over
several tiles: grids beyond the resident tiles (test_heat_tiles.py checks that these sizes
are), against the kernels per Clenshaw phase: the same bits and reports."""
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nx,ny", [("FP32", 900, 880), ("FP64", 760, 800)])
def test_loop_form_equals_the_kernels_per_phase(prec, nx, ny):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = inputs.heat_crowd_problem(nx, ny=ny, n_steps=2, tol=0.0, max_iter=3)
    out = []
    for loop in (2, 1):
        h = jko.create_from_problem(pb, precision=jko.Precision[prec], loop=loop)
        _, traj, infos = jko.jko_flow(h, torch.tensor(pb.q0, dtype=h.dtype, device="cuda"), 2)
        out.append((traj.clone(), [(i["iters"], i["residual_l1"], i["mass"]) for i in infos]))
        jko.jko_destroy(h)
    print(prec, nx, ny, out[0][1])
    assert [i[0] for i in out[0][1]] == [3, 3]
    assert out[0][1] == out[1][1]
    assert torch.equal(out[0][0], out[1][0])
