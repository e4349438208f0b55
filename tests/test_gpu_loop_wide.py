"""The TF32 loop kernel on units of two tiles (grids whose 64-wide tiles need more
than one round of CTAs) against the kernels per pass with 64-wide tiles: each output
adds the same products in the same order, so the same bits and pair counts.  Ragged
sizes with an odd number of tiles along one or both axes (the last unit has one
tile), a plain and a general prox."""
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nx,ny", [("crowd", 1600, 1304), ("porous", 1304, 1600),
                                        ("crowd", 2048, 1920), ("crowd", 1540, 1412)])
def test_wide_units_equal_the_kernels_per_pass(kind, nx, ny):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    if kind == "crowd":
        pb = inputs.crowd_problem(nx, gamma=2e-4, ny=ny, tol=0.0, max_iter=3)
    else:
        pb = inputs.porous_problem(nx, seed=3, gamma=2e-4, ny=ny, tol=0.0, max_iter=3)
    out, its = [], []
    for kw in (dict(loop=2, tile=64), dict(loop=1)):
        h = jko.create_from_problem(pb, precision=jko.Precision.TF32, **kw)
        p0 = torch.tensor(pb.q0, dtype=torch.float32, device="cuda")
        _, traj, infos = jko.jko_flow(h, p0, 2)
        out.append(traj.clone())
        its.append([(i["iters"], i["status"], i["residual_l1"]) for i in infos])
        jko.jko_destroy(h)
    assert its[0] == its[1]
    assert torch.equal(out[0], out[1])
