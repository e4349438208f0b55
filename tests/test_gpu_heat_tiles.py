"""The heat kernel on resident tiles beside obstacles that cover whole tiles or their
edges (blocks that read a block's words without free cells of their own beside it): the
same bits as the kernels per Clenshaw phase, at fixed pair counts."""
import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def problem(nx, ny, kind, pairs):
    pb = inputs.heat_crowd_problem(nx, ny=ny, n_steps=2, tol=0.0, max_iter=pairs)
    X, Y = np.meshgrid((np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny)
    mask = {"two rooms": np.asarray(pb.mask, bool).reshape(ny, nx),
            "thick wall": (np.abs(X - 0.5) < 0.12) & (np.abs(Y - 0.5) >= 0.1),
            "closed wall": np.abs(Y - 0.4) < 0.1,
            "disk": (X - 0.5) ** 2 + (Y - 0.5) ** 2 < 0.04,
            "square": (np.abs(X - 0.45) < 0.15) & (np.abs(Y - 0.45) < 0.15)}[kind]
    q = np.where(mask.ravel(), 0.0, pb.q0)
    pb.q0 = q / q.sum()
    pb.kappa = 1.2 * float(pb.q0.max())
    pb.mask = mask.ravel().astype(np.uint8)
    return pb


@pytest.mark.parametrize("prec,nx,ny,kind", [
    ("FP64", 30, 20, "two rooms"), ("FP32", 96, 90, "two rooms"), ("FP32", 150, 150, "two rooms"),
    ("FP64", 200, 200, "two rooms"), ("FP32", 48, 40, "thick wall"), ("FP64", 100, 100, "disk"),
    ("FP32", 100, 100, "square"), ("FP32", 37, 61, "closed wall")])
def test_tiles_equal_the_kernels_per_phase_beside_obstacles(prec, nx, ny, kind):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = problem(nx, ny, kind, pairs=25)
    out = []
    for loop in (2, 1):
        h = jko.create_from_problem(pb, precision=jko.Precision[prec], loop=loop)
        p0 = torch.tensor(pb.q0, dtype=h.dtype, device="cuda")
        _, traj, infos = jko.jko_flow(h, p0, 2)
        assert [i["iters"] for i in infos] == [25, 25]
        out.append(traj)
        jko.jko_destroy(h)
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("prec,nx,ny,steps", [
    ("FP32", 64, 64, 2), ("FP64", 40, 56, 2), ("FP32", 100, 100, 2), ("FP64", 50, 50, 2),
    ("FP32", 37, 61, 1), ("FP32", 1, 64, 1), ("FP64", 5, 4, 1)])
def test_residuals_have_the_bits_of_the_kernels_per_phase(prec, nx, ny, steps):
    """The residual decides the stop, so it is added in FP64 and in one order in every
    form: the reports are equal, not only the images."""
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = inputs.heat_crowd_problem(nx, ny=ny, n_steps=steps, tol=1e-6, max_iter=60) \
        if min(nx, ny) > 5 else problem_1d(nx, ny)
    out = []
    for loop in (2, 1):
        h = jko.create_from_problem(pb, precision=jko.Precision[prec], loop=loop)
        p0 = torch.tensor(pb.q0, dtype=h.dtype, device="cuda")
        _, traj, infos = jko.jko_flow(h, p0, steps)
        out.append([(i["iters"], int(i["status"]), i["residual_l1"], i["mass"]) for i in infos])
        jko.jko_destroy(h)
    print(prec, nx, ny, out)
    assert out[0] == out[1]


def problem_1d(nx, ny):
    n = nx * ny
    t = (np.arange(n) + 0.5) / n
    q0 = (t < 0.3).astype(np.float64)
    return inputs.Problem(nx=nx, ny=ny, gamma=1e-3, tau=0.01, q0=q0 / q0.sum(), w=3.0 * t,
                          kappa=float((q0 / q0.sum()).max()), heat_L=10, n_steps=1, tol=1e-6, max_iter=40)
