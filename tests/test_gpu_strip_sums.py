"""The residual of a step on strips is added in FP64 beyond a thread's own outputs.  The
kernel is narrowed to one tap (xi = Id) and the input to one cell in 16 along each axis, so
that after one pair the terms are |q E - q| with one rounding, at most one of them a thread
and item.  Their sum then equals NumPy's FP64 sum of the same FP32 terms to FP64 rounding,
n 2^-53 of it for n terms on either side, where FP32 partial sums would show 2^-24."""
import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def problem(nx, ny, seed):
    rng = np.random.default_rng(seed)
    q = np.zeros((ny, nx))
    q[::16, ::16] = rng.uniform(0.1, 1.0, q[::16, ::16].shape)
    gamma = 0.5 / (100.0 * max(nx, ny) ** 2)      # e^{-h^2 / gamma} < 1e-80
    # tol 0, one pair: the report holds the residual of b = q after it
    return inputs.Problem(nx=nx, ny=ny, gamma=gamma, tau=3.0 * gamma, q0=(q / q.sum()).ravel(),
                          w=rng.uniform(0.0, 1.0, nx * ny), n_steps=1, tol=0.0, max_iter=1)


@pytest.mark.parametrize("nx,ny", [(64, 64), (201, 149), (256, 256), (512, 512), (700, 512)])
def test_residual_is_added_in_fp64(nx, ny):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = problem(nx, ny, nx)
    p0 = torch.tensor(pb.q0, dtype=torch.float32, device="cuda")
    q = p0.cpu().numpy().astype(np.float64)
    E = np.exp(-pb.tau / pb.gamma * pb.w).astype(np.float32).astype(np.float64)
    exact = float(np.abs((q * E - q).astype(np.float32)).astype(np.float64).sum())
    h = jko.create_from_problem(pb, precision=jko.Precision.FP32)
    assert jko.jko_handle_info(h)["loop"] is True
    _, _, infos = jko.jko_flow(h, p0, 1)
    assert infos[0]["iters"] == 1
    jko.jko_destroy(h)
    b = jko.jko_batch_create([pb] * 12, precision=jko.Precision.FP32)
    _, table = jko.jko_batch_flow(b, [p0] * 12, 1)
    jko.jko_batch_destroy(b)
    res = [infos[0]["residual_l1"], table[0][0]["residual_l1"]]
    terms = -(-nx // 16) * -(-ny // 16)
    print(nx, ny, exact, [abs(r - exact) / exact for r in res])
    assert exact > 0.1
    assert all(abs(r - exact) <= 2 * terms * 2.0 ** -53 * exact for r in res)
