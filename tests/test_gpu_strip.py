"""The persistent CUDA-core form of a step (strip.cu) against the kernel-per-pass
form (loop = 2) on the same inputs: sizes at the edges of its tiles (one line,
lines that do not fill a work item, one more line than blocks, ragged last
blocks) and every energy kind.

Both forms add each output's terms in the same order; the persistent one applies
the two 1-D filters of xi b in the other order, so the images differ by rounding
alone: at most ~2 (2r + 2) 2^-p relative per pair and pass in the worst case,
sqrt of that as it accumulates; the bars are the precisions' own parity bars
(FP32 1e-5, FP64 1e-12 relative L1), with 8 pairs run on both sides (tol = 0)."""
import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu, rel_l1

pytestmark = pytest.mark.gpu


def problem(kind, nx, ny):
    if kind == "crowd":
        pb = inputs.crowd_problem(nx, gamma=4e-3, ny=ny, tol=0.0, max_iter=8)
    elif kind == "porous":
        pb = inputs.porous_problem(nx, seed=3, gamma=2e-3, ny=ny, tol=0.0, max_iter=8)
        pb.kappa = float(1.5 * pb.q0.max())
    elif kind == "entropy":
        pb = inputs.varying_exponent_problem(nx, seed=3, ny=ny, tol=0.0, max_iter=8)
        pb.m_field, pb.m, pb.alpha = None, 1.0, np.full(pb.N, 0.5)
        pb.w = 0.05 * np.linspace(0, 1, pb.N)
    else:
        pb = inputs.varying_exponent_problem(nx, seed=3, ny=ny, tol=0.0, max_iter=8)
    return pb


CASES = [("crowd", 1, 64), ("crowd", 64, 1), ("crowd", 33, 70), ("porous", 153, 152),
         ("entropy", 305, 41), ("exponents", 161, 333), ("porous", 513, 300),
         ("crowd", 1030, 150)]


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("kind,nx,ny", CASES)
def test_persistent_form_equals_the_kernels_per_pass(kind, nx, ny, prec):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = problem(kind, nx, ny)
    out, its, used = [], [], []
    for loop in (2, 0):
        h = jko.create_from_problem(pb, precision=jko.Precision[prec], loop=loop)
        p0 = torch.tensor(pb.q0, dtype=h.dtype, device="cuda")
        _, traj, infos = jko.jko_flow(h, p0, 2)
        _, traj2, _ = jko.jko_flow(h, p0, 2)      # the exchange buffers' epochs go on
        assert torch.equal(traj, traj2)
        out.append(traj.double().cpu().numpy())
        its.append([(i["iters"], i["status"]) for i in infos])
        used.append(jko.jko_handle_info(h)["loop"])
        jko.jko_destroy(h)
    print(kind, nx, ny, prec, "persistent", used[1], "rel L1", rel_l1(out[1], out[0]))
    assert not used[0]
    if prec == "FP32":
        assert used[1]
    assert its[0] == its[1]
    assert rel_l1(out[1], out[0]) <= (1e-12 if prec == "FP64" else 1e-5)


def test_stop_rule_of_the_persistent_form():
    """Converged, budget-bound and stalled steps report the same pairs and status
    as the kernels per pass; a non-finite potential is reported, not hung on."""
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = inputs.crowd_problem(96, gamma=1e-3, kappa_factor=1.2, n_steps=8, max_iter=60)
    for kw in (dict(tol=1e-6), dict(tol=1e-12, stall=3), dict(tol=0.0, max_iter=5)):
        infos = []
        for loop in (2, 0):
            h = jko.create_from_problem(pb, precision=jko.Precision.FP64, loop=loop, **kw)
            p0 = torch.tensor(pb.q0, dtype=torch.float64, device="cuda")
            infos.append(jko.jko_flow(h, p0, 8)[2])
            jko.jko_destroy(h)
        assert [(i["iters"], i["status"]) for i in infos[0]] == \
            [(i["iters"], i["status"]) for i in infos[1]], kw
        for a, b in zip(*infos):
            # sums of ~1e4 terms of at most ~1e-4, each with rounding ~1e-16 of it
            assert abs(a["residual_l1"] - b["residual_l1"]) <= 1e-13
    h = jko.create_from_problem(pb, precision=jko.Precision.FP32)
    p0 = torch.tensor(pb.q0, dtype=torch.float32, device="cuda")
    p_ok, _ = jko.jko_step(h, p0)
    w = torch.full((pb.N,), float("nan"), device="cuda")
    jko.jko_set_potential_device(h, w)
    _, info = jko.jko_step(h, p0)
    assert info["status"] == jko.Status.NUMERIC
    jko.jko_set_potential_device(h, torch.tensor(pb.w, dtype=torch.float32, device="cuda"))
    p_again, info = jko.jko_step(h, p0)
    assert torch.isfinite(p_again).all() and rel_l1(p_again.cpu().numpy(), p_ok.cpu().numpy()) <= 1e-6
    jko.jko_destroy(h)
