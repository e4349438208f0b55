"""Steps with several couplings as one persistent CUDA-core kernel (strip.cu)
against the kernels per pass (loop = 2) on the same inputs: the attraction (with
and without a mask), two species and the pairwise attraction, at one line a
block, ragged last blocks, several lines a block and lines of both kinds missing
from some blocks.

Both forms add each output's terms in the same order; the persistent one applies
the two 1-D filters of its second half in the other order, so the images differ
by rounding alone, as for one density: the precisions' own parity bars (FP32 1e-5,
FP64 1e-12 relative L1), with 8 pairs run on both sides (tol = 0)."""
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu, rel_l1

pytestmark = pytest.mark.gpu


def problem(kind, nx, ny):
    kw = dict(ny=ny, tol=0.0, max_iter=8)
    if kind == "attraction":
        return inputs.attraction_problem(nx, gamma=5e-3, tau=0.3, **kw)
    if kind == "rooms":
        return inputs.attraction_problem(nx, gamma=1e-2, tau=0.3, two_rooms=True, **kw)
    if kind == "species":
        return inputs.two_species_problem(nx, gamma=4e-3, **kw)
    return inputs.pairwise_attraction_problem(nx, gamma=8e-3, **kw)


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("nx,ny", [(33, 70), (64, 64), (153, 152), (200, 313), (460, 150)])
@pytest.mark.parametrize("kind", ["attraction", "rooms", "species", "pairwise"])
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


@pytest.mark.parametrize("kind", ["attraction", "species", "pairwise"])
def test_stop_rule_of_the_persistent_form(kind):
    """Converged, budget-bound and stalled steps report the same pairs, status and
    residual as the kernels per pass."""
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = problem(kind, 48, 40)
    for kw in (dict(tol=1e-6, max_iter=2000), dict(tol=1e-13, max_iter=3000, stall=3),
               dict(tol=0.0, max_iter=1)):
        infos = []
        for loop in (2, 0):
            h = jko.create_from_problem(pb, precision=jko.Precision.FP64, loop=loop, **kw)
            p0 = torch.tensor(pb.q0, dtype=torch.float64, device="cuda")
            infos.append(jko.jko_flow(h, p0, 2)[2])
            jko.jko_destroy(h)
        for a, b in zip(*infos):
            if "stall" not in kw:     # where it stalls is decided by rounding
                assert (a["iters"], a["status"]) == (b["iters"], b["status"]), kw
            # sums of at most ~6e3 terms, each with rounding ~1e-16 of masses below 1
            assert abs(a["residual_l1"] - b["residual_l1"]) <= 1e-12
