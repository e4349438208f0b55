"""The FFT form's passes over all transform lengths: odd and even log2 L, lines
that fill at most half of L and more, two and four columns a block, an odd number
of columns, the shortest lines.  One pair of the blur p = xi(q / xi 1) against the
band-limited filter on the same grid.  Bar: the transforms are accurate normwise,
~eps log2(L) of a line's largest entry per pass, four passes, and the blur's own values
stay within a few e-folds of it: 100 eps log2(L) covers them (FP64 3e-13, FP32
1e-4 at most); the bars of the oracle comparison, 1e-12 and 1e-5, are kept."""
import math

import numpy as np
import pytest

from paper_1502_06216_gb300 import inputs
from tests.gpu_util import need_gpu, rel_l1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,bar", [("FP64", 1e-12), ("FP32", 1e-5)])
@pytest.mark.parametrize("nx,ny,gamma", [(1, 8, 2e-2), (2, 3, 2e-1), (7, 5, 2e-2), (16, 9, 2e-3),
                                         (33, 64, 2e-2), (64, 401, 2e-3), (403, 100, 2e-2),
                                         (512, 70, 2e-2), (700, 405, 5e-4)])
def test_one_pair_equals_the_band_filter(nx, ny, gamma, prec, bar):
    torch = need_gpu()
    from paper_1502_06216_gb300 import jko
    pb = inputs.crowd_problem(nx, ny=ny, gamma=gamma, tau=0.02)
    q = np.random.default_rng(nx + ny).uniform(0.5, 1.0, pb.N)
    pb.q0, pb.w, pb.kappa = q / q.sum(), None, math.inf
    out = []
    for fft in (0, 1):
        h = jko.create_from_problem(pb, precision=jko.Precision[prec], tol=0.0, max_iter=1,
                                    renormalize=False, fft=fft)
        p0 = torch.tensor(pb.q0, dtype=h.dtype, device="cuda")
        out.append(jko.jko_step(h, p0)[0].double().cpu().numpy())
        jko.jko_destroy(h)
    err = rel_l1(out[1], out[0])
    print(prec, nx, ny, gamma, err)
    assert err <= bar
