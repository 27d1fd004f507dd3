"""Source grids so coarse that thousands of rays share a cell: the placement of
the rays by cell takes about as long as for a fine grid, and the results are
the oracle's.

The bound on the ray trace's time: one cell's atomics (16384 rays at some 10
clocks, twice) and its sort (105 steps of 8 comparisons a thread) come to about
0.25 ms; a sort that is quadratic in the cell's rays takes 200 ms."""
import numpy as np
import pytest
import torch

import synth
from oracle.solve import eval_candidate
from synth import Geometry, REG_IDENTITY

from .helpers import device_problem, make_problem
from .test_gpu_parity import _lam_t, _lens_t, ctx32, ctx64, mods  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sx,sy", [(2, 2), (3, 2), (2, 9), (5, 6), (12, 12)])
@pytest.mark.parametrize("n,sub", [(33, 1), (64, 2), (40, 3)])
def test_crowded_cells(mods, ctx32, ctx64, sx, sy, n, sub):
    # cells of tens to 14400 and 16384 rays; two runs, the same bits
    g = Geometry(n, n, 1.5 / n, sx, sy, -1.0, 1.0, -1.0, 1.0, 5, sub, REG_IDENTITY)
    prob = make_problem(g, seed=11, psf_sigma=1.0)
    lens, lams = np.array([0.05, 0.8, 0.3, 0.0, 0.0, 0.0, 0.0]), synth.lambda_grid(2, 1.0, 1e1)
    p = device_problem(prob, torch.float64)
    run = lambda ctx, p, tol: ctx.eval_batch([p], _lens_t([lens]), [0], _lam_t(lams, 1), [2], tol=tol, maxit=50000,
                                             want_all_x=True, phase_timing=True)
    a, b = run(ctx64, p, 1e-12), run(ctx64, p, 1e-12)
    torch.cuda.synchronize()
    assert ctx64.phase_ms()[0] < 3.0
    for key in a:
        assert torch.equal(a[key], b[key]), key
    r = eval_candidate(prob, lens, lams)
    np.testing.assert_allclose(a["chi2"][0].cpu().numpy(), r.chi2, rtol=1e-9)
    c = run(ctx32, device_problem(prob), 1e-6)
    torch.cuda.synchronize()
    assert ctx32.phase_ms()[0] < 3.0
    np.testing.assert_allclose(c["chi2"][0].cpu().numpy(), r.chi2, rtol=1e-4)
