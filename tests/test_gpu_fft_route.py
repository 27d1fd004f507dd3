"""Which calls convolve by FFT: the PSF spectra are a launch of their own, so an
evaluation by FFT has one launch more than the direct one (variant 6).  The
widest PSFs, grids of 128 and both precisions, where the shared memory of the
item kernel is fullest."""
import numpy as np
import pytest
import torch

import synth
from oracle.solve import eval_candidate
from synth import Geometry, REG_LAPLACIAN

from .helpers import device_problem, make_problem
from .test_gpu_parity import _lam_t, _lens_t, ctx32, ctx64, mods  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [23, 61, 63, 65])
@pytest.mark.parametrize("nx,ny", [(64, 64), (33, 40), (96, 90), (20, 24), (100, 70)])
@pytest.mark.parametrize("bits", [32, 64])
def test_wide_psfs_go_by_fft(mods, ctx32, ctx64, nx, ny, k, bits):
    # grids of 64, 128 and 256 points; the oracle's chi^2 in FP64
    ctx, dt = (ctx32, torch.float32) if bits == 32 else (ctx64, torch.float64)
    g = Geometry(nx, ny, 3.2 / max(nx, ny), 9, 8, -0.8, 0.8, -0.8, 0.8, k, 1, REG_LAPLACIAN)
    prob = make_problem(g, seed=5, psf_sigma=k / 6.0)
    p, lams = device_problem(prob, dt), synth.lambda_grid(2, 1.0, 1e1)
    tol = 1e-6 if bits == 32 else 1e-12
    run = lambda **kw: ctx.eval_batch([p], _lens_t([synth.TRUE_LENS]), [0], _lam_t(lams, 1), [2], tol=tol, **kw)
    run(variant=6, maxit=1)
    direct = ctx.launches()
    for variant in (0, 5):
        out = run(variant=variant, maxit=50000)
        assert ctx.launches() == direct + 1, variant
        if bits == 64 and variant == 0 and max(nx, ny) <= 64:
            r = eval_candidate(prob, synth.TRUE_LENS, lams)
            np.testing.assert_allclose(out["chi2"][0].cpu().numpy(), r.chi2, rtol=1e-9)
