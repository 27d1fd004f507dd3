"""Pixels without a finite value, in the cluster kernel and the general one.

An unusable pixel's weight is zero, but zero times a NaN or an infinity is a
NaN: a data value that is not finite makes chi^2 a NaN wherever the pixel
lies, and the solve as well when a mapped pixel sees it through the PSF.  The
cluster kernel convolves only tiles that hold a mapped pixel, and has to say
the same."""
import numpy as np
import pytest
import torch

import synth

from .test_gpu_cluster import G, L, _problem

pytestmark = pytest.mark.gpu


def _bits(t):
    t = t.detach().clone()
    if t.is_floating_point():
        t[torch.isnan(t)] = float("nan")  # one NaN
        t = t.view(torch.int64 if t.dtype == torch.float64 else torch.int32)
    return t


@pytest.mark.parametrize("nx,ny,sx,sy,k,reg,half,n", [
    (128, 128, 48, 48, 11, L, 0.8, 1),
    (128, 128, 48, 48, 11, L, 0.3, 1),  # few mapped pixels: empty tile rows above and below
    (97, 83, 31, 40, 7, G, 0.5, 2),
    (64, 64, 60, 62, 21, L, 0.4, 1),
])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("where", ["corner", "row", "masked", "none"])
def test_values_that_are_not_finite(nx, ny, sx, sy, k, reg, half, n, value, where):
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    p = _problem(ctx, nx, ny, sx, sy, k, reg, 3, masked=True, half=half)
    y, x = {"corner": (0, 0), "row": (ny - 1, nx // 2), "masked": (ny // 2, nx // 2), "none": (0, 0)}[where]
    p.mask.view(ny, nx)[y, x] = 0
    if where != "none":
        p.d.view(ny, nx)[y, x] = value
    lens = torch.as_tensor(synth.lens_population(np.random.default_rng(7), n), device="cuda")
    lams = torch.as_tensor(np.tile(synth.lambda_grid(3, 0.3, 1e2), (n, 1)), device="cuda")
    run = lambda v: ctx.eval_batch([p], lens, np.zeros(n), lams, np.full(n, 3), want_all_x=True, variant=v)  # noqa: E731
    a, b = run(0), run(4)
    assert bool(torch.isnan(b["chi2"]).all()) == (where != "none")
    for key in a:
        assert torch.equal(_bits(a[key]), _bits(b[key])), key
    ctx.close()
