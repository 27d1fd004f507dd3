"""Kernel variants that a batch's or an image's size selects, at the edges of
their ranges: where two variants add every sum in the same order they are
compared bit for bit, otherwise with the oracle under the parity tests' gates.
"""
import numpy as np
import pytest
import torch

import synth
from oracle.solve import eval_candidate, forward_chi2
from synth import Geometry, REG_GRADIENT, REG_IDENTITY, REG_LAPLACIAN

from .helpers import device_problem, make_problem
from .test_gpu_parity import _fp32_checks, _lam_t, _lens_t, ctx32, ctx64, mods  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu

KEYS = ("chi2", "reg", "iters", "relres", "item_status", "corner", "status", "kappa", "all_x")


def _same(one, many, n):
    """Every candidate of ``many`` (n copies of one candidate) as in ``one``."""
    for key in KEYS:
        a = one[key][0]
        for i in range(n):
            assert torch.equal(a, many[key][i]), (key, i)


@pytest.mark.parametrize("variant", [0, 1, 2, 3])
@pytest.mark.parametrize("nx,ny,sx,sy,k,reg,masked", [
    (64, 64, 32, 32, 9, REG_LAPLACIAN, False),
    (64, 64, 32, 32, 9, REG_LAPLACIAN, True),
    (61, 47, 31, 29, 7, REG_GRADIENT, True),
    (33, 50, 17, 11, 5, REG_IDENTITY, False),
])
def test_few_items_and_many_same_bits(mods, ctx32, variant, nx, ny, sx, sy, k, reg, masked):
    # one candidate (its CTAs have an SM each) and 64 copies of it (two CTAs per SM)
    g = Geometry(nx, ny, 3.2 / max(nx, ny), sx, sy, -0.8, 0.8, -0.8, 0.8, k, 1, reg)
    prob = make_problem(g, seed=3, mask=synth.annular_mask(g, 0.4, 1.3) if masked else None)
    p, lams, n = device_problem(prob), synth.lambda_grid(4, 1e-1, 1e1), 64
    run = lambda n, **kw: ctx32.eval_batch([p], _lens_t([synth.TRUE_LENS] * n), [0] * n, _lam_t(lams, n), [4] * n,
                                           want_all_x=True, variant=variant, **kw)
    _same(run(1), run(n), n)
    _same(run(1), run(3, mode=mods.MIRAGE_MODE_PLAIN), 3)


@pytest.mark.parametrize("nx,ny,sx,sy,k,sub,masked", [
    (32, 32, 16, 16, 5, 1, False),
    (23, 29, 11, 13, 7, 1, True),
    (37, 18, 12, 9, 3, 2, False),
    (13, 11, 5, 6, 9, 1, False),
])
def test_fp64_few_items_and_many_same_bits(mods, ctx64, nx, ny, sx, sy, k, sub, masked):
    # 160 copies x 8 lambdas have two CTAs per SM; both against the oracle's chi^2
    g = Geometry(nx, ny, 3.2 / max(nx, ny), sx, sy, -0.8, 0.8, -0.8, 0.8, k, sub, REG_GRADIENT)
    prob = make_problem(g, seed=4, psf_sigma=1.0, mask=synth.annular_mask(g, 0.4, 1.4) if masked else None)
    p, lams, n = device_problem(prob, torch.float64), synth.lambda_grid(8, 1e-1, 1e1), 160
    run = lambda n: ctx64.eval_batch([p], _lens_t([synth.TRUE_LENS] * n), [0] * n, _lam_t(lams, n), [8] * n,
                                     want_all_x=True, tol=1e-12, maxit=50000)
    one = run(1)
    _same(one, run(n), n)
    r = eval_candidate(prob, synth.TRUE_LENS, lams)
    np.testing.assert_allclose(one["chi2"][0].cpu().numpy(), r.chi2, rtol=1e-9)


@pytest.mark.parametrize("nx,ny,k", [(31, 27, 33), (33, 29, 3), (51, 37, 33), (64, 64, 65), (65, 45, 25)])
def test_fft_grids_in_shared_memory(mods, ctx32, ctx64, nx, ny, k):
    # grid sides 64 and 128, their fullest and emptiest images, FP32 and FP64
    g = Geometry(nx, ny, 3.2 / max(nx, ny), 15, 14, -0.8, 0.8, -0.8, 0.8, k, 1, REG_LAPLACIAN)
    prob = make_problem(g, seed=5, psf_sigma=min(3.0, k / 4.0))
    lams = synth.lambda_grid(4, 1e-2, 1e1)
    out = ctx32.eval_batch([device_problem(prob)], _lens_t([synth.TRUE_LENS]), [0], _lam_t(lams, 1), [4], tol=1e-6,
                           want_all_x=True, variant=5)
    _fp32_checks(out, prob, [synth.TRUE_LENS], lams, 1e-6)
    out = ctx64.eval_batch([device_problem(prob, torch.float64)], _lens_t([synth.TRUE_LENS]), [0], _lam_t(lams, 1), [4],
                           tol=1e-12, maxit=50000, variant=5)
    r = eval_candidate(prob, synth.TRUE_LENS, lams)
    np.testing.assert_allclose(out["chi2"][0].cpu().numpy(), r.chi2, rtol=1e-9)


@pytest.mark.parametrize("k", range(3, 23, 2))
@pytest.mark.parametrize("nx,ny,sub", [(97, 69, 1), (42, 55, 2)])
def test_forward_every_compiled_psf(mods, ctx32, k, nx, ny, sub):
    g = Geometry(nx, ny, 3.2 / max(nx, ny), 31, 24, -0.8, 0.8, -0.7, 0.7, k, sub, REG_LAPLACIAN)
    prob = make_problem(g, seed=6, psf_sigma=max(k / 6.0, 0.5))
    S = np.random.default_rng(7).uniform(0, 1, (3, g.ns))
    m_o, c_o = forward_chi2(prob, synth.TRUE_LENS, S)
    m_g, c_g, st = ctx32.forward(device_problem(prob), _lens_t(synth.TRUE_LENS)[0],
                                 torch.as_tensor(S, dtype=torch.float32, device="cuda"))
    assert int(st.item()) == 0
    assert np.abs(m_g.double().cpu().numpy() - m_o).max() <= 2e-6 * np.abs(m_o).max()
    np.testing.assert_allclose(c_g.cpu().numpy(), c_o, rtol=1e-4)


@pytest.mark.parametrize("n", [1, 40])
@pytest.mark.parametrize("nx,ny,sx,sy,k,reg", [
    (48, 48, 48, 48, 11, REG_LAPLACIAN),
    (48, 40, 33, 31, 3, REG_IDENTITY),
    (64, 64, 60, 62, 21, REG_LAPLACIAN),  # more rays than are staged
    (96, 83, 70, 61, 7, REG_GRADIENT),
])
def test_cluster_sources_as_fine_as_the_image(mods, ctx32, n, nx, ny, sx, sy, k, reg):
    # the cluster kernel's ray-by-ray form of L^T against the general kernel's (variant 4)
    g = Geometry(nx, ny, 3.2 / max(nx, ny), sx, sy, -0.8, 0.8, -0.8, 0.8, k, 1, reg)
    p = device_problem(make_problem(g, seed=8, psf_sigma=max(k / 6.0, 0.5)))
    lens = _lens_t(synth.lens_population(np.random.default_rng(9), n))
    lams = synth.lambda_grid(3, 1.0, 1e2)
    run = lambda v: ctx32.eval_batch([p], lens, [0] * n, _lam_t(lams, n), [3] * n, want_all_x=True, variant=v)
    a, b = run(0), run(4)
    for key in KEYS:
        assert torch.equal(a[key], b[key]), key


@pytest.mark.parametrize("n", [1, 24])
@pytest.mark.parametrize("nx,ny,sx,sy,k", [(32, 32, 16, 16, 13), (24, 20, 9, 24, 13), (28, 36, 24, 17, 15)])
def test_cluster_few_rays(mods, nx, ny, sx, sy, k, n):
    # fewer rays than threads in a CTA, and rays in the first source cell: a
    # fresh context (its work space is zeros where the driver hands out zeros)
    # and a used one against the general kernel (variant 4)
    g = Geometry(nx, ny, 1.5 / max(nx, ny), sx, sy, -0.7, 0.7, -0.7, 0.7, k, 1, REG_LAPLACIAN)
    prob = make_problem(g, seed=10, psf_sigma=2.0)
    lens = np.tile(np.array([0.02, 0.8, 0.3, 0.0, 0.0, 0.0, 0.0]), (n, 1))
    lams = synth.lambda_grid(2, 1e-2, 1.0)
    ctx = mods.Context(0, mods.MIRAGE_FP32)
    p = device_problem(prob)
    run = lambda v: ctx.eval_batch([p], _lens_t(lens), [0] * n, _lam_t(lams, n), [2] * n, want_all_x=True, variant=v)
    outs = [run(0), run(0), run(4), run(0)]
    for key in KEYS:
        for o in outs:
            assert torch.equal(o[key], outs[2][key]), key
    ctx.close()
