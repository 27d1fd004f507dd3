"""Which kernel the automatic choice gives a call's items: the general kernel or
the cluster kernel on 1, 2, 4 or 8 SMs.  A cluster of eight SMs shortens one
item's iterations and takes several times the SM time for them, so a call
with many items a SM must not go to it."""
import numpy as np
import pytest
import torch

import synth

from .test_gpu_cluster import L, _problem

pytestmark = pytest.mark.gpu


def _kernels(shapes, n, n_lam, maxit=1, **kw):
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    probs = [_problem(ctx, *shape, L, 3) for shape in shapes]
    lens = torch.as_tensor(synth.lens_population(np.random.default_rng(7), n), device="cuda")
    lams = torch.as_tensor(np.tile(synth.lambda_grid(n_lam, 1e-2, 1e2), (n, 1)), device="cuda")
    ctx.eval_batch(probs, lens, np.arange(n) % len(probs), lams, np.full(n, n_lam), maxit=maxit, **kw)
    out = ctx.item_kernels()
    assert sum(out.values()) == n * n_lam
    ctx.close()
    return out


@pytest.mark.parametrize("shape,n", [((64, 64, 32, 32, 15), 64), ((48, 48, 48, 48, 11), 40), ((100, 100, 30, 30, 3), 100),
                                     ((64, 64, 32, 32, 15), 1000), ((36, 36, 28, 28, 13), 55), ((100, 100, 36, 36, 9), 64)])
def test_full_calls_keep_off_wide_clusters(shape, n):
    # 64 x 64, K = 15, 64 candidates x 8 lambdas: 23 ms without clusters of eight, 47 with
    k = _kernels([shape], n, 8)
    assert k["cluster8"] == k["cluster4"] == 0, k


@pytest.mark.parametrize("shape", [(128, 128, 48, 48, 11), (100, 100, 36, 36, 9), (64, 64, 32, 32, 13)])
def test_single_candidates_run_on_clusters(shape):
    k = _kernels([shape], 1, 6)
    assert k["direct"] == 0 and k["cluster4"] + k["cluster8"] > 0, k


def test_options_that_name_a_kernel():
    s, f = (96, 96, 48, 48, 11), (64, 64, 32, 32, 9)
    assert _kernels([s], 2, 3, variant=4)["direct"] == 6
    assert _kernels([s], 2, 3, variant=5)["fft"] == 6
    assert _kernels([s], 2, 3, place=3)["direct"] == 6
    assert _kernels([f], 2, 3)["two_cta"] == 6
    assert _kernels([f, (48, 48, 24, 24, 33)], 4, 3)["fft"] == 6
    assert _kernels([f], 2, 3, use_graph=True)["two_cta"] == 6
