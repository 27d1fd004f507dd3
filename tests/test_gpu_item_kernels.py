"""Which kernel the automatic choice gives a call's items: the general kernel or
the cluster kernel on 1, 2, 4 or 8 SMs.  A cluster of eight SMs shortens one
item's iterations and takes several times the SM time for them, so a call
with many items a SM must not go to it."""
import numpy as np
import pytest
import torch

import synth

from .test_gpu_cluster import G, I, L, _problem

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


KEYS = ("chi2", "reg", "iters", "relres", "item_status", "corner", "status", "kappa", "all_x")


@pytest.mark.parametrize("shape,n,ran", [
    ((64, 64, 32, 32, 15, L), 12, ["cluster1", "cluster8"]),     # CTAs of 256 threads
    ((60, 44, 24, 27, 13, G), 100, ["cluster1"]),
    ((48, 40, 33, 31, 3, I), 4, ["cluster8"]),                   # L^T ray by ray
    ((64, 64, 60, 62, 21, L), 200, ["cluster1", "cluster2"]),
    ((100, 100, 36, 36, 9, L), 100, ["cluster1"]),               # CTAs of 512
    ((72, 72, 36, 36, 13, L), 100, ["cluster2"]),
    ((64, 64, 60, 62, 21, L), 100, ["cluster2"]),                # ray by ray, more rays than are staged
    ((131, 45, 17, 19, 5, I), 40, ["cluster2"]),
    ((128, 128, 48, 48, 11, L), 200, ["cluster2"]),              # 512
    ((128, 128, 48, 48, 11, L), 40, ["cluster4"]),
    ((32, 32, 16, 16, 13, L), 1, ["cluster4"]),
    ((200, 200, 96, 96, 15, L), 40, ["cluster4"]),               # 512
    ((97, 83, 31, 40, 7, G), 1, ["cluster8"]),
    ((200, 200, 96, 96, 15, L), 4, ["cluster8"]),                # 512
])
def test_every_cluster_size_gives_the_general_kernels_bits(shape, n, ran):
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    p = _problem(ctx, *shape, 3)
    lens = torch.as_tensor(synth.lens_population(np.random.default_rng(7), n), device="cuda")
    lams = torch.as_tensor(np.tile(synth.lambda_grid(3, 1.0, 1e2), (n, 1)), device="cuda")
    run = lambda v: ctx.eval_batch([p], lens, np.zeros(n), lams, np.full(n, 3), want_all_x=True, variant=v)  # noqa: E731
    a = run(0)
    k = ctx.item_kernels()
    assert all(k[r] for r in ran) and sum(k[r] for r in ran) == 3 * n, k
    b = run(4)
    assert ctx.item_kernels()["direct"] == 3 * n
    for key in KEYS:
        assert torch.equal(a[key], b[key]), key
    ctx.close()


@pytest.mark.parametrize("n", [8, 80])
def test_groups_side_by_side_or_in_turn(n):
    # four PSF widths of the two-CTA kernel in one call: with few items their
    # launches share the device (two a group), with many each takes all of it
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    probs = [_problem(ctx, 64, 64, 32, 32, k, L, k) for k in (5, 7, 9, 11)]
    lens = torch.as_tensor(synth.lens_population(np.random.default_rng(7), n), device="cuda")
    lams = torch.as_tensor(np.tile(synth.lambda_grid(12, 1.0, 1e2), (n, 1)), device="cuda")
    idx, nl = np.arange(n) % 4, np.full(n, 12)
    a = ctx.eval_batch(probs, lens, idx, lams, nl, want_all_x=True)
    launches = ctx.launches()
    assert ctx.item_kernels()["two_cta"] == 12 * n
    assert launches > 7 if n == 8 else launches == 2 + 4 + 1
    for i in range(4):  # each problem in a call of its own
        one = ctx.eval_batch([probs[i]], lens[i::4].contiguous(), [0] * (n // 4), lams[i::4].contiguous(), nl[i::4],
                             want_all_x=True, variant=1)
        for key in KEYS:
            assert torch.equal(a[key][i::4], one[key]), key
    ctx.close()


def test_short_chained_calls_run_on_wide_clusters():
    # a chain holds several lambdas: 12 candidates at 128 x 128 take 175 ms on clusters
    # of four, where their items one by one would go, and 115 on clusters of eight
    k = _kernels([(128, 128, 48, 48, 11)], 12, 16, lam_start=np.full(12, 8, np.int32))
    assert k["cluster8"] == 192, k
