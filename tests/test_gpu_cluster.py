"""The cluster CGLS kernel (csrc/cluster.cuh) against the general one-CTA
kernel (variant 4), bit for bit: both add every sum in the same order, so the
comparison is exact.  Sizes at the edges of its cut: bands that end inside a
tile row, more CTAs than some share of the rays fills, PSFs whose halo is a
whole band, several source pixels a thread, staged rays in several passes."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

G, I, L = synth.REG_GRADIENT, synth.REG_IDENTITY, synth.REG_LAPLACIAN


def _problem(ctx, nx, ny, sx, sy, k, reg, seed, masked=False, half=0.8, interp=0):
    from paper_1101_5803_gb300.problems import observe_on_device
    rng = np.random.default_rng(seed)
    g = synth.Geometry(nx, ny, 3.3 / max(nx, ny), sx, sy, -half, half, -half, half, k, 1, reg, interp=interp)
    mask = synth.annular_mask(g, 0.4, 1.3) if masked else None
    return observe_on_device(ctx, g, synth.gaussian_psf(k, max(k / 6.0, 0.4)), synth.drawn_source(rng), synth.TRUE_LENS,
                             rng, mask=mask)


CASES = [  # nx, ny, sx, sy, K, reg, candidates, lambdas, masked
    (128, 128, 48, 48, 11, L, 1, 3, False),
    (128, 128, 48, 48, 11, L, 40, 4, False),
    (97, 83, 31, 40, 7, L, 1, 4, True),
    (97, 83, 31, 40, 7, G, 20, 4, False),
    (131, 45, 17, 19, 5, I, 3, 4, True),
    (45, 131, 48, 13, 15, L, 2, 4, False),
    (112, 100, 64, 50, 21, L, 2, 3, False),
    (150, 150, 90, 96, 3, G, 1, 2, False),
    (64, 64, 32, 32, 15, L, 1, 6, False),
]


@pytest.mark.parametrize("nx,ny,sx,sy,k,reg,n,n_lam,masked", CASES)
def test_cluster_matches_general_kernel(nx, ny, sx, sy, k, reg, n, n_lam, masked):
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    p = _problem(ctx, nx, ny, sx, sy, k, reg, 3, masked)
    rng = np.random.default_rng(7)
    lens = torch.as_tensor(synth.lens_population(rng, n), device="cuda")
    lams = torch.as_tensor(np.tile(synth.lambda_grid(n_lam, 0.3, 1e2), (n, 1)), device="cuda")
    warm = torch.rand((n, n_lam, sx * sy), device="cuda")
    for kw in ({}, {"lam_start": np.full(n, n_lam // 2, np.int32)}, {"warm_x": warm},
               {"mode": binding.MIRAGE_MODE_PLAIN}, {"use_graph": True}):
        a = ctx.eval_batch([p], lens, np.zeros(n), lams, np.full(n, n_lam), want_all_x=True, **kw)
        b = ctx.eval_batch([p], lens, np.zeros(n), lams, np.full(n, n_lam), want_all_x=True, variant=4, **kw)
        torch.cuda.synchronize()
        for key in a:
            assert torch.equal(a[key], b[key]), (key, kw.keys())
        assert (a["item_status"] & (binding.ST_MAXIT | binding.ST_BREAKDOWN)).max().item() == 0
    ctx.close()


def test_cluster_statuses_and_mixed_batch():
    """Bad and empty candidates beside good ones, problems of several kernels
    in one call, nearest-neighbour rays, and a few reserved slots."""
    from paper_1101_5803_gb300 import binding
    ctx = binding.Context(0, binding.MIRAGE_FP32)
    probs = [_problem(ctx, 128, 128, 48, 48, 11, L, 1), _problem(ctx, 64, 64, 32, 32, 7, L, 2),
             _problem(ctx, 96, 80, 40, 48, 15, L, 3, True), _problem(ctx, 100, 100, 33, 35, 9, G, 4, interp=1),
             _problem(ctx, 128, 128, 48, 48, 7, L, 5)]
    probs[4].mask.zero_()
    n, ml = 10, 4
    rng = np.random.default_rng(9)
    lens = synth.lens_population(rng, n)
    lens[3, 1] = 2.0  # axis ratio out of range
    idx = np.arange(n, dtype=np.int32) % 5
    nl = np.array([4, 3, 4, 4, 4, 2, 4, 1, 4, 3], np.int32)
    lams = np.tile(synth.lambda_grid(ml, 1.0, 1e2), (n, 1))
    args = (probs, torch.as_tensor(lens, device="cuda"), idx, torch.as_tensor(lams, device="cuda"), nl)

    def outputs():
        z = lambda shape, dt: torch.zeros(shape, dtype=dt, device="cuda")  # noqa: E731
        return {"chi2": z((n, ml), torch.float64), "reg": z((n, ml), torch.float64), "iters": z((n, ml), torch.int32),
                "relres": z((n, ml), torch.float64), "item_status": z((n, ml), torch.int32),
                "corner": z((n,), torch.int32), "status": z((n,), torch.int32), "kappa": z((n, ml), torch.float64),
                "s": z((n, 48 * 48), torch.float32), "all_x": z((n, ml, 48 * 48), torch.float32)}

    a = ctx.eval_batch(*args, out=outputs())
    ctx.reserve_slots(8)
    c = ctx.eval_batch(*args, out=outputs())
    ctx.reserve_slots(0)
    torch.cuda.synchronize()
    for key in a:
        assert torch.equal(a[key], c[key]), key
    assert a["status"][3].item() & binding.ST_BAD_PARAM and a["status"][4].item() & binding.ST_EMPTY_MAP
    for i in range(n):  # each candidate as in a call of its own
        one = ctx.eval_batch([probs[idx[i]]], args[1][i:i + 1], [0], args[3][i:i + 1], nl[i:i + 1],
                             variant=0 if idx[i] == 1 else 4)
        m = nl[i]
        for key in ("chi2", "reg", "iters", "relres", "item_status"):
            assert torch.equal(one[key][0, :m], a[key][i, :m]), (i, key)
    ctx.close()
