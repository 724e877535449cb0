"""The FP32 CG kernels: columns shorter than a block and longer than a sweep of the grid, odd
lengths, one to many right-hand sides, a zero column, with and without the preconditioner."""
import math

import numpy as np
import pytest

RTOL = 1e-8


def residual_norms(ctx, kry, cov, B, X):
    e64 = ctx.embed(cov, kry.KRY_F64)
    row_sum = float(ctx.matvec(e64, B.new_ones((1, B.shape[1]))).max())
    return (B - ctx.matvec(e64, X)).norm(dim=1), row_sum


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nrhs", [(4, 4, 1), (5, 7, 3), (46, 45, 200), (362, 362, 1), (363, 363, 9), (257, 256, 10),
                                        (181, 181, 40), (1024, 1024, 2), (1025, 1024, 2)])
def test_residuals_and_iteration_counts(n1, n2, nrhs):
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    cov = I.Cov(1.0, 1.0 / max(n1, n2), 0.5, 1.0)
    mask = np.random.default_rng(n1).random((n1, n2)) >= 0.1
    mask[0, 0] = True
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    B = torch.randn((nrhs, p), generator=torch.Generator().manual_seed(n1 + nrhs), dtype=torch.float64)
    if nrhs > 2:
        B[1] = 0.0
    B = B.cuda()
    X, iters, relres, st = ctx.solve(ctx.embed(cov, kry.KRY_F32), B, rtol=RTOL, maxit=2000)
    rn, kappa = residual_norms(ctx, kry, cov, B, X)   # tau2 = 1: the largest row sum bounds the condition number
    assert st == kry.KRY_OK
    run = [k for k in range(nrhs) if nrhs <= 2 or k != 1]
    # the solver judges this same FP64 residual; 1e-3 covers the matvec's own rounding (1e-15 ||K|| ||x|| against 1e-8 ||b||)
    assert bool(torch.all(rn[run] <= RTOL * 1.001 * B[run].norm(dim=1)))
    if nrhs > 2:
        assert bool(torch.all(X[1] == 0))
    # CG's bound, with a block of 8 more after each of the (at most 9) replacements
    assert iters <= 0.5 * math.sqrt(kappa) * math.log(2.0 * kappa / RTOL) + 8 * 9
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nrhs", [(96, 81, 1), (128, 128, 7), (240, 333, 3)])
def test_preconditioned_residuals(n1, n2, nrhs):
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    cov = I.Cov(1.0, 0.1, 1.5, 0.05)
    mask = I.mask_circles(n1, n2, 0.4, 11)
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    B = torch.randn((nrhs, p), generator=torch.Generator().manual_seed(n1 + nrhs), dtype=torch.float64).cuda()
    emb = ctx.embed(cov, kry.KRY_F32)
    plain, pre = (ctx.solve(emb, B, rtol=1e-6, maxit=40000, precond=c) for c in (False, True))
    for X, it, rr, st in (plain, pre):
        assert st == kry.KRY_OK
        rn, _ = residual_norms(ctx, kry, cov, B, X)
        assert bool(torch.all(rn <= 1e-6 * 1.001 * B.norm(dim=1)))
    assert pre[1] < plain[1]
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("ncov,settings", [(1, 600), (8, 900)])
def test_search_of_many_columns(ncov, settings):
    """Batches past 1024 columns (a block's most threads) and past 8192 (the host flags' first size):
    every setting's result is the one that it has alone."""
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    n1, n2 = 12, 10
    g = torch.Generator().manual_seed(ncov)
    mask = np.random.default_rng(3).random((n1, n2)) >= 0.2
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    y = torch.randn(p, generator=g, dtype=torch.float64).cuda()
    X = torch.randn((ncov, p), generator=g, dtype=torch.float64).cuda()
    thetas = [I.Cov(1.0, 0.05 + 0.1 * k / settings, 0.5, 0.3) for k in range(settings)]
    opts = kry.Opts(prec=kry.KRY_F32, nprobe=2, nsteps=10, seed=1, rtol=RTOL, maxit=200, reorth=1)
    assert settings * ((ncov + 2) & ~1) > (1024 if ncov == 1 else 8192)   # columns [y, X] in pairs
    r = ctx.profile_loglik(y, X, thetas, opts)
    assert r["status"] == kry.KRY_OK
    for k in (0, settings // 2, settings - 1):
        one = ctx.profile_loglik(y, X, [thetas[k]], opts)
        # solves to 1e-8 of a system of condition number below 100, at most 9 columns: 1e-5 of the quadratic form
        assert abs(r["loglik"][k] - one["loglik"][0]) <= 1e-5 * abs(one["loglik"][0]) + 1e-5
        assert abs(r["logdet"][k] - one["logdet"][0]) <= 1e-5 * p
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nrhs", [(600, 90, 3), (40, 520, 2), (300, 300, 1), (64, 64, 12), (20, 20, 2)])
@pytest.mark.parametrize("cells", [0.05, 0.3, 0.7])
@pytest.mark.parametrize("precond", [False, True])
def test_systems_that_converge_within_a_block_of_iterations(n1, n2, nrhs, cells, precond):
    """Ranges below a cell: the recursive residual passes FP32's resolution before the first replacement."""
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    cov = I.Cov(1.0, cells / max(n1, n2), 0.5, 0.5)
    mask = np.random.default_rng(n1).random((n1, n2)) >= 0.2
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    B = torch.randn((nrhs, p), generator=torch.Generator().manual_seed(n2), dtype=torch.float64).cuda()
    X, iters, _, st = ctx.solve(ctx.embed(cov, kry.KRY_F32), B, rtol=RTOL, maxit=500, precond=precond)
    assert st == kry.KRY_OK
    rn, kappa = residual_norms(ctx, kry, cov, B, X)   # the largest row sum over tau2 bounds the condition number
    assert bool(torch.all(rn <= RTOL * 1.001 * B.norm(dim=1)))
    # CG's bound, with a block of 8 more after each of the (at most 9) replacements
    assert iters <= 0.5 * math.sqrt(kappa / 0.5) * math.log(2.0 * kappa / 0.5 / RTOL) + 8 * 9
    ctx.close()
