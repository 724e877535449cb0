"""Gauss quadrature of the Lanczos tridiagonal by the resolvent rule: its formula
against eigendecompositions (no GPU), and the kernel against the oracle at the
ends of its range (one step, the largest step count, no lower bound)."""
import math

import numpy as np
import pytest


def resolvent_rule(a, b, lb):
    """The kernel's rule: nodes of step 1/2 in u = log s, corrections below lb; None where it leaves
    the matrix to the eigenvalue iteration."""
    n, b2 = len(a), b * b
    r = np.abs(a) + np.concatenate([[0.0], np.abs(b)]) + np.concatenate([np.abs(b), [0.0]])
    u0 = math.log(lb) - 47.0
    span = math.log(r.max()) + 40.0 - u0
    s = np.exp(u0 + 0.5 * np.arange(math.ceil(2.0 * span) + 1))
    g = a[-1] + s
    for i in range(n - 2, -1, -1):
        g = (a[i] + s) - b2[i] / g
    f = math.log(lb) + 0.5 * np.sum(s / (lb + s) - s / g)
    th = np.linalg.eigvalsh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    for x in th[th < lb]:
        gi, dg = a[-1] - x, 1.0
        for i in range(n - 2, -1, -1):
            q = b2[i] / gi
            dg = 1.0 + q / gi * dg
            gi = (a[i] - x) - q
        if not abs(gi) <= 2.0 ** -44 * r.max() * dg:
            return None
        f += (math.log(lb) - math.log(x)) / dg
    return f


@pytest.mark.parametrize("n,below", [(1, 0), (2, 0), (2, 1), (7, 2), (50, 0), (50, 3), (120, 9)])
def test_rule_is_the_clamped_gauss_quadrature(n, below):
    r = np.random.default_rng(n + 100 * below)
    a, b = 1.0 + 5.0 * r.random(n), 0.4 * r.random(max(n - 1, 0))
    th, U = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    lb = th[0] * 0.9 if below == 0 else (0.5 * (th[below - 1] + th[below]) if below < n else th[-1] * 1.1)
    ref = np.sum(U[0] ** 2 * np.log(np.maximum(th, lb)))
    # log lb and the ~200 terms are of order one: 1e-13 absolute
    f = resolvent_rule(a, b, lb)
    if f is None:   # localised eigenvectors, whose weight on e1 is far below rounding
        assert np.min(U[0, th < lb] ** 2) < 1e-20
    else:
        assert abs(f - ref) <= 1e-13


@pytest.mark.gpu
@pytest.mark.parametrize("nsteps,tau2,nprobe", [(1, 0.1, 3), (2, 0.1, 1), (40, 0.1, 65), (40, 0.0, 2), (256, 0.3, 2)])
def test_kernel_at_the_ends_of_its_range(nsteps, tau2, nprobe):
    import torch

    from oracle import kryoracle as O
    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    n1, n2 = 24, 20
    cov = I.Cov(1.0, 0.03, 0.5, tau2)
    mask = I.mask_uniform(n1, n2, 0.3, 7)
    ctx = kry.Context(0)
    ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    emb = ctx.embed(cov, kry.KRY_F64)
    _, _, per = ctx.logdet(emb, nprobe, nsteps, 5, reorth=1)
    ref = O.FFTProblem(n1, n2, mask, cov).logdet(nprobe, nsteps, 5, reorth=True)[2]
    # FP64 Lanczos and eigenvalues at a condition number below 100: 1e-10 relative to the spread of log theta
    assert np.max(np.abs(per - ref)) <= 1e-10 * mask.sum()
    ctx.close()
