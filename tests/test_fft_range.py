"""Matvecs over the range of their precision: a power of two in the input is one in the output, also where the
forward transforms' values come near the largest number (FP32 results stay below 2^118)."""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2", [(20, 30), (32, 32), (64, 33), (40, 100), (128, 200), (256, 31), (300, 512), (512, 600),
                                   (1000, 90), (70, 1024), (2048, 40), (50, 2000), (4096, 33), (36, 4000)])
def test_power_of_two_of_the_input(n1, n2):
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    ctx = kry.Context(0)
    mask = np.random.default_rng(n1).random((n1, n2)) >= 0.3
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    emb = ctx.embed(I.Cov(1.0, 0.1, 0.5, 0.1), kry.KRY_F32)
    # random, and constant: its sum over the grid, at most 2^18, is the largest value of any transform
    V = torch.randn((3, p), generator=torch.Generator().manual_seed(n2)).clamp(-4, 4)
    V[2] = 1.0
    V = V.cuda()
    out = ctx.matvec(emb, V)
    # |re| + |im| of a pair's values and a third bit for the butterflies' sums; results below 2^116
    k = min(126 - int(np.ceil(np.log2(n1 * n2))) - 3, 116 - int(np.ceil(np.log2(float(out.abs().max())))))
    big = ctx.matvec(emb, V * 2.0 ** k)
    assert bool(torch.isfinite(big).all())
    assert torch.equal(big, out * 2.0 ** k)
    ctx.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2", [(4, 5), (20, 30), (32, 32), (64, 33), (40, 100), (256, 31), (300, 512), (1000, 90),
                                   (70, 1024), (2048, 40), (50, 2000), (4096, 33), (36, 4000)])
def test_power_of_two_of_the_input_f64(n1, n2):
    """FP64: values of any transform and results below 2^1012."""
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    ctx = kry.Context(0)
    mask = np.random.default_rng(n1).random((n1, n2)) >= 0.3
    mask[0, 0] = True
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    emb = ctx.embed(I.Cov(1.0, 0.1, 0.5, 0.1), kry.KRY_F64)
    V = torch.randn((3, p), generator=torch.Generator().manual_seed(n2), dtype=torch.float64).clamp(-4, 4)
    V[2] = 1.0
    V = V.cuda()
    out = ctx.matvec(emb, V)
    # 4 times the sum over the grid, |re| + |im| of a pair and a bit for the butterflies' sums; results likewise
    k = min(1012 - int(np.ceil(np.log2(n1 * n2))) - 4, 1010 - int(np.ceil(np.log2(float(out.abs().max())))))
    big = ctx.matvec(emb, V * 2.0 ** k)
    assert bool(torch.isfinite(big).all())
    assert torch.equal(big, out * 2.0 ** k)
    ctx.close()
