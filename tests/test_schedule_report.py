"""The autotuner's report names a schedule that can be set again, on the shortest tori too, whose
default blocks hold up to 64 transforms."""
import numpy as np
import pytest


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,prec", [(32, 32, "f32"), (40, 60, "f32"), (300, 32, "f32"), (5, 9, "f64"), (32, 200, "f64")])
@pytest.mark.parametrize("nvec", [1, 4, 130])
def test_reported_schedule_is_accepted(n1, n2, prec, nvec):
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    dt, pr = (torch.float64, kry.KRY_F64) if prec == "f64" else (torch.float32, kry.KRY_F32)
    mask = np.random.default_rng(n1 + n2).random((n1, n2)) >= 0.3
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    emb = ctx.embed(I.Cov(1.0, 0.1, 0.5, 0.1), pr)
    V = torch.randn((nvec, p), generator=torch.Generator().manual_seed(nvec), dtype=dt).cuda()
    best = ctx.autotune(emb, nvec)
    tuned = ctx.matvec(emb, V)
    ctx.set_schedule(emb, nvec, best["rows_per_block"], best["cols_per_block"], best["pairs_per_batch"])
    # the same transforms, whatever block they share
    assert torch.equal(ctx.matvec(emb, V), tuned)
    ctx.close()
