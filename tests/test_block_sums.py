"""Dot products of FP32 vectors: block sums keep FP64's precision and range, whatever the block."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

SRC = r"""
#include "dfloat.cuh"
template <int WARPS>
__global__ void k_sums(const float* hi, const float* lo, double* out) {
    kry::DFAcc acc[2];
    for (int k = 0; k < 2; ++k) {
        acc[k].hi = hi[k * blockDim.x + threadIdx.x];
        acc[k].lo = lo[k * blockDim.x + threadIdx.x];
    }
    const double s = kry::block_sums<2, WARPS>(acc);
    if (threadIdx.x % WARPS == 0 && threadIdx.x < 2 * WARPS) out[threadIdx.x / WARPS] = s;
}
template <int WARPS>
__global__ void k_sum(const float* hi, const float* lo, double* out) {
    kry::DFAcc acc[1];
    acc[0].hi = hi[threadIdx.x];
    acc[0].lo = lo[threadIdx.x];
    const double s = kry::block_sums<1, WARPS>(acc);
    if (threadIdx.x == 0) out[2] = s;
}
extern "C" int sums(const float* hi, const float* lo, double* out, int threads) {
    switch (threads) {
#define CASE(W) case 32 * W: k_sums<W><<<1, threads>>>(hi, lo, out); k_sum<W><<<1, threads>>>(hi, lo, out); break;
        CASE(1) CASE(2) CASE(4) CASE(8) CASE(16)
        case 96: k_sums<8><<<1, threads>>>(hi, lo, out); k_sum<32><<<1, threads>>>(hi, lo, out); break;
        default: return -1;
    }
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.gpu
@pytest.mark.parametrize("threads", [32, 64, 96, 128, 256, 512])
def test_block_sums_against_exact_sums(threads, tmp_path):
    import torch

    from paper_2012_13133_gb300 import build
    (tmp_path / "s.cu").write_text(SRC)
    subprocess.run([build.nvcc_path(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    build.CSRC, "-o", str(tmp_path / "s.so"), str(tmp_path / "s.cu")], check=True)
    lib = ctypes.CDLL(os.fspath(tmp_path / "s.so"))
    r = np.random.default_rng(threads)
    g = r.standard_normal((2, threads))
    spread = g * 10.0 ** r.uniform(-6, 6, (2, threads))
    cancel = np.concatenate([g[:, : threads // 2], -g[:, : threads // 2] * (1 + 1e-9)], axis=1)
    top = np.abs(g) * 2.0 ** 124   # no two of them may fit FP32 together
    edge = np.zeros((2, threads))
    edge[:, :: threads // 2] = 3e38   # finite in every warp, not over the block (one warp: not in the warp)
    for x in (np.abs(g), g, spread, cancel, top, edge, np.zeros((2, threads))):
        hi = x.astype(np.float32)
        lo = ((x - hi) + 2.0 ** -30 * x * r.standard_normal(x.shape)).astype(np.float32)   # not renormalised
        out = torch.zeros(3, dtype=torch.float64, device="cuda:0")
        dev = [torch.tensor(v, device="cuda:0") for v in (hi, lo)]
        torch.cuda.synchronize()
        assert lib.sums(*[ctypes.c_void_p(t.data_ptr()) for t in (*dev, out)], threads) == 0
        for i in range(3):
            k = i % 2   # out[2] is the first sum by itself
            terms = [Fraction(float(v)) for v in (*hi[k], *lo[k])]
            exact, size = sum(terms), sum(abs(t) for t in terms)
            err = abs(Fraction(float(out[i])) - exact)
            # the result's own rounding (twice: its last two parts are added first) and an FP64 tree's of 10 levels
            # where FP32 overflows; beside it three floats leave 2^-70 a level of the terms' sizes
            over = size > Fraction(float(np.finfo(np.float32).max))
            assert err <= abs(exact) * Fraction(2, 2 ** 53) + size * (Fraction(11, 2 ** 53) if over else Fraction(10, 2 ** 70))


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nrhs,power", [(150, 140, 1, 60), (600, 90, 3, 60), (40, 520, 2, 58)])
def test_solve_scales_with_its_right_hand_side(n1, n2, nrhs, power):
    """A power of two in the right-hand side is one in the solution, where a block's squares leave FP32's
    range (and a thread's, at most 16 of them times ||K||, do not)."""
    import torch

    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    mask = np.random.default_rng(n1).random((n1, n2)) >= 0.2
    ctx = kry.Context(0)
    p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
    B = torch.randn((nrhs, p), generator=torch.Generator().manual_seed(n2), dtype=torch.float64).cuda()
    emb = ctx.embed(I.Cov(1.0, 0.5 / min(n1, n2), 0.5, 0.5), kry.KRY_F32)
    X, it, _, st = ctx.solve(emb, B, rtol=1e-8, maxit=500)
    X, B2 = X.clone(), B * 2.0 ** power
    X2, it2, _, st2 = ctx.solve(emb, B2, rtol=1e-8, maxit=500)
    assert st == st2 == kry.KRY_OK and it == it2
    assert torch.equal(X2, X * 2.0 ** power)
    ctx.close()
