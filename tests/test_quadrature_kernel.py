"""The quadrature header compiled by itself: Sturm counts on the host, and the kernel on given
tridiagonals, the ones with Ritz values below the bound among them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

SRC = r"""
#include "quadrature.cuh"
extern "C" int sturm(const double* a, const double* b2, int n, double x) { return kry::sturm_count(a, b2, n, x); }
extern "C" int quad(const int* m, const double* a, const double* b, int nvec, int nsteps, double lb, double* out) {
    kry::k_quadrature<<<nvec, kry::QUAD_THREADS>>>(m, a, b, nsteps, 1.0, out, lb, nullptr, 0);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2012_13133_gb300 import build
    try:
        nvcc = build.nvcc_path()
    except RuntimeError:
        pytest.skip("needs nvcc")
    d = tmp_path_factory.mktemp("quadrature")
    (d / "q.cu").write_text(SRC)
    subprocess.run([nvcc, *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    "-o", str(d / "q.so"), str(d / "q.cu")], check=True)
    return ctypes.CDLL(os.fspath(d / "q.so"))


def count(lib, a, b2, x):
    a, b2 = np.array(a, dtype=np.float64), np.array(list(b2) + [0.0], dtype=np.float64)
    dp = ctypes.POINTER(ctypes.c_double)
    return lib.sturm(a.ctypes.data_as(dp), b2.ctypes.data_as(dp), len(a), ctypes.c_double(x))


def test_sturm_count_at_a_zero_pivot(lib):
    # the first pivot (i = 0), one in the middle, several: eigenvalues below x, exactly
    assert count(lib, [1.0, 1.0], [0.25], 1.0) == 1          # 1/2, 3/2
    assert count(lib, [2.0], [], 2.0) == 0                   # 2 is not below 2
    assert count(lib, [2.0, 1.5, 3.0], [1.0, 1.0], 1.0) == 1   # pivots 1, -1/2, 4
    assert count(lib, [2.0, 2.0, 2.0], [1.0, 1.0], 1.0) == 1   # 2 - sqrt(2), 2, 2 + sqrt(2); pivots 1, 0, -inf
    assert count(lib, [0.0] * 5, [1.0] * 4, 0.0) == 2        # symmetric spectrum with a zero: 2 below
    assert count(lib, [3.0, 3.0], [0.0], 3.0) == 0


@pytest.mark.parametrize("n", [1, 2, 9, 50, 256])
def test_sturm_count_of_random_matrices(lib, n):
    r = np.random.default_rng(n)
    a, b = r.standard_normal(n), r.standard_normal(max(n - 1, 0))
    th = np.linalg.eigvalsh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    for i in range(n + 1):   # halfway between neighbours
        x = 0.5 * ((th[i - 1] if i else th[0] - 2.0) + (th[i] if i < n else th[-1] + 2.0))
        assert count(lib, a, b * b, x) == i


def jacobi(theta, w):
    """Lanczos in long double: the tridiagonal with these eigenvalues and squared first components."""
    theta, q = np.array(theta, dtype=np.longdouble), np.sqrt(np.array(w, dtype=np.longdouble))
    q /= np.sqrt(np.sum(q * q))
    Q, a, b = [q], [], []
    for j in range(len(theta)):
        v = theta * Q[j]
        a.append(np.sum(v * Q[j]))
        for _ in range(2):
            for u in Q:
                v = v - np.sum(v * u) * u
        if j + 1 < len(theta):
            b.append(np.sqrt(np.sum(v * v)))
            Q.append(v / b[-1])
    return np.array(a, dtype=np.float64), np.array(b, dtype=np.float64)


def cases():
    """(alpha, beta) whose Ritz values lie below the bound 0.1 as the name says."""
    r = np.random.default_rng(1)
    up = np.sort(0.2 + 3.0 * r.random(20))
    ones = lambda k: np.ones(k) / k
    yield "one", jacobi(np.concatenate([[0.02], up]), ones(21))
    yield "four", jacobi(np.concatenate([[0.003, 0.01, 0.04, 0.09], up]), ones(24))
    yield "all", jacobi([0.001, 0.01, 0.05], ones(3))
    yield "single", (np.array([0.05]), np.zeros(0))
    yield "nothing", jacobi(up, ones(20))
    # Chebyshev matrices, delocalised: more than 128 and 240 of 256 values below (one point an interval)
    for name, mid, half in (("many", 0.0895, 0.088), ("most", 0.051, 0.0495)):
        yield name, (np.full(256, mid), np.full(255, half / 2))
    # what the eigenvalue iteration has to take
    yield "pair", jacobi(np.concatenate([[0.05, 0.05 * (1 + 1e-9)], up]), ones(22))
    yield "deep", jacobi(np.concatenate([[5e-5], up]), ones(21))
    yield "negative", jacobi(np.concatenate([[-0.3], up]), ones(21))
    yield "tiny weight", jacobi(np.concatenate([[0.05], up]), np.concatenate([[1e-24], ones(20)]))
    yield "zero pivot", (np.array([0.1, 0.1, 2.0]), np.array([0.0, 0.1]))


@pytest.mark.gpu
def test_kernel_with_ritz_values_below_the_bound(lib):
    import torch
    lb, c = 0.1, list(cases())
    A, B, M = np.zeros((len(c), 256)), np.zeros((len(c), 256)), np.zeros(len(c), dtype=np.int32)
    ref = []
    for k, (name, (a, b)) in enumerate(c):
        n = M[k] = len(a)
        A[k, :n], B[k, : n - 1] = a, b
        th, U = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
        below = int(np.sum(th < lb))
        want = {"one": 1, "four": 4, "all": 3, "single": 1, "nothing": 0}
        assert below == want.get(name, below), name
        assert {"many": below > 128, "most": below > 200}.get(name, True), (name, below)
        ref.append(np.sum(U[0] ** 2 * np.log(np.maximum(th, lb))))
    dev = [torch.tensor(x, device="cuda:0") for x in (M, A, B)]
    out = torch.full((len(c),), float("nan"), dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    assert lib.quad(*[ctypes.c_void_p(t.data_ptr()) for t in dev], len(c), 256, ctypes.c_double(lb),
                    ctypes.c_void_p(out.data_ptr())) == 0
    # ~250 terms of order one and up to 256 eigenvalues, whose errors 1e-16 ||T|| are 1e-14 of those from the
    # bound up: 1e-12
    err = np.abs(out.cpu().numpy() - np.array(ref))
    assert np.all(err <= 1e-12), dict(zip([n for n, _ in c], err))
