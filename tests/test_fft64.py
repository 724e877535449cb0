"""FP64 transforms: the stage structure and table addressing of every compiled
length (no GPU); the passes, the torus eigenvalues and the sampler against the
oracle at the ends of their ranges."""
import numpy as np
import pytest

SIZES = [(B, 4) for B in range(3, 10)] + [(B, 16) for B in range(10, 14)]


def brev(x, b):
    return int(format(x, f"0{b}b")[::-1], 2) if b else 0


def plan(B, E):
    le = E.bit_length() - 1
    r0 = 1 << (B % le) if B % le else E
    st, ns = [(r0, 1)], r0
    while ns < 1 << B:
        st.append((E, ns))
        ns *= E
    return st


@pytest.mark.parametrize("B,E", SIZES)
def test_addressing(B, E):
    L, LT = 1 << B, (1 << B) // E
    PS = 2 if E == 4 or L == 1024 else 3 if L in (128, 512, 2048) else 4

    def pad(x):
        return x + (x >> PS)
    assert len(plan(B, E)) >= 2
    for R, NS in plan(B, E):
        outs = set()
        for t in range(LT):
            k = t & (NS - 1)
            for u in range(E // R):
                for s in range(R):
                    c = u * LT * R + s * NS
                    assert pad((t - k) * R + k + c) == pad((t - k) * R + k) + pad(c)
                    outs.add((t - k) * R + k + c)
            for m in range(E):
                assert pad(t + m * LT) == pad(t) + pad(m * LT)
            if NS > 1:
                assert 2 <= NS <= 512 and 8 * (NS - 2) + (E // 2 - 1) * NS + k < 8 * 1022
        assert outs == set(range(L)) and pad(L - 1) < L + (L >> PS)


@pytest.mark.parametrize("B,E", SIZES[:9])
def test_stages_are_the_transform(B, E):
    L = 1 << B
    r = np.random.default_rng(B)
    x = r.standard_normal(L) + 1j * r.standard_normal(L)
    y = x.copy()
    for R, NS in plan(B, E):
        n, out = R.bit_length() - 1, np.empty(L, complex)
        for j in range(L // R):
            k = j % NS
            v = [y[j + q * (L // R)] for q in range(R)]
            for lev in range(1, n + 1):
                D = R >> lev
                for p in range(R):
                    if not p & D:
                        w = np.exp(-2j * np.pi * (k / NS + brev(p // (2 * D), lev - 1)) / (1 << lev)) * v[p + D]
                        v[p], v[p + D] = v[p] + w, v[p] - w
            for s in range(R):
                out[(j - k) * R + k + s * NS] = v[brev(s, n)]
        y = out
    # FP64 rounding of B butterfly levels
    assert np.max(np.abs(y - np.fft.fft(x))) <= 1e-14 * B * np.max(np.abs(y))


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nvec", [(4, 4, 1), (5, 300, 2), (16, 17, 3), (33, 9, 40), (64, 65, 1), (128, 130, 2),
                                        (300, 260, 5), (512, 33, 64), (1030, 40, 2), (40, 2100, 3)])
def test_fp64_matvec_sample_and_eigenvalues(n1, n2, nvec):
    import torch

    from oracle import kryoracle as O
    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    rng = np.random.default_rng(n1 * 7 + n2)
    # isotropic (even covariance), rotated (averaged images at half the torus), a Bessel order
    for cov in (I.Cov(1.0, 0.07, 1.5, 0.1), I.Cov(0.7, 0.05, 0.5, 0.1, angle=0.4, ratio=1.7),
                I.Cov(1.0, 0.06, 1.1, 0.1, angle=0.9, ratio=1.0)):
        mask = rng.random((n1, n2)) >= 0.4
        mask[0, 0] = True
        P = O.FFTProblem(n1, n2, mask, cov)
        ctx = kry.Context(0)
        p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
        V = rng.standard_normal((nvec, p))
        emb = ctx.embed(cov, kry.KRY_F64)
        out = ctx.matvec(emb, torch.tensor(V, device="cuda:0")).cpu().numpy()
        ref = P.matvec(V)
        # the FP64 tolerance of every matvec test
        assert np.max(np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)) <= 1e-12
        # a pair of vectors gives the same bits alone as in the batch
        one = ctx.matvec(emb, torch.tensor(V[:2], device="cuda:0")).cpu().numpy()
        assert np.array_equal(one, out[:2])
        # BCCB log-determinant (eigenvalues and their range derivatives on the torus)
        ld, dl = ctx.bccb_logdet(cov)
        rld, rdl = O.bccb_logdet(n1, n2, cov, "scaled")
        assert abs(ld - rld) <= 1e-9 * abs(rld) and abs(dl - rdl) <= 1e-7 * max(abs(rdl), abs(rld))
        # a sample on the smallest torus and on one twice as long each way
        M1, M2 = P.M1, P.M2
        for q in (1, 2):
            if max(M1, M2) * q <= 8192:
                xi = rng.standard_normal((2, q * M1, q * M2))
                f = ctx.sample(cov, q * M1, q * M2, torch.tensor(xi, device="cuda:0")).cpu().numpy()
                g = O.sample_field(n1, n2, q * M1, q * M2, cov, xi)
                # sqrt of eigenvalues that are rounding (1e-16 of the largest) adds up to 1e-8 of a standard deviation
                assert np.max(np.abs(f - g)) <= 1e-7
        ctx.close()
