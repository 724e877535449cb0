"""Host-side checks of the two-lane FP32 matvec passes (no GPU): shared-memory
and table addressing of every compiled block, the stage structure in exact
arithmetic, and (on a GPU) the passes at the edges of their tiles."""
import numpy as np
import pytest

B_ALL = range(6, 14)


E = 16   # values per thread


def blocks(B):
    lt = (1 << (B - 1)) // E
    cap = 512 if B >= 12 else 256 if B >= 8 else 128
    return [th for th in (32, 64, 128, 256, 512) if th >= lt and th <= cap]


def pad_shift(H):
    return 2 if H == 1024 else 3 if H in (128, 512, 2048) else 4


def plan(H):
    b = H.bit_length() - 1
    le = E.bit_length() - 1
    r0 = 1 << (b % le) if b % le else E
    st, ns = [(r0, 1)], r0
    while ns < H:
        st.append((E, ns))
        ns *= E
    return st


def brev(x, b):
    return int(format(x, f"0{b}b")[::-1], 2) if b else 0


@pytest.mark.parametrize("B", B_ALL)
def test_addressing(B):
    H = 1 << (B - 1)
    LT = H // E
    for th in blocks(B):
        NT = th // LT
        PS = pad_shift(H)
        smem = (H + (H >> PS)) * NT   # 16-byte words
        assert smem * 16 <= 227 * 1024 - 1024

        def pad(x):
            return x + (x >> PS)
        for s, (R, NS) in enumerate(plan(H)):
            outs = set()
            for t in range(LT):
                k = t & (NS - 1)
                bo = (t - k) * R + k
                for u in range(E // R):
                    for r in range(R):
                        c = u * LT * R + r * NS
                        j = t + u * LT
                        assert bo + c == (j - j % NS) * R + j % NS + r * NS
                        assert pad(bo + c) == pad(bo) + pad(c)
                        outs.add(bo + c)
                for m in range(E):
                    assert pad(t + m * LT) == pad(t) + pad(m * LT)
                if NS > 1:   # twiddle words: 8 (NS - 2) + e NS + k forward, 4 (NS - 2) + (e/2) NS + k inverse
                    assert 2 <= NS <= 256
                    last = E // 2 - 1
                    assert 8 * (NS - 2) + last * NS + k < 8 * 510
                    assert 4 * (NS - 2) + last // 2 * NS + k < 4 * 510
            assert outs == set(range(H))
            assert (pad(max(outs)) + 1) * NT <= smem
        assert (H - 32) + (LT - 1) + (E - 1) * LT < 8160   # post factors
    # the eigenvalue permutation is one to one within a column
    M1 = 2 * H
    slots = set()
    for k1 in range(M1):
        q, k = k1 & 1, k1 >> 1
        t, s = k & (LT - 1), k // LT
        slots.add(((s >> 1) * LT + t) * 4 + (s & 1) * 2 + q)
    assert slots == set(range(M1))


def tree(v, R, theta, inv):
    """Radix-2 levels of a radix-R decimation-in-time tree, base angle theta; slots in bit-reversed order."""
    n = R.bit_length() - 1
    for lev in range(1, n + 1):
        D = R >> lev
        for p in range(R):
            if p & D:
                continue
            a = theta * D + 2 * np.pi * brev(p // (2 * D), lev - 1) / (1 << lev)
            w = np.exp((1j if inv else -1j) * a) * v[p + D]
            v[p], v[p + D] = v[p] + w, v[p] - w
    return v


def lane(x, delta, inv):
    H = x.size
    for R, NS in plan(H):
        y = np.empty_like(x)
        for j in range(H // R):
            k = j % NS
            v = tree([x[j + r * (H // R)] for r in range(R)], R, 2 * np.pi * (k + delta) / (R * NS), inv)
            for s in range(R):
                y[(j - k) * R + k + s * NS] = v[brev(s, R.bit_length() - 1)]
        x = y
    return x


@pytest.mark.parametrize("B", [6, 7, 8, 9, 10, 11])
def test_two_lanes_are_the_zero_padded_transform(B):
    H = 1 << (B - 1)
    r = np.random.default_rng(B)
    x = r.standard_normal(H) + 1j * r.standard_normal(H)
    X = np.fft.fft(x, 2 * H)
    x0, x1 = lane(x, 0.0, False), lane(x, 0.5, False)
    # FP64 rounding of log2(H) <= 9 butterfly levels
    assert np.max(np.abs(x0 - X[0::2])) <= 1e-13 * np.max(np.abs(X)) * B
    assert np.max(np.abs(x1 - X[1::2])) <= 1e-13 * np.max(np.abs(X)) * B
    Y = r.standard_normal(2 * H) + 1j * r.standard_normal(2 * H)
    y = lane(Y[0::2], 0.0, True) + np.exp(1j * np.pi * np.arange(H) / H) * lane(Y[1::2], 0.0, True)
    ref = np.fft.ifft(Y)[:H] * 2 * H
    assert np.max(np.abs(y - ref)) <= 1e-13 * np.max(np.abs(ref)) * B


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nvec", [(17, 32, 1), (32, 33, 2), (64, 31, 3), (65, 128, 1), (129, 100, 5),
                                        (256, 257, 2), (511, 19, 4), (600, 1025, 3), (20, 2049, 1), (2050, 24, 2)])
def test_matvec_at_tile_edges(n1, n2, nvec):
    import torch

    from oracle import kryoracle as O
    from paper_2012_13133_gb300 import inputs as I
    from paper_2012_13133_gb300 import kry
    cov = I.Cov(1.0, 0.07, 1.5, 0.1, angle=0.4, ratio=1.7)
    rng = np.random.default_rng(n1 * 7 + n2)
    for frac in (0.0, 0.4, 0.97):
        mask = rng.random((n1, n2)) >= frac
        mask[0, 0] = True
        P = O.FFTProblem(n1, n2, mask, cov)
        ctx = kry.Context(0)
        p = ctx.set_mask(torch.from_numpy(mask.astype(np.uint8)).cuda())
        V = rng.standard_normal((nvec, p))
        ref = P.matvec(V)
        emb = ctx.embed(cov, kry.KRY_F32)
        Vt = torch.tensor(V, dtype=torch.float32, device="cuda:0")
        outs = [ctx.matvec(emb, Vt)]
        for g, c in ((1, 1), (2, 16), (16, 4)):   # smallest and largest blocks
            ctx.set_schedule(emb, nvec, g, c, 0)
            outs.append(ctx.matvec(emb, Vt))
        for out in outs:
            out = out.double().cpu().numpy()
            # FP32 rounding of ~4 log2(M) butterfly levels on values of unit size: 1e-6 relative
            err = np.linalg.norm(out - ref, axis=1) / np.linalg.norm(ref, axis=1)
            assert err.max() <= 1e-6, (frac, err)
        ctx.close()
