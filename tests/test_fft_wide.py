"""The FP32 passes for torus sides 1024 and 2048 (32 values per thread): addressing and the
two-stage structure without a GPU; with one, the passes at the edges of their tiles."""
import numpy as np
import pytest

E = 32


def brev(x, b):
    return int(format(x, f"0{b}b")[::-1], 2) if b else 0


@pytest.mark.parametrize("B", [10, 11])
def test_addressing(B):
    H = 1 << (B - 1)
    LT = R0 = H // E
    NB = E // R0
    words = H + 32   # shared memory of one transform and q, in complex values
    out, inp = set(), set()
    for t in range(LT):
        for u in range(NB):
            for s in range(R0):
                pos = (t + u * LT) * R0 + s
                off = t * (R0 + 1) + u * LT * (R0 + 1) + s
                assert off == pos + pos // R0 < words
                out.add(off)
        for r in range(E):
            pos = t + r * LT
            off = t + r * LT + r * LT // R0
            assert off == pos + pos // R0
            inp.add(off)
    assert out == inp and len(out) == H
    for ns, base in ((1, 0), (16, 32), (32, 32 + 512)):   # twiddle table
        assert base + 15 * 2 * ns + 2 * (ns - 1) + 1 < 32 + 512 + 1024
    M1, lt = 2 * H, H // 16
    slots = set()
    for k1 in range(M1):
        q, k = k1 & 1, k1 >> 1
        t, s = k % (lt // 2), k // (lt // 2)
        slots.add(((s >> 2) * lt + 2 * t + q) * 4 + (s & 3))
    assert slots == set(range(M1))
    for logc in (2, 3, 4, 5):   # slab columns 2 t + q + s 2 LT: whole tiles between s and s + 1
        n1, row = 7, 3
        for t in range(LT):
            for q in (0, 1):
                for s in range(E):
                    col, c0 = 2 * t + q + s * 2 * LT, 2 * t + q
                    at = (((col >> logc) * n1 + row) << logc) + col % (1 << logc)
                    assert at == (((c0 >> logc) * n1 + row) << logc) + c0 % (1 << logc) + s * n1 * 2 * LT


def tree(v, theta, inv):
    R = len(v)
    for lev in range(1, R.bit_length()):
        D = R >> lev
        for p in range(R):
            if p & D:
                continue
            a = theta * D + 2 * np.pi * brev(p // (2 * D), lev - 1) / (1 << lev)
            w = np.exp((1j if inv else -1j) * a) * v[p + D]
            v[p], v[p + D] = v[p] + w, v[p] - w
    return [v[brev(s, R.bit_length() - 1)] for s in range(R)]


def lane(x, delta, inv):
    H = x.size
    R0 = H // E
    y = np.empty_like(x)
    for j in range(E):
        y[j * R0:(j + 1) * R0] = tree([x[j + r * E] for r in range(R0)], 2 * np.pi * delta / R0, inv)
    z = np.empty_like(x)
    for t in range(R0):
        z[t::R0] = tree([y[t + r * R0] for r in range(E)], 2 * np.pi * (t + delta) / H, inv)
    return z


@pytest.mark.parametrize("B", [10, 11])
def test_two_stages_are_the_zero_padded_transform(B):
    H = 1 << (B - 1)
    r = np.random.default_rng(B)
    x = r.standard_normal(H) + 1j * r.standard_normal(H)
    X = np.fft.fft(x, 2 * H)
    for q in (0, 1):   # FP64 rounding of 10 butterfly levels
        assert np.max(np.abs(lane(x, 0.5 * q, False) - X[q::2])) <= 1e-12 * np.max(np.abs(X))
    Y = r.standard_normal(2 * H) + 1j * r.standard_normal(2 * H)
    y = lane(Y[0::2], 0.0, True) + np.exp(1j * np.pi * np.arange(H) / H) * lane(Y[1::2], 0.0, True)
    ref = np.fft.ifft(Y)[:H] * 2 * H
    assert np.max(np.abs(y - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.gpu
@pytest.mark.parametrize("n1,n2,nvec", [(257, 33, 1), (30, 512, 2), (512, 511, 3), (513, 1024, 1), (1024, 300, 4),
                                        (1000, 2049, 2), (40, 600, 33)])
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
