// FP32 FFT building blocks of the covariance matvec passes, specialised at
// compile time.
//
// Every transform of the matvec is zero padded: H of the 2H = L torus points
// hold data, and only H of the inverse's outputs are kept.  Instead of a
// length-L transform whose first (last) stage skips half its inputs (outputs),
// a thread runs two length-H transforms side by side, in the two lanes of
// packed FP32 registers:
//   forward  lane q:  X[2k + q] = sum_j x_j W_H^{j (k + q/2)}        (k < H)
//   inverse  lane q:  g_q(j) = sum_k X[2k + q] W_H^{-jk},
//            y_j = g_0(j) + W_L^{-j} g_1(j)                          (j < H)
// Both lanes run the same butterflies; forward, lane 1's twiddles belong to
// the half-integer frequency k + 1/2, so no separate modulation pass is
// needed.  A packed instruction (add/fma.rn.f32x2) does the work of two at the
// FMA pipe rate of two, so the gain is everywhere else: half the instructions
// to issue, one 16-byte shared-memory access where there were two of 8, one
// address per two values, and one barrier-separated stage fewer where L =
// 512 or 8192 (H = 256 = 16^2, 4096 = 16^3).  Measured against one length-L
// transform per thread group with 8-byte accesses: 4 vectors on 4096^2 2,070 ->
// 1,263 us.  What bounds the passes now is the shared-memory and L1 pipe (column
// pass of side 2048, before mvwide.cuh took it over: 860 wavefronts per warp, 512
// of them the four exchanges, 68% busy), then latency at 16 warps per SM.
//
// Stages (Stockham after Govindaraju et al., SC 2008): radix R0 = 2^(log2 H
// mod 4) (16 when that is 1) first, then radix 16; a thread holds 16 packed
// complex values, H / 16 threads run a transform.
//
// Butterflies: a radix-R stage is its log2 R levels of radix-2 butterflies
// a +- w b, w = c (1 - i T), T = tan, taken as u = b - i T b (2 FMAs), a +- c u
// (4 FMAs): 6 FMA-pipe operations instead of 8 (E. Linzer & E. Feig,
// "Implementation of efficient FFT algorithms on fused multiply-add
// architectures", IEEE Trans. Signal Processing 41, 1993).  The twiddles of a
// whole radix-16 stage are then 8 pairs (c, T) (the other seven are these
// times -i), all from a table; the products that formed 12 of 15 twiddles
// before are gone.  Rounding: u carries a relative error of |T| eps |b|, which
// the factor c scales back to eps |sin| |b|, so a large T costs no accuracy.  Level
// 1, whose angles reach half a turn, takes p = a + w b with (cos, sin) in its table
// entry and 2 a - p (8 operations); from level 2 on they stay below a quarter turn.
//
// Range: T reaches R NS / 2 pi at the last level of a stage of radix R and stride NS, 652
// at side 8192, so intermediate values are to stay below 2^118.  Forward they can be
// as large as the sum over the grid; pass A therefore scales its input by FWD_SCALE
// and the eigenvalues of pass B take it back, both exactly.  What is left of it: a
// result K v beyond 2^118 overflows.  ((cos, sin), or tangents of at most one, at
// every level: no limit, but 25% more error on ordinary values.)
#pragma once

#include <cuda_runtime.h>

namespace kspec {

typedef unsigned long long u64;

// Two packed FP32 lanes per word: complex values of lane 0 and lane 1.
struct c2 {
    u64 r, i;
};

__device__ __forceinline__ u64 pk(float a, float b) {
    u64 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float2 upk(u64 a) {
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(a));
    return f;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 neg2(u64 a) { return a ^ 0x8000000080000000ull; }

// Pad shift of the interleaved shared-memory layout: element p of transform n
// (NT transforms, 16 bytes each) at (p + (p >> PS)) NT + n; the shift with the
// fewest bank conflicts over all stages of H = 2^(B-1) (a quarter warp per
// 16-byte wavefront).  For every stage pad(x + c) = pad(x) + pad(c), so an
// access is one per-thread base plus an immediate.
__host__ __device__ constexpr int pad_shift(int H) {
    return H == 128 || H == 2048 ? 3 : 4;
}

__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x >> 1); }

template <int B>   // transform pair length L = 2^B = 2 H
struct Plan {
    static constexpr int L = 1 << B;
    static constexpr int H = L >> 1;
    static constexpr int E = 16;              // values per thread = radix of all stages but the first
    static constexpr int LE = ilog2c(E);
    static constexpr int LT = H / E;          // threads per transform
    static constexpr int R0 = ((B - 1) % LE) ? (1 << ((B - 1) % LE)) : E;   // radix of the first stage
    static constexpr int S = (B - 2 + LE) / LE;                             // number of stages
};

// Padded shared-memory offset of position x for NT interleaved transforms.
template <int PS, int NT>
__device__ __forceinline__ constexpr int soff(int x) {
    return (x + (x >> PS)) * NT;
}

__host__ __device__ constexpr int brev(int x, int b) {
    int y = 0;
    for (int i = 0; i < b; ++i) y |= ((x >> i) & 1) << (b - 1 - i);
    return y;
}

// cos and tan of 2 pi m / 32, m = 0..7
__device__ __forceinline__ constexpr float cos32(int m) {
    constexpr float c[8] = {1.0f, 0.980785280403230431f, 0.923879532511286738f, 0.831469612302545236f,
                           0.707106781186547573f, 0.555570233019602289f, 0.382683432365089837f, 0.195090322016128331f};
    return c[m];
}
__device__ __forceinline__ constexpr float tan32(int m) {
    constexpr float t[8] = {0.0f, 0.198912367379658006f, 0.414213562373095034f, 0.668178637919298879f,
                           0.999999999999999889f, 1.49660576266548895f, 2.41421356237309492f, 5.0273394921258463f};
    return t[m];
}

// One radix-2 butterfly (a, b) -> (a + w b, a - w b) in both lanes, w = c -+ i s
// (forward / inverse).
template <bool INV>
__device__ __forceinline__ void bfly_cs(c2& a, c2& b, u64 c, u64 s) {
    const u64 ns = neg2(s);
    const u64 pr = fma2(INV ? ns : s, b.i, fma2(c, b.r, a.r)), pi = fma2(INV ? s : ns, b.r, fma2(c, b.i, a.i));
    b = {sub2(add2(a.r, a.r), pr), sub2(add2(a.i, a.i), pi)};   // a - w b = 2 a - (a + w b)
    a = {pr, pi};
}

// One radix-2 butterfly (a, b) -> (a + w b, a - w b) in both lanes, w = c (1 -+ i T)
// (forward / inverse), times -+i with ROT.
template <bool INV, bool ROT>
__device__ __forceinline__ void bfly(c2& a, c2& b, u64 c, u64 T) {
    const u64 nT = neg2(T), nc = neg2(c);
    const u64 ur = fma2(INV ? nT : T, b.i, b.r), ui = fma2(INV ? T : nT, b.r, b.i);
    if constexpr (!ROT) {
        b = {fma2(nc, ur, a.r), fma2(nc, ui, a.i)};
        a = {fma2(c, ur, a.r), fma2(c, ui, a.i)};
    } else if constexpr (!INV) {   // -i u = (ui, -ur)
        b = {fma2(nc, ui, a.r), fma2(c, ur, a.i)};
        a = {fma2(c, ui, a.r), fma2(nc, ur, a.i)};
    } else {   // i u = (-ui, ur)
        b = {fma2(c, ui, a.r), fma2(nc, ur, a.i)};
        a = {fma2(nc, ui, a.r), fma2(c, ur, a.i)};
    }
}

// w = 1 (ROT: w = -+i)
template <bool INV, bool ROT>
__device__ __forceinline__ void bfly1(c2& a, c2& b) {
    const c2 x = a, y = b;
    if constexpr (!ROT) {
        a = {add2(x.r, y.r), add2(x.i, y.i)};
        b = {sub2(x.r, y.r), sub2(x.i, y.i)};
    } else if constexpr (!INV) {
        a = {add2(x.r, y.i), sub2(x.i, y.r)};
        b = {sub2(x.r, y.i), add2(x.i, y.r)};
    } else {
        a = {sub2(x.r, y.i), add2(x.i, y.r)};
        b = {add2(x.r, y.i), sub2(x.i, y.r)};
    }
}

// Level l of a radix-R decimation-in-time tree on R values (distance D = R >>
// l between partners): partner pair p, p + D has sub-frequency s = the bits of
// p above D, reversed; its twiddle is omega^D W_{2^l}^s, held as entry
// s' + 2^{l-2} (1, 1, 2, 4 entries for l = 1..4; s >= 2^{l-2} is entry s -
// 2^{l-2} times -+i).  Output s of the tree ends in slot bitrev(s).
__host__ __device__ constexpr int tw_base(int l) { return l == 1 ? 0 : 1 << (l - 2); }

// Twiddles of one level: MODE 0 from the registers (c, T) (level 1: (c, s)); MODE 1 the first
// forward stage's (lane 0: W_{2^l}^s, lane 1: that times omega^D, omega =
// W_{2R}); MODE 2 the first inverse stage's (both lanes W_{2^l}^s).
template <int R, int LEV, bool INV, int MODE>
__device__ __forceinline__ void level(c2* v, const u64* c, const u64* T) {
    constexpr int D = R >> LEV;
#pragma unroll
    for (int p = 0; p < R; ++p) {
        if (p & D) continue;
        const int s = brev(p / (2 * D), LEV - 1);
        const bool rot = LEV >= 2 && s >= (1 << (LEV - 2));
        const int e = rot ? s - (1 << (LEV - 2)) : s;
        u64 cc = 0, tt = 0;
        if constexpr (MODE == 0) {
            cc = c[tw_base(LEV) + e];
            tt = T[tw_base(LEV) + e];
            if constexpr (LEV == 1) {
                bfly_cs<INV>(v[p], v[p + D], cc, tt);
                continue;
            }
        } else {
            const int m0 = e * (32 >> LEV), m1 = MODE == 1 ? m0 + (16 >> LEV) : m0;
            if (MODE == 2 && e == 0) {
                if (rot) bfly1<INV, true>(v[p], v[p + D]);
                else bfly1<INV, false>(v[p], v[p + D]);
                continue;
            }
            cc = pk(cos32(m0), cos32(m1));
            tt = pk(tan32(m0), tan32(m1));
        }
        if (rot) bfly<INV, true>(v[p], v[p + D], cc, tt);
        else bfly<INV, false>(v[p], v[p + D], cc, tt);
    }
}

template <int R, int LEV, bool INV, int MODE>
__device__ __forceinline__ void levels(c2* v, const u64* c, const u64* T) {
    if constexpr ((1 << LEV) <= R) {
        level<R, LEV, INV, MODE>(v, c, T);
        levels<R, LEV + 1, INV, MODE>(v, c, T);
    }
}

// Level 1 of the first forward stage: both lanes start from the same x; lane
// 1's twiddle is omega^{R/2} = -i.  (Unpacked adds write the packed halves.)
__device__ __forceinline__ void first_pair(float2 a, float2 b, c2& p, c2& m) {
    p = {pk(a.x + b.x, a.x + b.y), pk(a.y + b.y, a.y - b.x)};
    m = {pk(a.x - b.x, a.x - b.y), pk(a.y - b.y, a.y + b.x)};
}

// Twiddle tables, one section per stage stride NS (a power of two in [2,
// 256]).  Entry e = s + 2^{l-2} of level l at frequency k has the angle (k / NS
// + s) / 2^l turns, whatever the stage's radix.  Entry-major, so that threads
// with consecutive k = t mod NS read consecutive 16-byte words:
//   forward  word 8 (NS - 2) + e NS + k      = (c, c', T, T')  lanes k, k + 1/2
//   inverse  word 4 (NS - 2) + (e/2) NS + k  = (c_e, T_e, c_{e+1}, T_{e+1})
// with sin instead of tan for entry 0 (level 1).
constexpr int TWF_WORDS = 8 * 510, TWI_WORDS = 4 * 510;
// Post factors exp(+2 pi i j / L) of the inverse: word L/2 - 32 + j, j < L/2
// (64 <= L <= 8192).
constexpr int POST_WORDS = 8160;

// What pass A scales its input by, and the eigenvalues of pass B (lam32P) by its inverse.
constexpr float FWD_SCALE = 0x1p-10f;

// Twiddles of one radix-E stage.
template <int E>
struct StageTw {
    u64 c[E / 2], T[E / 2];
};

template <int E, int NS, bool INV>
__device__ __forceinline__ void load_twiddles(StageTw<E>& s, const float4* __restrict__ tw, int t) {
    const float4* w = tw + (INV ? 4 : 8) * (NS - 2) + (t & (NS - 1));
    if constexpr (INV) {
#pragma unroll
        for (int e = 0; e < E / 4; ++e) {
            const float4 f = __ldg(w + e * NS);
            s.c[2 * e] = pk(f.x, f.x);
            s.T[2 * e] = pk(f.y, f.y);
            s.c[2 * e + 1] = pk(f.z, f.z);
            s.T[2 * e + 1] = pk(f.w, f.w);
        }
    } else {
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            const float4 f = __ldg(w + e * NS);
            s.c[e] = pk(f.x, f.y);
            s.T[e] = pk(f.z, f.w);
        }
    }
}

// Stores of a stage's outputs: butterfly u of thread t (slots u R .. u R + R -
// 1), output s to position (j - k) R + k + s NS, j = t + u H/E, k = t mod NS.
template <int B, int R, int NS, class ST>
__device__ __forceinline__ void store_outputs(const c2* v, int t, ST&& st) {
    constexpr int LT = Plan<B>::LT, NB = Plan<B>::E / R;
    const int k = t & (NS - 1);
    const int bo = (t - k) * R + k;
#pragma unroll
    for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int s = 0; s < R; ++s) st(bo, u * LT * R + s * NS, v[u * R + brev(s, ilog2c(R))]);
}

// First forward stage on x[m] = input position t + m H/E (zeros where there
// is no data).
template <int B, class ST>
__device__ __forceinline__ void first_forward(const float2* x, int t, ST&& st) {
    using P = Plan<B>;
    constexpr int R = P::R0, NB = P::E / R;
    c2 v[P::E];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
#pragma unroll
        for (int r = 0; r < R / 2; ++r)
            first_pair(x[u + r * NB], x[u + (r + R / 2) * NB], v[u * R + r], v[u * R + r + R / 2]);
        levels<R, 2, false, 1>(v + u * R, nullptr, nullptr);
    }
    store_outputs<B, R, 1>(v, t, st);
}

// First inverse stage from the registers a forward transform ends with (w[m] =
// position t + m H/E).
template <int B, class ST>
__device__ __forceinline__ void first_inverse(const c2* w, int t, ST&& st) {
    using P = Plan<B>;
    constexpr int R = P::R0, NB = P::E / R;
    c2 v[P::E];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[u * R + r] = w[u + r * NB];
        levels<R, 1, true, 2>(v + u * R, nullptr, nullptr);
    }
    store_outputs<B, R, 1>(v, t, st);
}

// Stages S_ .. S-1 of a transform whose earlier stages are in shared memory (not
// yet synchronised), w the twiddles of stage S_; the last one leaves its
// outputs in registers, position t + s H/E in slot bitrev(s).
template <int B, int S_, bool INV, class LDS, class STS>
__device__ __forceinline__ void later_stages(c2* v, const StageTw<16>& w, int t, const float4* __restrict__ tw,
                                             LDS&& lds, STS&& sts) {
    using P = Plan<B>;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < P::E; ++r) v[r] = lds(r * P::LT);
    levels<P::E, 1, INV, 0>(v, w.c, w.T);
    if constexpr (S_ + 1 < P::S) {
        constexpr int NS = P::R0 << (P::LE * (S_ - 1));
        __syncthreads();
        store_outputs<B, P::E, NS>(v, t, sts);
        StageTw<16> w2;
        load_twiddles<P::E, NS * P::E, INV>(w2, tw, t);
        later_stages<B, S_ + 1, INV>(v, w2, t, tw, lds, sts);
    }
}

}  // namespace kspec
