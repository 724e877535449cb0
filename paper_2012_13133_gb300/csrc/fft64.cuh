// FP64 FFT building blocks, specialised at compile time: transforms of length L =
// 2^B by L / E threads holding E complex values each.
//
// GB300 issues an FP64 instruction of a warp once in 64 cycles per scheduler
// (1.05 TFLOP/s of FMAs over the chip), so these transforms cost what their FP64
// instructions cost; loads, shared memory and address arithmetic hide behind
// them.  Two things follow:
//  * Butterflies in their FMA form (E. Linzer & E. Feig, IEEE Trans. Signal
//    Processing 41, 1993): a +- w b, w = c (1 - i T), as u = b - i T b, a +- c u,
//    6 instructions.  A radix-16 stage takes 192 for 16 values, twiddles
//    included, against 264 before (60 for the twiddle products, 36 for forming
//    nine of them, 168 for the 16-point DFT); its eight distinct (c, T) pairs are
//    loaded.
//  * E = 16 for long transforms, E = 4 up to 512 points: a thread's serial chain is
//    a quarter as long, and small grids have too few warps for the chip's 608
//    schedulers otherwise.
// Level 1, whose angles reach half a turn (cos = 0), takes p = a + w b with (cos,
// sin) in its table entry, and 2 a - p: 6 instructions too.  The other levels' T
// goes up to 1304 (side 8192), so intermediate values are to stay below 2^1013.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace kf64 {

__host__ __device__ constexpr int ilog2c(int x) { return x <= 1 ? 0 : 1 + ilog2c(x >> 1); }
__host__ __device__ constexpr int brev(int x, int b) {
    int y = 0;
    for (int i = 0; i < b; ++i) y |= ((x >> i) & 1) << (b - 1 - i);
    return y;
}

template <int B, int E_>
struct Plan {
    static constexpr int L = 1 << B, E = E_, LE = ilog2c(E_);
    static constexpr int LT = L / E;                              // threads per transform
    static constexpr int R0 = (B % LE) ? 1 << (B % LE) : E;       // radix of the first stage
    static constexpr int S = (B + LE - 1) / LE;                   // number of stages (at least two)
    // one padding slot every 2^PS positions of the interleaved shared-memory layout
    static constexpr int PS = E == 4 ? 2 : L == 1024 ? 2 : L == 128 || L == 512 || L == 2048 ? 3 : 4;
    static constexpr int SLOTS = L + (L >> PS);                   // 16-byte slots of one transform
};

template <int PS, int NT>
__device__ __forceinline__ constexpr int soff(int x) {
    return (x + (x >> PS)) * NT;
}

// cos and tan of 2 pi m / 16, m = 0..3
__device__ __forceinline__ constexpr double cos16(int m) {
    constexpr double c[4] = {1.0, 0.92387953251128675613, 0.70710678118654752440, 0.38268343236508977173};
    return c[m];
}
__device__ __forceinline__ constexpr double tan16(int m) {
    constexpr double t[4] = {0.0, 0.41421356237309504880, 1.0, 2.41421356237309504880};
    return t[m];
}

// (a, b) -> (a + w b, a - w b), w = c (1 -+ i T) (forward / inverse), times -+i
// with ROT; PLUS: only the sum.
template <bool INV, bool ROT, bool PLUS>
__device__ __forceinline__ void bfly(double2& a, double2& b, double c, double T) {
    const double ur = INV ? fma(-T, b.y, b.x) : fma(T, b.y, b.x), ui = INV ? fma(T, b.x, b.y) : fma(-T, b.x, b.y);
    double2 p, m;
    if constexpr (!ROT) {
        p = make_double2(fma(c, ur, a.x), fma(c, ui, a.y));
        if constexpr (!PLUS) m = make_double2(fma(-c, ur, a.x), fma(-c, ui, a.y));
    } else if constexpr (!INV) {   // -i u = (ui, -ur)
        p = make_double2(fma(c, ui, a.x), fma(-c, ur, a.y));
        if constexpr (!PLUS) m = make_double2(fma(-c, ui, a.x), fma(c, ur, a.y));
    } else {   // i u = (-ui, ur)
        p = make_double2(fma(-c, ui, a.x), fma(c, ur, a.y));
        if constexpr (!PLUS) m = make_double2(fma(c, ui, a.x), fma(-c, ur, a.y));
    }
    a = p;
    if constexpr (!PLUS) b = m;
}

// The same for w = c -+ i s.
template <bool INV, bool PLUS>
__device__ __forceinline__ void bfly_cs(double2& a, double2& b, double c, double s) {
    const double2 p = make_double2(fma(INV ? -s : s, b.y, fma(c, b.x, a.x)), fma(INV ? s : -s, b.x, fma(c, b.y, a.y)));
    if constexpr (!PLUS) b = make_double2(fma(2.0, a.x, -p.x), fma(2.0, a.y, -p.y));
    a = p;
}

// w = 1 (ROT: w = -+i)
template <bool INV, bool ROT, bool PLUS>
__device__ __forceinline__ void bfly1(double2& a, double2& b) {
    const double2 x = a, y = ROT ? (INV ? make_double2(-b.y, b.x) : make_double2(b.y, -b.x)) : b;
    a = make_double2(x.x + y.x, x.y + y.y);
    if constexpr (!PLUS) b = make_double2(x.x - y.x, x.y - y.y);
}

// Level l of a radix-R tree, as in fftspec.cuh: partners p, p + D, D = R >> l;
// twiddle entry e + 2^{l-2}, -+i for the upper half of the sub-frequencies;
// output s ends in slot bitrev(s).  CONST: the first stage (omega = 1).  ZIN:
// inputs of the upper half are zero (their slots are not read).  LOW: only
// outputs s < R/2 are formed (slots with bit 0 clear).
__host__ __device__ constexpr int tw_base(int l) { return l == 1 ? 0 : 1 << (l - 2); }

template <int R, int LEV, bool INV, bool CONST, bool ZIN, bool LOW>
__device__ __forceinline__ void level(double2* v, const double2* w) {
    constexpr int D = R >> LEV;
    constexpr bool PLUS = LOW && D == 1;
#pragma unroll
    for (int p = 0; p < R; ++p) {
        if (p & D) continue;
        if constexpr (ZIN && LEV == 1) {
            v[p + D] = v[p];
            continue;
        }
        const int s = brev(p / (2 * D), LEV - 1);
        const bool rot = LEV >= 2 && s >= (1 << (LEV - 2));
        const int e = rot ? s - (1 << (LEV - 2)) : s;
        if (CONST && e == 0) {
            if (rot) bfly1<INV, true, PLUS>(v[p], v[p + D]);
            else bfly1<INV, false, PLUS>(v[p], v[p + D]);
            continue;
        }
        const double c = CONST ? cos16(e * (16 >> LEV)) : w[tw_base(LEV) + e].x;
        const double T = CONST ? tan16(e * (16 >> LEV)) : w[tw_base(LEV) + e].y;
        if (!CONST && LEV == 1) bfly_cs<INV, PLUS>(v[p], v[p + D], c, T);
        else if (rot) bfly<INV, true, PLUS>(v[p], v[p + D], c, T);
        else bfly<INV, false, PLUS>(v[p], v[p + D], c, T);
    }
}

template <int R, int LEV, bool INV, bool CONST, bool ZIN, bool LOW>
__device__ __forceinline__ void levels(double2* v, const double2* w) {
    if constexpr ((1 << LEV) <= R) {
        level<R, LEV, INV, CONST, ZIN, LOW>(v, w);
        levels<R, LEV + 1, INV, CONST, ZIN, LOW>(v, w);
    }
}

// Twiddle table: section 8 (NS - 2) of stage stride NS (a power of two in [2,
// 512]), word e NS + k = (c, T) of entry e = s + 2^{l-2} of level l at frequency
// k, angle (k / NS + s) / 2^l turns; entry 0 (level 1): (cos, sin).
constexpr int TW_WORDS = 8 * 1022;

template <class P, int NT, int R, int NS>
__device__ __forceinline__ void store_outputs(double2* sb, const double2* v, int t) {
    constexpr int NB = P::E / R;
    const int k = t & (NS - 1);
    const int base = soff<P::PS, NT>((t - k) * R + k);
#pragma unroll
    for (int u = 0; u < NB; ++u)
#pragma unroll
        for (int s = 0; s < R; ++s)
            sb[base + soff<P::PS, NT>(u * P::LT * R + s * NS)] = v[u * R + brev(s, ilog2c(R))];
}

template <class P, int NT, int S_, bool INV, bool LOW>
__device__ __forceinline__ void later_stages(double2* sb, double2* v, int t, const double2* __restrict__ tw) {
    constexpr int NS = P::R0 << (P::LE * (S_ - 1));
    constexpr bool last = S_ + 1 == P::S;
    double2 w[P::E / 2];
    const double2* q = tw + 8 * (NS - 2) + (t & (NS - 1));
#pragma unroll
    for (int e = 0; e < P::E / 2; ++e) w[e] = __ldg(q + e * NS);
    __syncthreads();
    const int tb = soff<P::PS, NT>(t);
#pragma unroll
    for (int r = 0; r < P::E; ++r) v[r] = sb[tb + soff<P::PS, NT>(r * P::LT)];
    levels<P::E, 1, INV, false, false, LOW && last>(v, w);
    if constexpr (!last) {
        __syncthreads();
        store_outputs<P, NT, P::E, NS>(sb, v, t);
        later_stages<P, NT, S_ + 1, INV, LOW>(sb, v, t, tw);
    }
}

// A whole transform: v[m] = input position t + m LT (ZIN: those of the upper
// half of the positions are zero and not read); on return slot bitrev(s) holds
// output position t + s LT (LOW: only s < E/2).  sb: the block's buffer offset
// by the transform's index n < NT.  The buffer must be free on entry, and the
// caller synchronises before it is written again.
template <class P, int NT, bool INV, bool ZIN, bool LOW>
__device__ __forceinline__ void transform(double2* sb, double2* v, int t, const double2* __restrict__ tw) {
    constexpr int R = P::R0, NB = P::E / R;
    double2 w[P::E];
#pragma unroll
    for (int u = 0; u < NB; ++u) {
#pragma unroll
        for (int r = 0; r < (ZIN ? R / 2 : R); ++r) w[u * R + r] = v[u + r * NB];
        levels<R, 1, INV, true, ZIN, false>(w + u * R, nullptr);
    }
    store_outputs<P, NT, R, 1>(sb, w, t);
    later_stages<P, NT, 1, INV, LOW>(sb, v, t, tw);
}

}  // namespace kf64
