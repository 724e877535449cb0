// Shared-memory Stockham FFT building blocks (power-of-two lengths).
//
// A length-L transform is run by L / 8 threads, each holding 8 complex values
// in registers per stage.  The stages are Stockham autosort steps
// (the formulation of Govindaraju et al., "High performance discrete Fourier
// transforms on graphics processors", SC 2008): butterfly j of a radix-R stage
// with stride Ns reads x[j + r L/R] (r < R), twiddles them by
// exp(-+2 pi i r (j mod Ns) / (Ns R)), runs an R-point DFT in registers and
// writes x[(j div Ns) Ns R + (j mod Ns) + r Ns].  The buffer is transformed in
// place: every thread reads its inputs, the block synchronises, every thread
// writes, the block synchronises.  One radix-2 or radix-4 stage comes first
// when log2 L is not a multiple of 3; all other stages are radix 8.
//
// Forward transforms use exp(-2 pi i jk / L) and are unscaled; inverse
// transforms use exp(+2 pi i jk / L) and are unscaled too.
#pragma once

#include <cuda_runtime.h>

#include "kry_internal.cuh"

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
    return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
// multiply by -i (forward) or +i (inverse)
template <bool INV> __device__ __forceinline__ float2 cmul_mi(float2 a) {
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// R-point DFTs in registers, sign by INV.
template <bool INV> __device__ __forceinline__ void dft2(float2& a, float2& b) {
    float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

template <bool INV> __device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
    float2 t0 = cadd(a0, a2), t1 = csub(a0, a2);
    float2 t2 = cadd(a1, a3), t3 = cmul_mi<INV>(csub(a1, a3));
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    a1 = cadd(t1, t3);
    a3 = csub(t1, t3);
}

template <bool INV> __device__ __forceinline__ void dft8(float2* v) {
    const float h = 0.70710678118654752440f;
    // even / odd halves
    dft4<INV>(v[0], v[2], v[4], v[6]);
    dft4<INV>(v[1], v[3], v[5], v[7]);
    // twiddle the odd half by w8^k, w8 = exp(-+2 pi i / 8)
    float2 o1 = v[3], o2 = v[5], o3 = v[7];
    // w8^1 = h (1 -+ i)
    float2 w1 = INV ? make_float2(h * (o1.x - o1.y), h * (o1.x + o1.y)) : make_float2(h * (o1.x + o1.y), h * (o1.y - o1.x));
    // w8^2 = -+ i
    float2 w2 = cmul_mi<INV>(o2);
    // w8^3 = h (-1 -+ i)
    float2 w3 = INV ? make_float2(-h * (o3.x + o3.y), h * (o3.x - o3.y)) : make_float2(h * (o3.y - o3.x), -h * (o3.x + o3.y));
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1];
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, w1);
    v[5] = csub(e1, w1);
    v[2] = cadd(e2, w2);
    v[6] = csub(e2, w2);
    v[3] = cadd(e3, w3);
    v[7] = csub(e3, w3);
}

template <int R, bool INV> __device__ __forceinline__ void dftR(float2* v) {
    if constexpr (R == 2) {
        dft2<INV>(v[0], v[1]);
    } else if constexpr (R == 4) {
        dft4<INV>(v[0], v[1], v[2], v[3]);
    } else {
        dft8<INV>(v);
    }
}

// One Stockham stage on buf[0..L), run by threads t in [0, L/8).
template <int R, bool INV>
__device__ __forceinline__ void stockham_stage(float2* buf, int L, int Ns, int t, const float2* __restrict__ tw) {
    constexpr int NB = 8 / R;
    float2 v[8];
    const int LR = L / R;
    const int LT = L / 8;
    const int twstep = KRY_TWN / (Ns * R);
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        const int j = t + u * LT;
        const int k = j & (Ns - 1);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float2 x = buf[j + r * LR];
            if (r > 0 && Ns > 1) {
                const float2 w = tw[r * k * twstep];
                x = INV ? cmulc(x, w) : cmul(x, w);
            }
            v[u * R + r] = x;
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < NB; ++u) {
        dftR<R, INV>(&v[u * R]);
        const int j = t + u * LT;
        const int k = j & (Ns - 1);
        const int base = (j - k) * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) buf[base + r * Ns] = v[u * R + r];
    }
    __syncthreads();
}

// Full in-place transform of buf[0..L) by the L / 8 threads t of one group.
// Every thread of the block must call this (it synchronises the block).
template <bool INV>
__device__ __forceinline__ void fft_smem(float2* buf, int L, int t, const float2* __restrict__ tw) {
    int logL = 31 - __clz(L);
    int Ns = 1;
    const int rem = logL % 3;
    if (rem == 1) {
        stockham_stage<2, INV>(buf, L, 1, t, tw);
        Ns = 2;
    } else if (rem == 2) {
        stockham_stage<4, INV>(buf, L, 1, t, tw);
        Ns = 4;
    }
    while (Ns < L) {
        stockham_stage<8, INV>(buf, L, Ns, t, tw);
        Ns *= 8;
    }
}
