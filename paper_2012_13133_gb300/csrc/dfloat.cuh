// Double-float arithmetic (an unevaluated FP32 pair hi + lo) for the FP32 path.
//
// GB300's FP64 pipe runs at a small fraction of its FP32 rate, so per-element
// FP64 work in the FP32 kernels (a float->double conversion and an FP64 FMA per
// product) makes them FP64-bound.  The accumulations below keep FP64-class
// accuracy with FP32 instructions only:
//   * the exact product a*b = p + e, p = fl(a*b), e = fma(a, b, -p) (the FMA
//     computes a*b - p exactly because that difference is representable);
//   * the exact sum a + b = s + t by Knuth's TwoSum (TAOCP vol. 2, 4.2.2).
// The intrinsics round explicitly, so the compiler cannot contract the steps
// into FMAs, which would break the error-free identities.
#pragma once

#include <cuda_runtime.h>

namespace kry {

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& t) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// Running sum of products held as hi + lo; value() converts once to FP64.
struct DFAcc {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add_prod(float a, float b) {
        const float p = __fmul_rn(a, b);
        const float e = __fmaf_rn(a, b, -p);
        float s, t;
        two_sum(hi, p, s, t);
        hi = s;
        lo = __fadd_rn(lo, __fadd_rn(t, e));
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// (hi, lo) += (ohi, olo), double-float.
__device__ __forceinline__ void df_add(float& hi, float& lo, float ohi, float olo) {
    float s, t;
    two_sum(hi, ohi, s, t);
    hi = s;
    lo = __fadd_rn(__fadd_rn(lo, olo), t);
}

// A sum across threads as three floats a + b + c.  Adding two of them with exact
// first and second components leaves an error of about 2^-70 of the sum, so a tree
// of these loses less than one of FP64 additions (2^-53), without the FP64 pipe.
struct TFloat {
    float a, b, c;
    __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};
__device__ __forceinline__ void tf_add(TFloat& x, const TFloat& y) {
    float s, e, t, f, u, g;
    two_sum(x.a, y.a, s, e);
    two_sum(x.b, y.b, t, f);
    two_sum(t, e, u, g);
    x = {s, u, __fadd_rn(__fadd_rn(x.c, y.c), __fadd_rn(f, g))};
}

__device__ __forceinline__ TFloat tf_xor(const TFloat& x, int o) {
    return {__shfl_xor_sync(0xffffffffu, x.a, o), __shfl_xor_sync(0xffffffffu, x.b, o),
            __shfl_xor_sync(0xffffffffu, x.c, o)};
}

// Block sums of N = 1 or 2 running dot products over a block of at most WARPS warps
// in a fixed order: thread k WARPS returns the k-th, k < N.  Added as three floats;
// where finite sums leave the FP32 range together, in FP64 (a warp's FP64
// instruction holds its scheduler's FP64 pipe for 64 cycles on GB300: an FP64
// shuffle tree in every block of a streaming kernel takes longer than the
// streaming).  Two sums share a tree, each half a warp's lanes.  Against sums in
// double-float, whose 48 bits and FP32 range are less than FP64's, a CG iteration
// for 4 columns takes 25.4 -> 26.3 us on 128^2, 49.6 -> 50.4 us on 500^2.
template <int N, int WARPS>
__device__ __forceinline__ double block_sums(const DFAcc (&acc)[N]) {
    static_assert(N <= 2 && N * WARPS <= 32 && (WARPS & (WARPS - 1)) == 0, "a warp adds the warps' sums");
    __shared__ __align__(16) TFloat red[N][WARPS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    constexpr int HALF = 32 / N;
    TFloat x = {acc[0].hi, acc[0].lo, 0.f};
    if constexpr (N == 2) {
        const TFloat y = {acc[1].hi, acc[1].lo, 0.f};
        const bool second = lane >= 16;
        const TFloat keep = second ? y : x, give = second ? x : y;
        x = keep;
        tf_add(x, tf_xor(give, 16));
    }
#pragma unroll
    for (int o = HALF / 2; o > 0; o >>= 1) tf_add(x, tf_xor(x, o));
    const bool mine = (lane & (HALF - 1)) == 0;
    if (mine) red[lane / HALF][w] = x;
    if (!__syncthreads_or(mine && !isfinite(x.a))) {
        if (w != 0) return 0.0;
        const int k = min(lane / WARPS, N - 1), v = lane & (WARPS - 1);
        x = v < nw ? red[k][v] : TFloat{0.f, 0.f, 0.f};
#pragma unroll
        for (int o = WARPS / 2; o > 0; o >>= 1) tf_add(x, tf_xor(x, o));
        if (v != 0) return 0.0;
        if (isfinite(x.a)) return x.value();
        double s = 0.0;
        for (int i = 0; i < nw; ++i) s += red[k][i].value();
        return s;
    }
    double* red64 = reinterpret_cast<double*>(&red[0][0]);   // nobody reads red on this path
#pragma unroll
    for (int k = 0; k < N; ++k) {
        double v = acc[k].value();
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) red64[k * WARPS + w] = v;
    }
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x < N * WARPS && (threadIdx.x & (WARPS - 1)) == 0)
        for (int i = 0; i < nw; ++i) s += red64[threadIdx.x + i];
    return s;
}

// Dot-product accumulator of the vector precision: double-float for FP32
// vectors, plain FP64 FMAs for FP64 vectors.
template <typename T>
struct DotAcc;
template <>
struct DotAcc<float> {
    DFAcc a;
    __device__ __forceinline__ void add_prod(float x, float y) { a.add_prod(x, y); }
    __device__ __forceinline__ double value() const { return a.value(); }
};
template <>
struct DotAcc<double> {
    double s = 0.0;
    __device__ __forceinline__ void add_prod(double x, double y) { s = fma(x, y, s); }
    __device__ __forceinline__ double value() const { return s; }
};

// (hi, lo) += (ahi + alo) * p, where ahi + alo is an FP64 coefficient split
// into two floats: the product ahi * p exactly (p1 + e1), alo * p rounded (it
// is 2^-24 of the first), TwoSum into hi, then TwoSum again to renormalise
// (hi and the correction can cancel, so FastTwoSum's ordering may not hold).
__device__ __forceinline__ void df_axpy(float& hi, float& lo, float ahi, float alo, float p) {
    const float p1 = __fmul_rn(ahi, p);
    const float e1 = __fmaf_rn(ahi, p, -p1);
    float s, t;
    two_sum(hi, p1, s, t);
    const float l = __fadd_rn(lo, __fadd_rn(t, __fmaf_rn(alo, p, e1)));
    two_sum(s, l, hi, lo);
}

// Split an FP64 value into hi + lo floats (hi = fl32(a), lo = fl32(a - hi)).
__device__ __forceinline__ void df_split(double a, float& hi, float& lo) {
    hi = (float)a;
    lo = (float)(a - (double)hi);
}

}  // namespace kry
