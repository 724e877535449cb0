// The three FP32 matvec passes for torus sides 1024 and 2048 (half lengths H =
// 512 = 16 x 32 and 1024 = 32 x 32): 32 values per thread, so that a length-H
// transform is two stages with one exchange through shared memory.
//
// As in fftspec.cuh, a zero-padded transform of length 2H is two transforms of
// length H, q = 0, 1 (X[2k + q]).  Here they run on two neighbouring threads, in
// scalar registers, instead of in the two lanes of one thread's packed
// registers: 32 packed values would take 128 registers and leave 8 warps per
// SM, 16 packed values need a third stage at these lengths, and the
// shared-memory and L1 pipe is what bounds the passes (fftspec.cuh).  Per warp
// of the column pass: 256 wavefronts for the two exchanges (512 with three
// stages), 32 for the shuffles that bring g_0(j) and g_1(j) together.
// Butterflies whose partners share a twiddle (all levels but the last) are packed
// two to an instruction (21 -> 18 million warp instructions, no faster: issue is
// not what bounds).
// Measured against 16 packed values: 4 vectors on 1024^2 69.7 -> 57.5 us (passes
// 15.3 + 36.3 + 20.0 -> 13.5 + 30.3 + 16.6), 64 vectors 921 -> 799 us, 32 vectors
// on 512^2 121 -> 99 us, 5 vectors on 363 x 730 46.5 -> 37.4 us.  What is left:
// the L1 pipe 69% busy while the SMs are, FMA pipe 50%, and 15% (columns) to
// 25% (rows) of a launch's time to start and to run out.
//
// Sides up to 512 and from 4096 up have the same number of stages with 16 and
// 32 values and keep the packed passes.
#pragma once

#include "mvspec.cuh"

namespace kspec {

struct cx {
    float r, i;
};

template <int B>
struct Wide {
    static constexpr int H = 1 << (B - 1);
    static constexpr int E = 32;
    static constexpr int LT = H / E;       // threads per transform and q
    static constexpr int R0 = LT;          // radix of the first stage (the second has 32, at stride R0)
    static constexpr int NB = E / R0;      // first-stage butterflies per thread
    static constexpr int PS = ilog2c(R0);  // shared-memory padding: one position per R0
    static_assert(H == R0 * E && R0 <= E, "two stages");
};

constexpr int wide_nt(int B, int TH) { return TH / lt_of(B); }
constexpr size_t wide_smem(int B, int TH) {
    return (size_t)((1 << (B - 1)) + 32) * wide_nt(B, TH) * 2 * sizeof(float2);
}

// One radix-2 butterfly (a, b) -> (a + w b, a - w b), w = c (1 -+ i T) (forward /
// inverse), times -+i with ROT; bfly of fftspec.cuh on scalars.
template <bool INV, bool ROT>
__device__ __forceinline__ void wbfly(cx& a, cx& b, float c, float T) {
    const float s = INV ? -T : T;
    const float ur = fmaf(s, b.i, b.r), ui = fmaf(-s, b.r, b.i);
    if constexpr (!ROT) {
        b = {fmaf(-c, ur, a.r), fmaf(-c, ui, a.i)};
        a = {fmaf(c, ur, a.r), fmaf(c, ui, a.i)};
    } else if constexpr (!INV) {
        b = {fmaf(-c, ui, a.r), fmaf(c, ur, a.i)};
        a = {fmaf(c, ui, a.r), fmaf(-c, ur, a.i)};
    } else {
        b = {fmaf(c, ui, a.r), fmaf(-c, ur, a.i)};
        a = {fmaf(-c, ui, a.r), fmaf(c, ur, a.i)};
    }
}
template <bool INV, bool ROT>
__device__ __forceinline__ void wbfly1(cx& a, cx& b) {
    const cx x = a, y = b;
    if constexpr (!ROT) {
        a = {x.r + y.r, x.i + y.i};
        b = {x.r - y.r, x.i - y.i};
    } else if constexpr (!INV) {
        a = {x.r + y.i, x.i - y.r};
        b = {x.r - y.i, x.i + y.r};
    } else {
        a = {x.r - y.i, x.i + y.r};
        b = {x.r + y.i, x.i - y.r};
    }
}

// Level 1 on two packed partners: bfly_cs of fftspec.cuh by way of u = w b, which is
// the faster form here (64 vectors on 1024^2 799 us against 810; both forms' error is
// 1.7e-7).
template <bool INV>
__device__ __forceinline__ void wbfly_cs(c2& a, c2& b, u64 c, u64 s) {
    const u64 ns = neg2(s);
    const u64 ur = fma2(INV ? ns : s, b.i, mul2(c, b.r)), ui = fma2(INV ? s : ns, b.r, mul2(c, b.i));
    b = {sub2(a.r, ur), sub2(a.i, ui)};
    a = {add2(a.r, ur), add2(a.i, ui)};
}

// Levels LEV .. log2 R of a radix-R tree (level of fftspec.cuh): twiddle entry
// e at tw[e stride], or (CONST) the constants of a first inverse stage. sign =
// -1 swaps outputs s and s + R/2.
template <int R, int LEV, bool INV, bool CONST>
__device__ __forceinline__ void wlevels(cx* v, const float2* __restrict__ tw, int stride, float sign = 1.f) {
    if constexpr ((1 << LEV) <= R) {
        constexpr int D = R >> LEV, NE = LEV == 1 ? 1 : 1 << (LEV - 2);
        float2 w[NE];
        if constexpr (!CONST) {
#pragma unroll
            for (int e = 0; e < NE; ++e) {
                w[e] = __ldg(tw + (tw_base(LEV) + e) * stride);
                if ((1 << LEV) == R) w[e].x *= sign;
            }
        }
#pragma unroll
        for (int p = 0; p < R; ++p) {
            if (p & D) continue;
            const int s = brev(p / (2 * D), LEV - 1);
            const bool rot = LEV >= 2 && s >= NE;
            const int e = rot ? s - NE : s;
            if constexpr (D >= 2) {   // partners p, p + 1 share the twiddle: one packed butterfly
                if (p & 1) continue;
                c2 a = {pk(v[p].r, v[p + 1].r), pk(v[p].i, v[p + 1].i)};
                c2 b = {pk(v[p + D].r, v[p + D + 1].r), pk(v[p + D].i, v[p + D + 1].i)};
                if (CONST && e == 0) {
                    if (rot) bfly1<INV, true>(a, b);
                    else bfly1<INV, false>(a, b);
                } else {
                    const float c = CONST ? cos32(e * (32 >> LEV)) : w[e].x, T = CONST ? tan32(e * (32 >> LEV)) : w[e].y;
                    if (LEV == 1) wbfly_cs<INV>(a, b, pk(c, c), pk(T, T));
                    else if (rot) bfly<INV, true>(a, b, pk(c, c), pk(T, T));
                    else bfly<INV, false>(a, b, pk(c, c), pk(T, T));
                }
                const float2 ar = upk(a.r), ai = upk(a.i), br = upk(b.r), bi = upk(b.i);
                v[p] = {ar.x, ai.x};
                v[p + 1] = {ar.y, ai.y};
                v[p + D] = {br.x, bi.x};
                v[p + D + 1] = {br.y, bi.y};
                continue;
            }
            if (CONST && e == 0) {
                if (rot) wbfly1<INV, true>(v[p], v[p + D]);
                else wbfly1<INV, false>(v[p], v[p + D]);
                continue;
            }
            const float c = CONST ? cos32(e * (32 >> LEV)) : w[e].x, T = CONST ? tan32(e * (32 >> LEV)) : w[e].y;
            if (rot) wbfly<INV, true>(v[p], v[p + D], c, T);
            else wbfly<INV, false>(v[p], v[p + D], c, T);
        }
        wlevels<R, LEV + 1, INV, CONST>(v, tw, stride, sign);
    }
}

// Twiddle table: for stride NS = 1, 16 and 32, entry e of thread (k, q) at
// section + e 2 NS + 2 k + q: (cos, tan) of (k + q / 2) / NS + s over 2^l turns (entry 0: (cos, sin)).
// Inverse stages take q = 0.
constexpr int wide_section(int NS) { return NS == 1 ? 0 : NS == 16 ? 32 : 32 + 16 * 32; }

// The exchange: a thread's first-stage outputs R0 j + s to shared memory, j = t
// + u LT; then v[r] = position t + r LT of the same transform.
template <int B, bool INV>
__device__ __forceinline__ void wide_exchange(cx* v, float2* __restrict__ sb, int t, int nt2) {
    using P = Wide<B>;
    constexpr int R = P::R0;
    float2* o = sb + t * (R + 1) * nt2;
#pragma unroll
    for (int u = 0; u < P::NB; ++u)
#pragma unroll
        for (int s = 0; s < R; ++s) {
            const cx z = v[u * R + brev(s, ilog2c(R))];
            o[(u * P::LT * (R + 1) + s) * nt2] = make_float2(z.r, z.i);
        }
    __syncthreads();
    const float2* in = sb + t * nt2;   // t < R0: no padding between 0 and t
#pragma unroll
    for (int r = 0; r < P::E; ++r) {
        const float2 z = in[(r * P::LT + r * P::LT / R) * nt2];
        v[r] = {z.x, z.y};
    }
}

// Forward transform q of the inputs at positions t + m LT; pair(m, P, M) gives
// x[m] + b and x[m] - b, b = x[m + 16] (q = 1: times -i): level 1 of the first
// stage.  Frequency k = t + s LT ends in slot bitrev(s).
template <int B, class F>
__device__ __forceinline__ void wide_forward(F&& pair, cx* v, float2* sb, int t, int q, int nt2,
                                             const float2* __restrict__ tw) {
    using P = Wide<B>;
    constexpr int R = P::R0, NB = P::NB;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
#pragma unroll
        for (int r = 0; r < R / 2; ++r) pair(u + r * NB, v[u * R + r], v[u * R + r + R / 2]);
        wlevels<R, 2, false, false>(v + u * R, tw + wide_section(1) + q, 2);
    }
    wide_exchange<B, false>(v, sb, t, nt2);
    wlevels<P::E, 1, false, false>(v, tw + wide_section(R) + 2 * t + q, 2 * R);
}

// Inverse transform g_q of w[m] = frequency t + m LT (w and v may not overlap);
// output t + s LT ends in slot bitrev(s), with s and s + 16 swapped for q = 1.
template <int B>
__device__ __forceinline__ void wide_inverse(const cx* w, cx* v, float2* sb, int t, int q, int nt2,
                                             const float2* __restrict__ tw) {
    using P = Wide<B>;
    constexpr int R = P::R0, NB = P::NB;
#pragma unroll
    for (int u = 0; u < NB; ++u) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[u * R + r] = w[u + r * NB];
        wlevels<R, 1, true, true>(v + u * R, nullptr, 0);
    }
    wide_exchange<B, true>(v, sb, t, nt2);
    wlevels<P::E, 1, true, false>(v, tw + wide_section(R) + 2 * t, 2 * R, q ? -1.f : 1.f);
}

// y_j = g_0(j) + W_L^{-j} g_1(j): the threads q = 0, 1 trade halves, and thread
// q keeps the 16 outputs j = t + (s + 16 q) LT.
template <int B>
__device__ __forceinline__ void wide_post(const cx* v, float2* y, int t, int q, const float2* __restrict__ post) {
    using P = Wide<B>;
    const float2* pw = post + (P::H - 32) + t + q * 16 * P::LT;
#pragma unroll
    for (int s = 0; s < 16; ++s) {
        const cx k = v[brev(s, 5)], g = v[brev(s + 16, 5)];
        const float rr = __shfl_xor_sync(0xffffffffu, g.r, 1), ri = __shfl_xor_sync(0xffffffffu, g.i, 1);
        const float2 f = __ldg(pw + s * P::LT);
        const float ar = q ? rr : k.r, ai = q ? ri : k.i, br = q ? k.r : rr, bi = q ? k.i : ri;
        y[s] = make_float2(fmaf(f.x, br, fmaf(-f.y, bi, ar)), fmaf(f.x, bi, fmaf(f.y, br, ai)));
    }
}

// A pair's slab addressed by 32-bit byte offsets (n1 M2 8 <= 2^28).
__device__ __forceinline__ float2& at(float2* base, unsigned off) {
    return *reinterpret_cast<float2*>(reinterpret_cast<char*>(base) + off);
}
__device__ __forceinline__ float2 at(const float2* base, unsigned off) {
    return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(base) + off);
}

// ---------------------------------------------------------------- passes
// As ks_pass_a, _b, _c; thread = (t, transform n, q), q fastest.

template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    kw_pass_a(const float* __restrict__ vin, int64_t ld, const double* __restrict__ scale, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int logCs, float2* __restrict__ slab,
              const float2* __restrict__ tw, const int* __restrict__ skip) {
    using P = Wide<B>;
    constexpr int LT = P::LT, NT = wide_nt(B, TH);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int q = threadIdx.x & 1, n = (threadIdx.x >> 1) & (NT - 1), t = threadIdx.x / (2 * NT);
    pdl_wait();
    pdl_launch_dependents();
    const int row = blockIdx.x * NT + n;
    const int pair = pair0 + blockIdx.y;
    const int va = 2 * pair, vb = 2 * pair + 1;
    const bool has_b = vb < nvec;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const bool live = row < n1;

    float2 own[16];   // cells t + (i + 16 q) LT; the other half comes from the neighbouring thread
    {
        const float sa = FWD_SCALE * (scale ? (float)scale[va] : 1.f);
        const float sbv = FWD_SCALE * ((scale && has_b) ? (float)scale[vb] : 1.f);
        const float* pa = vin + (int64_t)va * ld;
        const float* pb = has_b ? vin + (int64_t)vb * ld : pa;
        int c[16];
        cell_indices<LT, 16>(bits + (int64_t)min(row, n1 - 1) * wpr, wpr, live, t + q * 16 * LT, c);
#pragma unroll
        for (int i = 0; i < 16; ++i) own[i] = make_float2(pa[max(c[i], 0)], pb[max(c[i], 0)]);
#pragma unroll
        for (int i = 0; i < 16; ++i)
            own[i] = make_float2(c[i] >= 0 ? own[i].x * sa : 0.f, c[i] >= 0 && has_b ? own[i].y * sbv : 0.f);
    }
    cx v[P::E];
    const float sg = q ? -1.f : 1.f;
    auto pair_sum = [&](int m, cx& p, cx& d) {
        // q = 0: own +- other; q = 1: other +- (-i own)
        const float2 o = own[m];
        const float rx = __shfl_xor_sync(0xffffffffu, o.x, 1), ry = __shfl_xor_sync(0xffffffffu, o.y, 1);
        const float zr = q ? o.y : o.x, zi = q ? -o.x : o.y;
        p = {zr + rx, zi + ry};
        d = {sg * (zr - rx), sg * (zi - ry)};
    };
    wide_forward<B>(pair_sum, v, reinterpret_cast<float2*>(smem_raw) + n * 2 + q, t, q, 2 * NT, tw);
    if (!live) return;
    // columns 2k + q, k = t + s LT: 2 LT columns are whole tiles (tiles of at most 32 columns)
    const unsigned col = 2 * t + q;
    float2* out = slab + (((int64_t)blockIdx.y * n1) << B);
    const unsigned off = (((((col >> logCs) * n1 + row) << logCs) + (col & ((1u << logCs) - 1))) * 8), step = n1 * (2 * LT * 8);
#pragma unroll
    for (int s = 0; s < P::E; ++s) {
        const cx z = v[brev(s, 5)];
        at(out, off + s * step) = make_float2(z.r, z.i);
    }
}

template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    kw_pass_b(float2* __restrict__ slab, const float* __restrict__ lamP, int n1, int M2, int logCs,
              const float2* __restrict__ tw, const float2* __restrict__ post, int pair0, int64_t lam_stride, int vpt,
              const int* __restrict__ skip, int nvec) {
    using P = Wide<B>;
    constexpr int LT = P::LT, NT = wide_nt(B, TH);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int q = threadIdx.x & 1, n = (threadIdx.x >> 1) & (NT - 1), t = threadIdx.x / (2 * NT);
    const int col = blockIdx.x * NT + n;
    const int theta = vpt ? (2 * (pair0 + (int)blockIdx.y)) / vpt : 0;
    const float4* lam = reinterpret_cast<const float4*>(lamP + theta * lam_stride + (int64_t)col * (2 * P::H)) + 2 * t + q;
    float2* sb = reinterpret_cast<float2*>(smem_raw) + n * 2 + q;
    pdl_wait();   // the slab comes from pass A
    pdl_launch_dependents();
    if (skip) {
        const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
        if (skip[va] && (vb >= nvec || skip[vb])) return;
    }
    float2* blk = slab + (int64_t)blockIdx.y * n1 * M2;
    const unsigned off = ((((col >> logCs) * n1 + t) << logCs) + (col & ((1u << logCs) - 1))) * 8, step = (LT * 8) << logCs;
    const bool whole = n1 == P::H;   // no row to leave out (uniform)
    cx v[P::E], w[P::E];
    {
        float2 x[P::E];
        if (whole) {
#pragma unroll
            for (int m = 0; m < P::E; ++m) x[m] = at(blk, off + m * step);
        } else {
#pragma unroll
            for (int m = 0; m < P::E; ++m) x[m] = (t + m * LT < n1) ? at(blk, off + m * step) : make_float2(0.f, 0.f);
        }
        auto pair_sum = [&](int m, cx& p, cx& d) {
            const float2 a = x[m], b = x[m + 16];
            const float br = q ? b.y : b.x, bi = q ? -b.x : b.y;
            p = {a.x + br, a.y + bi};
            d = {a.x - br, a.y - bi};
        };
        wide_forward<B>(pair_sum, v, sb, t, q, 2 * NT, tw);
    }
#pragma unroll
    for (int s = 0; s < P::E; s += 4) {
        const float4 l = __ldg(lam + (s >> 2) * (2 * LT));
        const cx a = v[brev(s, 5)], b = v[brev(s + 1, 5)], c = v[brev(s + 2, 5)], d = v[brev(s + 3, 5)];
        w[s] = {a.r * l.x, a.i * l.x};
        w[s + 1] = {b.r * l.y, b.i * l.y};
        w[s + 2] = {c.r * l.z, c.i * l.z};
        w[s + 3] = {d.r * l.w, d.i * l.w};
    }
    __syncthreads();   // every read of the forward transform's exchange is done
    wide_inverse<B>(w, v, sb, t, q, 2 * NT, tw);
    float2 y[16];
    wide_post<B>(v, y, t, q, post);
    const unsigned o = off + q * 16 * step;
#pragma unroll
    for (int i = 0; i < 16; ++i)
        if (whole || t + (i + 16 * q) * LT < n1) at(blk, o + i * step) = y[i];
}

template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    kw_pass_c(const float2* __restrict__ slab, const float* __restrict__ vin, int64_t ld_in,
              const double* __restrict__ scale, float* __restrict__ vout, int64_t ld_out, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int logCs, double tau2, double* __restrict__ dots,
              int ndot_stride, const float2* __restrict__ tw, const float2* __restrict__ post,
              const double* __restrict__ tau2v, int vpt, const int* __restrict__ skip) {
    using P = Wide<B>;
    constexpr int LT = P::LT, NT = wide_nt(B, TH);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int q = threadIdx.x & 1, n = (threadIdx.x >> 1) & (NT - 1), t = threadIdx.x / (2 * NT);
    pdl_wait();   // the slab comes from pass B
    pdl_launch_dependents();
    const int row = blockIdx.x * NT + n;
    const int pair = pair0 + blockIdx.y;
    const int va = 2 * pair, vb = 2 * pair + 1;
    const bool has_b = vb < nvec;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const bool live = row < n1;
    float2 y[16];
    {
        cx w[P::E], v[P::E];
        const unsigned col = 2 * t + q;
        const float2* in = slab + (((int64_t)blockIdx.y * n1) << B);
        const unsigned off = ((((col >> logCs) * n1 + min(row, n1 - 1)) << logCs) + (col & ((1u << logCs) - 1))) * 8;
        const unsigned step = n1 * (2 * LT * 8);
#pragma unroll
        for (int s = 0; s < P::E; ++s) {
            const float2 f = at(in, off + s * step);
            w[s] = {f.x, f.y};
        }
        wide_inverse<B>(w, v, reinterpret_cast<float2*>(smem_raw) + n * 2 + q, t, q, 2 * NT, tw);
        wide_post<B>(v, y, t, q, post);
    }
    kry::DFAcc acc[2];
    {
        const float sa = scale ? (float)scale[va] : 1.f;
        const float sbv = (scale && has_b) ? (float)scale[vb] : 1.f;
        const float t2 = (float)(tau2v ? tau2v[vpt ? va / vpt : 0] : tau2);
        const float* pa = vin + (int64_t)va * ld_in;
        const float* pb = has_b ? vin + (int64_t)vb * ld_in : pa;
        float* oa = vout + (int64_t)va * ld_out;
        float* ob = vout + (int64_t)vb * ld_out;
        int c[16];
        cell_indices<LT, 16>(bits + (int64_t)min(row, n1 - 1) * wpr, wpr, live, t + q * 16 * LT, c);
        float2 x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = make_float2(pa[max(c[i], 0)], pb[max(c[i], 0)]);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            x[i] = make_float2(x[i].x * sa, x[i].y * sbv);
            y[i] = make_float2(y[i].x + t2 * x[i].x, y[i].y + t2 * x[i].y);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            if (c[i] >= 0) oa[c[i]] = y[i].x;
            if (c[i] >= 0 && has_b) ob[c[i]] = y[i].y;
        }
        if (dots) {
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const bool on = c[i] >= 0;   // what lies in unobserved cells stays out of the sums
                acc[0].add_prod(on ? x[i].x : 0.f, on ? y[i].x : 0.f);
                acc[1].add_prod(on ? x[i].y : 0.f, on ? y[i].y : 0.f);
            }
        }
    }
    if (dots != nullptr) {
        const double s = kry::block_sums<2, TH / 32>(acc);
        if (threadIdx.x == 0) dots[(int64_t)va * ndot_stride + blockIdx.x] = s;
        if (threadIdx.x == TH / 32 && has_b) dots[(int64_t)vb * ndot_stride + blockIdx.x] = s;
    }
}

}  // namespace kspec
