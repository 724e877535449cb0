// The three FP32 matvec passes (Sec. 3: K v = A F^-1 (Lambda . F (A^T v)) +
// tau^2 v on the circulant embedding) specialised for torus side L = 2^B and
// a block of TH threads; see fftspec.cuh for the transforms.  Each translation
// unit mvspec_{a,b,c}.cu instantiates one pass for every supported (B, TH)
// and exposes a runtime dispatcher; matvec.cu calls them for FP32 batches.
//
// Layouts:
//  * slab: per complex pair an n1 x M2 complex intermediate, stored in column
//    tiles slab[pair][tile][i][c], c < Cs, tile = column / Cs (Cs even, so the
//    two columns 2k, 2k + 1 that a row transform produces in its two lanes
//    are one 16-byte word);
//  * lamP: eigenvalues per column j at j M1, scaled by 1 / (M1 M2 FWD_SCALE), permuted
//    so that the values a column-pass thread multiplies are 16-byte words
//    consecutive over threads (lam_slot);
//  * bits: per 32 cells of a grid row, the observation bits and the index of
//    the first observed cell among them, so that a thread finds the vector
//    index of any cell with one load and a bit count.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "dfloat.cuh"
#include "fftspec.cuh"
#include "kry_internal.cuh"

namespace kspec {

// Threads per transform of torus side 2^B, transforms per block of TH threads.
__host__ __device__ constexpr int lt_of(int B) { return (1 << (B - 1)) / 16; }
constexpr int nt_of(int B, int TH) { return TH / lt_of(B); }
// Registers: 64 of a thread's 128 hold the transform: 512 threads per SM.
// (Measured on side 2048 with 16 packed values, 64 vectors: 96 registers and 640
// threads 1195 us against 913 us; 32 packed values, one shared-memory exchange
// fewer, but 8 warps per SM, 982 us.)
// Sides up to 256 are latency, not throughput: their passes load everything as
// soon as they may, into up to 255 registers (4 vectors on 128^2 10.7 -> 9.6 us, a
// CG iteration on them 24.1 -> 22.1 us).
constexpr bool early(int B) { return B <= 8; }
constexpr int minb(int B, int TH) {
    const int resident = early(B) ? 256 : 512;
    return TH >= resident ? 1 : resident / TH;
}

// Shared-memory bytes of a block.
constexpr size_t smem_bytes(int B, int TH) {
    return (size_t)((1 << (B - 1)) + ((1 << (B - 1)) >> pad_shift(1 << (B - 1)))) * nt_of(B, TH) * 16;
}

// Torus sides whose passes hold 32 values per thread (mvwide.cuh).
__host__ __device__ constexpr bool is_wide(int B) { return B == 10 || B == 11; }

// Offset within a column of M1 eigenvalues of torus row k1 = 2 k + q, k = t +
// s lt, lt = threads per transform: word (s/2) lt + t holds (s even: q = 0, 1;
// s odd: q = 0, 1).  Sides with 32 values per thread: k = t + s lt/2, and word
// (s/4) lt + 2t + q holds s .. s + 3.
__host__ __device__ __forceinline__ int lam_slot(int k1, int M1, int lt) {
    const int q = k1 & 1, k = k1 >> 1;
    if (M1 == 1024 || M1 == 2048) {
        const int h = lt >> 1, t = k & (h - 1), s = k / h;
        return ((s >> 2) * lt + 2 * t + q) * 4 + (s & 3);
    }
    const int t = k & (lt - 1), s = k / lt;
    return ((s >> 1) * lt + t) * 4 + (s & 1) * 2 + q;
}

// Vector indices of a thread's E cells j = t + m LT of a row with wpr
// observation words w, -1 where the cell is not observed (or beyond the row:
// the bits of a row's last word end at its last cell).  All loads are
// unconditional, at clamped addresses: behind branches the compiler issues
// the dependent load chains one after the other (pass A 473 us instead of
// 209, 64 vectors on 1024^2).
template <int LT, int E>
__device__ __forceinline__ void cell_indices(const uint2* __restrict__ w, int wpr, bool live, int t, int (&q)[E]) {
    uint2 b[E];
#pragma unroll
    for (int m = 0; m < E; ++m) b[m] = __ldg(w + min((t + m * LT) >> 5, wpr - 1));
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int j = t + m * LT;
        const unsigned bit = 1u << (j & 31);
        const bool on = live && (b[m].x & bit) != 0u && (j >> 5) < wpr;
        q[m] = on ? (int)(b[m].y + __popc(b[m].x & (bit - 1u))) : -1;
    }
}

// Post factors of a thread's E outputs t + s LT.
template <int E, int LT>
__device__ __forceinline__ void load_post(float2 (&f)[E], const float2* __restrict__ pw) {
#pragma unroll
    for (int s = 0; s < E; ++s) f[s] = __ldg(pw + s * LT);
}

// ---------------------------------------------------------------- pass A
// Row transforms of NT rows: every thread picks its cells' values straight
// from the observed vectors (two real vectors as re/im; the observed cells of
// a row are in column order, so neighbouring threads read neighbouring
// values), forward FFT, columns 2k and 2k + 1 to the slab as one word.
template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    ks_pass_a(const float* __restrict__ vin, int64_t ld, const double* __restrict__ scale, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int logCs, float4* __restrict__ slab,
              const float4* __restrict__ twf, const int* __restrict__ skip) {
    using P = Plan<B>;
    constexpr int H = P::H, E = P::E, LT = P::LT, NT = nt_of(B, TH), PS = pad_shift(H);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    StageTw<16> tw1;   // constant tables: their latency lies behind the kernel before
    load_twiddles<E, P::R0, false>(tw1, twf, t);
    pdl_wait();        // the vectors and skip flags come from the kernel before
    pdl_launch_dependents();
    const int row = blockIdx.x * NT + n;
    const int pair = pair0 + blockIdx.y;
    const int va = 2 * pair, vb = 2 * pair + 1;
    const bool has_b = vb < nvec;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const bool live = row < n1;
    c2* sb = reinterpret_cast<c2*>(smem_raw) + n;

    float2 x[E];
    {
        const float sa = FWD_SCALE * (scale ? (float)scale[va] : 1.f);
        const float sbv = FWD_SCALE * ((scale && has_b) ? (float)scale[vb] : 1.f);
        const float* pa = vin + (int64_t)va * ld;
        const float* pb = has_b ? vin + (int64_t)vb * ld : pa;
        int q[E];
        cell_indices<LT, E>(bits + (int64_t)min(row, n1 - 1) * wpr, wpr, live, t, q);
#pragma unroll
        for (int m = 0; m < E; ++m) x[m] = make_float2(pa[max(q[m], 0)], pb[max(q[m], 0)]);
#pragma unroll
        for (int m = 0; m < E; ++m)
            x[m] = make_float2(q[m] >= 0 ? x[m].x * sa : 0.f, q[m] >= 0 && has_b ? x[m].y * sbv : 0.f);
    }
    const int tb = soff<PS, NT>(t);
    auto lds = [&](int c) { return sb[tb + soff<PS, NT>(c)]; };
    auto sts = [&](int bo, int c, c2 z) { sb[soff<PS, NT>(bo) + soff<PS, NT>(c)] = z; };
    first_forward<B>(x, t, sts);
    c2 v[E];
    later_stages<B, 1, false>(v, tw1, t, twf, lds, sts);
    if (!live) return;
    // word of columns 2k, 2k + 1, k = t + s LT
    const int logk = logCs - 1;   // words per tile row
    float4* out = slab + (((int64_t)blockIdx.y * n1) << (B - 1));
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int k = t + s * LT;
        const c2 z = v[brev(s, P::LE)];
        const float2 re = upk(z.r), im = upk(z.i);
        out[(((int64_t)(k >> logk) * n1 + row) << logk) + (k & ((1 << logk) - 1))] = make_float4(re.x, im.x, re.y, im.y);
    }
}

// ---------------------------------------------------------------- pass B
// Column transforms of NT columns: forward, multiply by Lambda in registers,
// inverse, keep rows < n1 (in place in the slab).
template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    ks_pass_b(float2* __restrict__ slab, const float* __restrict__ lamP, int n1, int M2, int logCs,
              const float4* __restrict__ twf, const float4* __restrict__ twi, const float2* __restrict__ post, int pair0,
              int64_t lam_stride, int vpt, const int* __restrict__ skip, int nvec) {
    using P = Plan<B>;
    constexpr int L = P::L, H = P::H, E = P::E, LT = P::LT, NT = nt_of(B, TH), PS = pad_shift(H);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int col = blockIdx.x * NT + n;
    // constant tables: their latency lies behind the kernel before
    StageTw<16> tw1;
    load_twiddles<E, P::R0, false>(tw1, twf, t);
    const int theta = vpt ? (2 * (pair0 + (int)blockIdx.y)) / vpt : 0;
    const float4* lam = reinterpret_cast<const float4*>(lamP + theta * lam_stride + (int64_t)col * L) + t;
    const float2* pw = post + (H - 32) + t;
    float2 f[E];
    if constexpr (early(B)) load_post<E, LT>(f, pw);
    pdl_wait();   // the slab comes from pass A
    pdl_launch_dependents();
    if (skip) {
        const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
        if (skip[va] && (vb >= nvec || skip[vb])) return;
    }
    c2* sb = reinterpret_cast<c2*>(smem_raw) + n;
    float2* blk = slab + (int64_t)blockIdx.y * n1 * M2 + (((int64_t)(col >> logCs) * n1 + t) << logCs) +
                  (col & ((1 << logCs) - 1));
    const int tb = soff<PS, NT>(t);
    auto lds = [&](int c) { return sb[tb + soff<PS, NT>(c)]; };
    auto sts = [&](int bo, int c, c2 z) { sb[soff<PS, NT>(bo) + soff<PS, NT>(c)] = z; };
    c2 v[E];
    float4 lw[E / 2];
    {
        float2 x[E];
#pragma unroll
        for (int m = 0; m < E; ++m)
            x[m] = (t + m * LT < n1) ? blk[(int64_t)(m * LT) << logCs] : make_float2(0.f, 0.f);
        if constexpr (early(B)) {
#pragma unroll
            for (int s = 0; s < E / 2; ++s) lw[s] = __ldg(lam + s * LT);
        }
        first_forward<B>(x, t, sts);
    }
    later_stages<B, 1, false>(v, tw1, t, twf, lds, sts);

    c2 w[E];
#pragma unroll
    for (int s = 0; s < E; s += 2) {
        const float4 l = early(B) ? lw[s >> 1] : __ldg(lam + (s >> 1) * LT);
        const c2 a = v[brev(s, P::LE)], b = v[brev(s + 1, P::LE)];
        const u64 la = pk(l.x, l.y), lb = pk(l.z, l.w);
        w[s] = {mul2(a.r, la), mul2(a.i, la)};
        w[s + 1] = {mul2(b.r, lb), mul2(b.i, lb)};
    }
    __syncthreads();   // every read of the forward transform's last stage is done
    first_inverse<B>(w, t, sts);
    load_twiddles<E, P::R0, true>(tw1, twi, t);
    later_stages<B, 1, true>(v, tw1, t, twi, lds, sts);
#pragma unroll
    for (int s = 0; s < E; ++s) {
        if (t + s * LT < n1) {
            const c2 z = v[brev(s, P::LE)];
            const float2 re = upk(z.r), im = upk(z.i), g = early(B) ? f[s] : __ldg(pw + s * LT);
            blk[(int64_t)(s * LT) << logCs] = make_float2(fmaf(g.x, re.y, fmaf(-g.y, im.y, re.x)),
                                                          fmaf(g.x, im.y, fmaf(g.y, re.y, im.x)));
        }
    }
}

// ---------------------------------------------------------------- pass C
// Inverse row transforms of NT slab rows; every thread then writes its observed
// cells of K v straight from registers, adds the nugget and (dots != NULL)
// accumulates v . K v, one FP64 partial per block.
template <int B, int TH>
__global__ void __launch_bounds__(TH, minb(B, TH))
    ks_pass_c(const float4* __restrict__ slab, const float* __restrict__ vin, int64_t ld_in,
              const double* __restrict__ scale, float* __restrict__ vout, int64_t ld_out, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int logCs, double tau2,
              double* __restrict__ dots, int ndot_stride, const float4* __restrict__ twi,
              const float2* __restrict__ post, const double* __restrict__ tau2v, int vpt,
              const int* __restrict__ skip) {
    using P = Plan<B>;
    constexpr int H = P::H, E = P::E, LT = P::LT, NT = nt_of(B, TH), PS = pad_shift(H);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    StageTw<16> tw1;   // constant tables: their latency lies behind the kernel before
    load_twiddles<E, P::R0, true>(tw1, twi, t);
    const float2* pw = post + (H - 32) + t;
    float2 pf[E];
    if constexpr (early(B)) load_post<E, LT>(pf, pw);
    pdl_wait();   // the slab comes from pass B
    pdl_launch_dependents();
    const int row = blockIdx.x * NT + n;
    const int pair = pair0 + blockIdx.y;
    const int va = 2 * pair, vb = 2 * pair + 1;
    const bool has_b = vb < nvec;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const bool live = row < n1;
    c2* sb = reinterpret_cast<c2*>(smem_raw) + n;
    const int tb = soff<PS, NT>(t);
    auto lds = [&](int c) { return sb[tb + soff<PS, NT>(c)]; };
    auto sts = [&](int bo, int c, c2 z) { sb[soff<PS, NT>(bo) + soff<PS, NT>(c)] = z; };
    const float* pa = vin + (int64_t)va * ld_in;
    const float* pb = has_b ? vin + (int64_t)vb * ld_in : pa;
    const uint2* bw = bits + (int64_t)min(row, n1 - 1) * wpr;
    int q[E];
    float2 x[E];
    auto load_cells = [&]() {
        cell_indices<LT, E>(bw, wpr, live, t, q);
#pragma unroll
        for (int i = 0; i < E; ++i) x[i] = make_float2(pa[max(q[i], 0)], pb[max(q[i], 0)]);
    };
    c2 v[E];
    {
        const int logk = logCs - 1;
        const float4* in = slab + (((int64_t)blockIdx.y * n1) << (B - 1));
        c2 w[E];
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const int k = t + s * LT;
            const float4 f = in[(((int64_t)(k >> logk) * n1 + min(row, n1 - 1)) << logk) + (k & ((1 << logk) - 1))];
            w[s] = {pk(f.x, f.z), pk(f.y, f.w)};
        }
        if constexpr (early(B)) load_cells();
        first_inverse<B>(w, t, sts);
    }
    later_stages<B, 1, true>(v, tw1, t, twi, lds, sts);

    kry::DFAcc acc[2];
    {
        const float sa = scale ? (float)scale[va] : 1.f;
        const float sbv = (scale && has_b) ? (float)scale[vb] : 1.f;
        const float t2 = (float)(tau2v ? tau2v[vpt ? va / vpt : 0] : tau2);
        float* oa = vout + (int64_t)va * ld_out;
        float* ob = vout + (int64_t)vb * ld_out;
        if constexpr (!early(B)) load_cells();
        float2 y[E];
#pragma unroll
        for (int i = 0; i < E; ++i) {
            const c2 z = v[brev(i, P::LE)];
            const float2 re = upk(z.r), im = upk(z.i), f = early(B) ? pf[i] : __ldg(pw + i * LT);
            y[i] = make_float2(fmaf(f.x, re.y, fmaf(-f.y, im.y, re.x)), fmaf(f.x, im.y, fmaf(f.y, re.y, im.x)));
        }
#pragma unroll
        for (int i = 0; i < E; ++i) {
            x[i] = make_float2(x[i].x * sa, x[i].y * sbv);
            y[i] = make_float2(y[i].x + t2 * x[i].x, y[i].y + t2 * x[i].y);
        }
#pragma unroll
        for (int i = 0; i < E; ++i) {
            if (q[i] >= 0) oa[q[i]] = y[i].x;
            if (q[i] >= 0 && has_b) ob[q[i]] = y[i].y;
        }
        if (dots) {
#pragma unroll
            for (int i = 0; i < E; ++i) {
                const bool on = q[i] >= 0;   // what lies in unobserved cells stays out of the sums
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

// ---------------------------------------------------------------- dispatch

// Arguments of one specialised matvec pass triple (per batch of pairs).
struct SpecArgs {
    const float* vin;
    int64_t ld_in;
    const double* scale;
    float* vout;
    int64_t ld_out;
    int nvec, pair0, np;
    const uint2* bits;
    int wpr;
    int n1, M1, M2;
    int G, C, logCs;   // rows per block (A, C), columns per block (B), log2 of the slab tile width
    float2* slab;
    const float* lamP;   // column-permuted FP32 eigenvalues (kry_embed::lam32P)
    int64_t lam_stride;
    int vpt;
    double tau2;
    const double* tau2v;
    double* dots;
    int nds;
    const float4* twf;
    const float4* twi;
    const float2* post;
    const float2* tww;   // twiddles of the 32-value passes
    const int* skip;
};

// Largest block compiled for torus side 2^B.
constexpr int max_threads(int B) { return B >= 12 ? 512 : B >= 8 ? 256 : 128; }

// Threads per transform of torus side M.
int transform_threads(int M);

// Threads per block of a pass that puts nt transforms of torus side M in a
// block: at least a warp, at most max_threads, never more transforms than
// `most`.
int block_threads(int M, int nt, int most);

// Launch pass A, B or C (false if the shape is not compiled).
bool launch_a(const SpecArgs& a, cudaStream_t st);
bool launch_b(const SpecArgs& a, cudaStream_t st);
bool launch_c(const SpecArgs& a, cudaStream_t st);

// Words (16 bytes) of the tables that fill_tables writes: forward twiddles,
// inverse twiddles, post factors and the 32-value passes' twiddles (two per word).
constexpr int TWW_WORDS = 32 + 16 * 32 + 16 * 64;
constexpr int TABLE_WORDS = TWF_WORDS + TWI_WORDS + POST_WORDS / 2 + TWW_WORDS / 2;
void fill_tables(float4* tab_dev, cudaStream_t st);

}  // namespace kspec

namespace kspec {

// Calls f.template run<B, TH>() for a runtime (B, TH); false otherwise.
template <int B, int TH, class F>
bool dispatch_one(const F& f) {
    if constexpr (lt_of(B) <= TH && TH <= max_threads(B)) return f.template run<B, TH>();
    return false;
}

template <int B, class F>
bool dispatch_th(int th, const F& f) {
    switch (th) {
        case 32: return dispatch_one<B, 32>(f);
        case 64: return dispatch_one<B, 64>(f);
        case 128: return dispatch_one<B, 128>(f);
        case 256: return dispatch_one<B, 256>(f);
        case 512: return dispatch_one<B, 512>(f);
        default: return false;
    }
}

template <class F>
bool dispatch(int b, int th, const F& f) {
    switch (b) {
        case 6: return dispatch_th<6>(th, f);
        case 7: return dispatch_th<7>(th, f);
        case 8: return dispatch_th<8>(th, f);
        case 9: return dispatch_th<9>(th, f);
        case 10: return dispatch_th<10>(th, f);
        case 11: return dispatch_th<11>(th, f);
        case 12: return dispatch_th<12>(th, f);
        case 13: return dispatch_th<13>(th, f);
        default: return false;
    }
}

inline int ilog2i(int x) { return 31 - __builtin_clz((unsigned)x); }

}  // namespace kspec
