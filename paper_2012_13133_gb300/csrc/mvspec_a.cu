// Pass A of the specialised FP32 matvec (mvspec.cuh) for every supported
// (log2 M2, threads per block), the block sizes and the twiddle tables.
#include "kry_internal.cuh"
#include "mvspec.cuh"
#include "mvwide.cuh"

namespace kspec {

int transform_threads(int M) { return lt_of(ilog2i(M)); }

int block_threads(int M, int nt, int most) {
    const int lt = transform_threads(M), cap = max_threads(ilog2i(M));
    int th = lt;
    while (th < lt * nt && 2 * th <= cap && 2 * (th / lt) <= most) th *= 2;
    while (th < 32) th *= 2;
    return th;
}

// Entry e = s + 2^{l-2} of level l at stride ns, frequency k: (cos, tan) of its angle,
// (k / ns + s) / 2^l of a turn, the tangent that goes with the rounded cosine; entry
// 0 (level 1): (cos, sin).
__device__ __forceinline__ float2 entry(int e, int ns, double k) {
    const int l = e == 0 ? 1 : 2 + (31 - __clz(e));
    double s, c;
    sincospi(2.0 * (k / ns + (e - tw_base(l))) / (double)(1 << l), &s, &c);
    return make_float2((float)c, (float)(e == 0 ? s : s / (double)(float)c));
}

__global__ void k_tables(float4* __restrict__ tab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < TWF_WORDS) {
        const int ns = 1 << (31 - __clz(i / 8 + 2));   // sections of 8 ns words from 8 (ns - 2)
        const int r = i - 8 * (ns - 2), e = r / ns, k = r - e * ns;
        const float2 a = entry(e, ns, k), b = entry(e, ns, k + 0.5);
        tab[i] = make_float4(a.x, b.x, a.y, b.y);
    } else if (i < TWF_WORDS + TWI_WORDS) {
        const int w = i - TWF_WORDS;
        const int ns = 1 << (31 - __clz(w / 4 + 2));
        const int r = w - 4 * (ns - 2), e = r / ns, k = r - e * ns;
        const float2 a = entry(2 * e, ns, k), b = entry(2 * e + 1, ns, k);
        tab[i] = make_float4(a.x, a.y, b.x, b.y);
    } else if (i < TWF_WORDS + TWI_WORDS + POST_WORDS / 2) {
        float2 f[2];
        for (int q = 0; q < 2; ++q) {
            const int w = 2 * (i - TWF_WORDS - TWI_WORDS) + q;   // sections of h words from h - 32
            const int h = 1 << (31 - __clz(w + 32));
            double s, c;
            sincospi((double)(w + 32 - h) / (double)h, &s, &c);
            f[q] = make_float2((float)c, (float)s);
        }
        tab[i] = make_float4(f[0].x, f[0].y, f[1].x, f[1].y);
    } else if (i < TABLE_WORDS) {
        const int w = 2 * (i - TWF_WORDS - TWI_WORDS - POST_WORDS / 2);
        const int ns = w < wide_section(16) ? 1 : w < wide_section(32) ? 16 : 32;
        const int r = w - wide_section(ns), e = r / (2 * ns), k = (r - e * 2 * ns) >> 1;
        const float2 a = entry(e, ns, k), b = entry(e, ns, k + 0.5);
        tab[i] = make_float4(a.x, a.y, b.x, b.y);
    }
}

void fill_tables(float4* tab_dev, cudaStream_t st) {
    k_tables<<<(TABLE_WORDS + 255) / 256, 256, 0, st>>>(tab_dev);
    KRY_CHECK_LAUNCH();
}

namespace {
struct RunA {
    const SpecArgs& a;
    cudaStream_t st;
    template <int B, int TH>
    bool run() const {
        constexpr int NT = nt_of(B, TH);
        dim3 grid((a.n1 + NT - 1) / NT, a.np);
        if constexpr (is_wide(B)) {
            auto k = kw_pass_a<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), wide_smem(B, TH), st, a.vin, a.ld_in, a.scale, a.nvec, a.pair0, a.bits, a.wpr,
                       a.n1, a.logCs, a.slab, a.tww, a.skip);
        } else {
            auto k = ks_pass_a<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), smem_bytes(B, TH), st, a.vin, a.ld_in, a.scale, a.nvec, a.pair0, a.bits, a.wpr,
                       a.n1, a.logCs, reinterpret_cast<float4*>(a.slab), a.twf, a.skip);
        }
        return true;
    }
};
}  // namespace

bool launch_a(const SpecArgs& a, cudaStream_t st) { return dispatch(ilog2i(a.M2), a.G * transform_threads(a.M2), RunA{a, st}); }

}  // namespace kspec
