// Circulant embedding of the BTTB covariance and its eigenvalues (Sec. 3.3:
// the block-circulant matrix built from one row of Sigma; Appendix A,
// Eq. circ_diag: a BCCB matrix is diagonalised by the 2-D Fourier matrix),
// and Gaussian-process sampling on the same embedding (Sec. 3.5 bootstrap;
// Sec. 3.6 caveat on negative eigenvalues).
//
// The first row c of the embedding lives on an M1 x M2 torus, M_d the
// smallest power of two >= 2 n_d.  A torus index j maps to the lag of its
// minimal image (j, or j - M when j > M/2); at j = M/2 the two images +-M/2
// are averaged, which keeps c symmetric under j -> -j (and Lambda real) for
// anisotropic covariances too.  Lambda = FFT2(c) in FP64.
#include <algorithm>

#include "fft64.cuh"
#include "kry_internal.cuh"
#include "matern.cuh"
#include "mv64.cuh"
#include "mvspec.cuh"

namespace kry {

// ------------------------------------------------------------------ twiddles

__global__ void k_twiddles(float2* tw32) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= KRY_TWN) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)KRY_TWN, &s, &c);
    tw32[k] = make_float2((float)c, (float)s);
}

void init_twiddles(kry_ctx* ctx) {
    ctx->tw32.ensure(KRY_TWN * sizeof(float2));
    k_twiddles<<<(KRY_TWN + 255) / 256, 256, 0, ctx->stream>>>(ctx->tw32.as<float2>());
    KRY_CHECK_LAUNCH();
    ctx->tab64.ensure((size_t)kf64::TW_WORDS * sizeof(double2));
    kf64::fill_table(ctx->tab64.as<double2>(), ctx->stream);
    ctx->spec_tab.ensure((size_t)kspec::TABLE_WORDS * sizeof(float4));
    kspec::fill_tables(ctx->spec_tab.as<float4>(), ctx->stream);
}

// ------------------------------------------------------------------ lag covariance

// Covariance parameters of one evaluation, scaled for it: x = s d with s =
// sqrt(2 nu) / range.
struct CovDev {
    double sigma2, inv_range, nu, s, ca, sa, ratio, dx1, dx2;
    int kind;   // 0, 1, 2: nu = 1/2, 3/2, 5/2 (closed forms); 3: any other nu
    bool even;  // d is even in each lag coordinate by itself
};

// Any other nu (Bessel functions), at distance d.
__device__ __noinline__ double lag_general(const CovDev& p, double d, bool drange) {
    const double r = d * p.inv_range;
    if (!drange) return p.sigma2 * kry_matern(r, p.nu);
    return r <= 0.0 ? 0.0 : p.sigma2 * kry_matern_dr(r, p.nu) * (-r * p.inv_range);
}

// sigma^2 rho_nu at lag (l1, l2) grid steps (drange: its derivative with respect
// to the range; with r = d / range, dr / d(range) = -r / range).
__device__ __forceinline__ double lag_entry(const CovDev& p, double l1, double l2, bool drange) {
    const double h1 = l1 * p.dx1, h2 = l2 * p.dx2;
    const double u = p.ca * h1 + p.sa * h2, v = p.ratio * (p.ca * h2 - p.sa * h1);
    const double d = sqrt(u * u + v * v);
    if (p.kind == 3) return lag_general(p, d, drange);
    const double x = d * p.s, e = exp(-x);
    double f;
    if (!drange) f = p.kind == 0 ? 1.0 : p.kind == 1 ? 1.0 + x : 1.0 + x + x * x * (1.0 / 3.0);
    else f = p.inv_range * (p.kind == 0 ? x : p.kind == 1 ? x * x : x * x * (1.0 + x) * (1.0 / 3.0));
    return p.sigma2 * f * e;
}

// Entry (j1, j2) of the first row of the block-circulant extension on the M1 x
// M2 torus.
__device__ __noinline__ double torus_entry(const CovDev& p, int j1, int j2, int M1, int M2, bool drange) {
    const int a1 = (2 * j1 <= M1) ? j1 : j1 - M1, a2 = (2 * j2 <= M2) ? j2 : j2 - M2;
    double v = lag_entry(p, a1, a2, drange);
    if (!p.even && (2 * j1 == M1 || 2 * j2 == M2)) {   // a lag of half the torus averages its images
        const int b1 = (2 * j1 < M1) ? j1 : j1 - M1, b2 = (2 * j2 < M2) ? j2 : j2 - M2;
        if (a1 == b1) v = 0.5 * (v + lag_entry(p, a1, b2, drange));
        else if (a2 == b2) v = 0.5 * (v + lag_entry(p, b1, a2, drange));
        else v = 0.25 * (v + lag_entry(p, a1, b2, drange) + lag_entry(p, b1, a2, drange) + lag_entry(p, b1, b2, drange));
    }
    return v;
}

// ------------------------------------------------------------------ FP64 2-D FFTs
//
// The torus covariance c is real and c[-j] = c[j], so Lambda = FFT2(c) is real
// and even, and a quarter of the transforms of a full complex FFT2 gives it:
//   rows   R[j1][k] for j1 = 0 .. M1/2 only (R[-j1][k] is its conjugate), two
//          real rows as one complex transform, k = 0 .. M2/2 kept;
//   columns two columns k, k + 1 as one complex transform (each has a real
//          result, its input being Hermitian), k = 0 .. M2/2 only (Lambda[-k1][-k2]
//          = Lambda[k1][k2]).
// Everything is FP64-pipe bound (fft64.cuh), so that is also what it gains:
// eigenvalues on the 2048^2 torus 270 us (1,045 us before).
// A sample, Re FFT2(a xi), is FFT2 of the Hermitian part of a xi: rows k1 = 0 ..
// M1/2, then the same column transforms (252 us; 527 before).

// Row transforms of the lag covariance: transform pr takes rows 2 pr and 2 pr + 1,
// evaluated on the spot (even covariances: half of a row, the rest mirrored).
// z[j1][k], j1 <= M1/2, k <= M2/2, leading dimension M2/2 + 1.
template <int B, int E, int NT>
__global__ void __launch_bounds__(NT * ((1 << B) / E), kf64::minb(NT * ((1 << B) / E), E))
    ke_rows(CovDev p, bool drange, double2* __restrict__ z, int M1, const double2* __restrict__ tw) {
    using P = kf64::Plan<B, E>;
    constexpr int L = P::L, LT = P::LT, PS = P::PS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    double2* sb = reinterpret_cast<double2*>(smem_raw) + n;
    const int ja = min(2 * ((int)blockIdx.x * NT + n), M1 / 2);
    const bool live = 2 * ((int)blockIdx.x * NT + n) <= M1 / 2, two = ja + 1 <= M1 / 2;
    double2 v[E];
    if (p.even) {
#pragma unroll 1
        for (int j = t; j <= L / 2; j += LT)
            sb[kf64::soff<PS, NT>(j)] = make_double2(torus_entry(p, ja, j, M1, L, drange),
                                                    two ? torus_entry(p, ja + 1, j, M1, L, drange) : 0.0);
        __syncthreads();
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int j = t + m * LT;
            v[m] = sb[kf64::soff<PS, NT>(min(j, L - j))];
        }
        __syncthreads();
    } else {
#pragma unroll 1
        for (int j = t; j < L; j += LT)
            sb[kf64::soff<PS, NT>(j)] = make_double2(torus_entry(p, ja, j, M1, L, drange),
                                                    two ? torus_entry(p, ja + 1, j, M1, L, drange) : 0.0);
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = sb[kf64::soff<PS, NT>(t + m * LT)];   // the thread's own
        __syncthreads();
    }
    kf64::transform<P, NT, false, false, false>(sb, v, t, tw);
    __syncthreads();
#pragma unroll
    for (int s = 0; s < E; ++s) sb[kf64::soff<PS, NT>(t + s * LT)] = v[kf64::brev(s, P::LE)];
    __syncthreads();
    if (!live) return;
    double2* za = z + (int64_t)ja * (L / 2 + 1);
    double2* zb = za + (L / 2 + 1);
    for (int k = t; k <= L / 2; k += LT) {
        const double2 a = sb[kf64::soff<PS, NT>(k)], b = sb[kf64::soff<PS, NT>((L - k) & (L - 1))];
        za[k] = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
        if (two) zb[k] = make_double2(0.5 * (a.y + b.y), 0.5 * (b.x - a.x));
    }
}

// Row transforms of a sample: row k1 of the Hermitian part of sqrt(max(lam, 0)
// scale) (xi_re + i xi_im).  z[k1][j], k1 <= M1/2, j < ldz.
template <int B, int E, int NT>
__global__ void __launch_bounds__(NT * ((1 << B) / E), kf64::minb(NT * ((1 << B) / E), E))
    ke_rows_noise(const double* __restrict__ lam, const double* __restrict__ xi, double scale,
                  double2* __restrict__ z, int M1, int ldz, const double2* __restrict__ tw) {
    using P = kf64::Plan<B, E>;
    constexpr int L = P::L, LT = P::LT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int row = (int)blockIdx.x * NT + n;
    const bool live = row <= M1 / 2;
    const int ra = min(row, M1 / 2), rb = (M1 - ra) & (M1 - 1);
    const double *re_a = xi + (int64_t)ra * L, *re_b = xi + (int64_t)rb * L;
    const double *im_a = re_a + (int64_t)M1 * L, *im_b = re_b + (int64_t)M1 * L;
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = t + m * LT, kb = (L - k) & (L - 1);
        const double a = 0.5 * sqrt(fmax(lam[(int64_t)ra * L + k], 0.0) * scale);
        v[m] = make_double2(a * (re_a[k] + re_b[kb]), a * (im_a[k] - im_b[kb]));
    }
    kf64::transform<P, NT, false, false, false>(reinterpret_cast<double2*>(smem_raw) + n, v, t, tw);
    if (!live) return;
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int j = t + s * LT;
        if (j < ldz) z[(int64_t)row * ldz + j] = v[kf64::brev(s, P::LE)];
    }
}

// Order-preserving map of doubles to integers (min and max without the FP64
// pipe) and back.
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double order_value(long long k) {
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}

// Column transforms of Hermitian columns 2q and 2q + 1 of z (rows 0 .. M1/2
// given, leading dimension ldz; columns >= ncol are zero) as one complex
// transform.  OUT 0: lam[k1][j] for every column of the M1 x M2 torus (columns
// past M2/2 by symmetry) and the block's smallest and largest value as order
// keys in part; OUT 1: out[i][j], i < n1, j < n2.
template <int B, int E, int NT, int OUT>
__global__ void __launch_bounds__(NT * ((1 << B) / E), kf64::minb(NT * ((1 << B) / E), E))
    ke_cols(const double2* __restrict__ z, int ldz, int ncol, double* __restrict__ out, int M2, int n1, int n2,
            const double2* __restrict__ tw, long long* __restrict__ part) {
    using P = kf64::Plan<B, E>;
    constexpr int L = P::L, LT = P::LT, TH = NT * LT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ long long red[2][TH / 32];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int j0 = 2 * ((int)blockIdx.x * NT + n);
    const bool one = j0 < ncol, two = j0 + 1 < ncol;
    const double2* za = z + (one ? j0 : 0);
    const double2* zb = z + (two ? j0 + 1 : 0);
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int j = t + m * LT;
        const int64_t r = (int64_t)min(j, L - j) * ldz;
        const double2 a = za[r], b = zb[r];
        const double sg = 2 * j > L ? -1.0 : 1.0;   // rows past the middle: conjugates
        v[m] = make_double2(two ? a.x - sg * b.y : a.x, two ? sg * a.y + b.x : sg * a.y);
    }
    kf64::transform<P, NT, false, false, false>(reinterpret_cast<double2*>(smem_raw) + n, v, t, tw);
    if constexpr (OUT == 1) {
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const int i = t + s * LT;
            const double2 f = v[kf64::brev(s, P::LE)];
            if (i < n1 && j0 < n2) out[(int64_t)i * n2 + j0] = f.x;
            if (i < n1 && j0 + 1 < n2) out[(int64_t)i * n2 + j0 + 1] = f.y;
        }
    } else {
        long long lo = 0x7fffffffffffffffll, hi = -0x7fffffffffffffffll - 1;
#pragma unroll
        for (int s = 0; s < E; ++s) {
            const int k1 = t + s * LT;
            const double2 f = v[kf64::brev(s, P::LE)];
            double* o = out + (int64_t)k1 * M2;
            double* om = out + (int64_t)((L - k1) & (L - 1)) * M2;
            if (one) {
                o[j0] = f.x;
                if (j0 > 0 && 2 * j0 < M2) om[M2 - j0] = f.x;
                const long long k = order_key(f.x);
                if (f.x == f.x) {
                    lo = min(lo, k);
                    hi = max(hi, k);
                }
            }
            if (two) {
                o[j0 + 1] = f.y;
                if (2 * (j0 + 1) < M2) om[M2 - j0 - 1] = f.y;
                const long long k = order_key(f.y);
                if (f.y == f.y) {
                    lo = min(lo, k);
                    hi = max(hi, k);
                }
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if ((threadIdx.x & 31) == 0) {
            red[0][threadIdx.x >> 5] = lo;
            red[1][threadIdx.x >> 5] = hi;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int w = 1; w < TH / 32; ++w) {
                lo = min(lo, red[0][w]);
                hi = max(hi, red[1][w]);
            }
            part[2 * blockIdx.x] = lo;
            part[2 * blockIdx.x + 1] = hi;
        }
    }
}

// Smallest and largest value over the column blocks (one block).
__global__ void k_minmax_final(const long long* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ long long slo[8], shi[8];
    long long lo = 0x7fffffffffffffffll, hi = -0x7fffffffffffffffll - 1;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        lo = min(lo, part[2 * b]);
        hi = max(hi, part[2 * b + 1]);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        slo[threadIdx.x >> 5] = lo;
        shi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        lo = min(lo, slo[w]);
        hi = max(hi, shi[w]);
    }
    out[0] = order_value(lo);
    out[1] = order_value(hi);
}

namespace {

struct RunRows {
    CovDev p;
    bool drange;
    double2* z;
    int M1;
    const double2* tw;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = kf64::Plan<B, E>;
        auto k = ke_rows<B, E, NT>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<(M1 / 4 + NT) / NT, NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(p, drange, z, M1, tw);
        KRY_CHECK_LAUNCH();
    }
};
struct RunNoise {
    const double *lam, *xi;
    double scale;
    double2* z;
    int M1, ldz;
    const double2* tw;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = kf64::Plan<B, E>;
        auto k = ke_rows_noise<B, E, NT>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<(M1 / 2 + NT) / NT, NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(lam, xi, scale, z, M1, ldz, tw);
        KRY_CHECK_LAUNCH();
    }
};
template <int OUT>
struct RunCols {
    const double2* z;
    int ldz, ncol;
    double* out;
    int M2, n1, n2;
    const double2* tw;
    DevBuf* red;   // order keys of every block, then the two results
    int* nblocks;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = kf64::Plan<B, E>;
        const int nb = ((ncol + 1) / 2 + NT - 1) / NT;
        if (OUT == 0) red->ensure((size_t)(2 * nb + 2) * sizeof(long long));
        *nblocks = nb;
        auto k = ke_cols<B, E, NT, OUT>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<nb, NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(z, ldz, ncol, out, M2, n1, n2, tw,
                                                             OUT == 0 ? red->as<long long>() : nullptr);
        KRY_CHECK_LAUNCH();
    }
};

}  // namespace

static CovDev cov_dev(const kry_cov& cov, double dx1, double dx2) {
    CovDev p;
    p.sigma2 = cov.sigma2;
    p.inv_range = 1.0 / cov.range;
    p.nu = cov.nu;
    p.s = sqrt(2.0 * cov.nu) / cov.range;
    p.ca = cos(cov.aniso_angle);
    p.sa = sin(cov.aniso_angle);
    p.ratio = cov.aniso_ratio;
    if (p.ratio == 1.0) {   // isotropic: the angle does not matter
        p.ca = 1.0;
        p.sa = 0.0;
    }
    p.dx1 = dx1;
    p.dx2 = dx2;
    p.kind = cov.nu == 0.5 ? 0 : cov.nu == 1.5 ? 1 : cov.nu == 2.5 ? 2 : 3;
    p.even = p.ca == 0.0 || p.sa == 0.0;
    return p;
}

// Eigenvalues (drange: of the range derivative) on the M1 x M2 torus, natural
// order, into out; the blocks' order keys are left in ctx->red.  Returns their
// number.
static int torus_eigs(kry_ctx* ctx, bool drange, const kry_cov& cov, double dx1, double dx2, int M1, int M2, double* out) {
    const int ldz = M2 / 2 + 1;
    ctx->eig_z.ensure((size_t)(M1 / 2 + 1) * ldz * sizeof(double2));
    double2* z = ctx->eig_z.as<double2>();
    const double2* tw = ctx->tab64.as<double2>();
    int nb = 0;
    kf64::dispatch<false>(M2, kf64::shape(M2), RunRows{cov_dev(cov, dx1, dx2), drange, z, M1, tw, ctx->stream});
    kf64::dispatch<false>(M1, kf64::shape(M1),
                   RunCols<0>{z, ldz, ldz, out, M2, 0, 0, tw, &ctx->red, &nb, ctx->stream});
    return nb;
}

void compute_eigs(kry_ctx* ctx, const kry_cov& cov, int n1, int n2, double dx1, double dx2, int M1, int M2,
                  double* lam_min, double* lam_max) {
    (void)n1;
    (void)n2;
    ctx->eig_c.ensure((size_t)M1 * M2 * sizeof(double));
    const int nb = torus_eigs(ctx, false, cov, dx1, dx2, M1, M2, ctx->eig_c.as<double>());
    double* res = ctx->red.as<double>() + 2 * nb;
    k_minmax_final<<<1, 256, 0, ctx->stream>>>(ctx->red.as<long long>(), nb, res);
    KRY_CHECK_LAUNCH();
    KRY_CUDA(cudaMemcpyAsync(ctx->host_pinned, res, 2 * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    KRY_CUDA(cudaStreamSynchronize(ctx->stream));
    *lam_min = ctx->host_pinned[0];
    *lam_max = ctx->host_pinned[1];
}

// Eigenvalues of (S + tau2 I)^-1 from those of the embedding S (in
// ctx->eig_c): 1 / (max(Lambda, 0) + tau2).  Negative embedding eigenvalues
// are reset to zero first (Sec. 3.6 caveat) so that the inverse stays
// positive definite.
__global__ void k_invert_eigs(double* __restrict__ c, int64_t MM, double tau2) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < MM; i += (int64_t)gridDim.x * blockDim.x)
        c[i] = 1.0 / (fmax(c[i], 0.0) + tau2);
}

void invert_eigs(kry_ctx* ctx, int M1, int M2, double tau2) {
    const int64_t MM = (int64_t)M1 * M2;
    k_invert_eigs<<<(unsigned)std::min<int64_t>((MM + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        ctx->eig_c.as<double>(), MM, tau2);
    KRY_CHECK_LAUNCH();
}

// ------------------------------------------------------------------ BCCB log-determinant
//
// Sec. 3.3's approximation log det Sigma ~ sum log D1 and its range
// derivative dL ~ sum D2 / D1 (Appendix A, Eq. circ_diag and Eq.
// trace_approx), D1 and D2 the eigenvalues of the block-circulant extensions
// of Sigma and d Sigma / d(range).  Reading: the matvec's power-of-two
// M1 x M2 torus, all frequencies, scaled by n1 n2 / (M1 M2) (the paper's
// (2n - 1)-point extension is not a power of two).  Eigenvalues below
// eps * max D1 are reset to that value (Sec. 3.6) and add no derivative term.

// Per-block sums of log(max(D1, floor)) and, where D1 > floor, D2 / D1.
__global__ void k_bccb_partials(const double* __restrict__ d1, const double* __restrict__ d2, int64_t n,
                                double floor_v, double* __restrict__ part) {
    double a = 0.0, b = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double l = d1[i];
        const bool keep = l > floor_v;
        a += log(keep ? l : floor_v);
        if (keep && d2) b += d2[i] / l;
    }
    __shared__ double sa[256], sb[256];
    sa[threadIdx.x] = a;
    sb[threadIdx.x] = b;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            sa[threadIdx.x] += sa[threadIdx.x + o];
            sb[threadIdx.x] += sb[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = sa[0];
        part[2 * blockIdx.x + 1] = sb[0];
    }
}

__global__ void k_bccb_final(const double* __restrict__ part, int nb, double* __restrict__ out) {
    double a = 0.0, b = 0.0;
    for (int i = 0; i < nb; ++i) {
        a += part[2 * i];
        b += part[2 * i + 1];
    }
    out[0] = a;
    out[1] = b;
}

void bccb_logdet(kry_ctx* ctx, const kry_cov& cov, bool deriv, double* logdet, double* dlogdet) {
    const int n1 = ctx->n1, n2 = ctx->n2;
    int M1 = 1, M2 = 1;
    while (M1 < 2 * n1) M1 <<= 1;
    while (M2 < 2 * n2) M2 <<= 1;
    const int64_t MM = (int64_t)M1 * M2;
    double lo, hi;
    compute_eigs(ctx, cov, n1, n2, ctx->dx1, ctx->dx2, M1, M2, &lo, &hi);   // D1 in eig_c
    double* d1 = ctx->eig_c.as<double>();
    double* d2 = nullptr;
    if (deriv) {
        ctx->eig_d.ensure(MM * sizeof(double));
        d2 = ctx->eig_d.as<double>();
        torus_eigs(ctx, true, cov, ctx->dx1, ctx->dx2, M1, M2, d2);
    }
    const int nb = 256;
    ctx->red.ensure((2 * nb + 2) * sizeof(double));
    double* part = ctx->red.as<double>();
    k_bccb_partials<<<nb, 256, 0, ctx->stream>>>(d1, d2, MM, 2.220446049250313e-16 * hi, part);
    KRY_CHECK_LAUNCH();
    k_bccb_final<<<1, 1, 0, ctx->stream>>>(part, nb, part + 2 * nb);
    KRY_CHECK_LAUNCH();
    KRY_CUDA(cudaMemcpyAsync(ctx->host_pinned, part + 2 * nb, 2 * sizeof(double), cudaMemcpyDeviceToHost,
                             ctx->stream));
    KRY_CUDA(cudaStreamSynchronize(ctx->stream));
    const double scale = (double)n1 * (double)n2 / (double)MM;
    *logdet = scale * ctx->host_pinned[0];
    if (dlogdet) *dlogdet = scale * ctx->host_pinned[1];
}

// lamT[j][k] = lam[k][j] * scale (FP64 and optionally FP32), 32 x 32 tiles.
// With t32p != NULL also the column-permuted FP32 copy (kspec::lam_slot), scaled by 1 / FWD_SCALE more.
__global__ void k_transpose_scale(const double* __restrict__ lam, int M1, int M2, double scale,
                                  double* __restrict__ t64, float* __restrict__ t32, float* __restrict__ t32p,
                                  int lt) {
    __shared__ double tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int k = by + r, j = bx + threadIdx.x;
        if (k < M1 && j < M2) tile[r][threadIdx.x] = lam[(int64_t)k * M2 + j];
    }
    __syncthreads();
    for (int r = threadIdx.y; r < 32; r += blockDim.y) {
        const int j = bx + r, k = by + threadIdx.x;
        if (k < M1 && j < M2) {
            const double v = tile[threadIdx.x][r] * scale;
            t64[(int64_t)j * M1 + k] = v;
            if (t32) t32[(int64_t)j * M1 + k] = (float)v;
            if (t32p) t32p[(int64_t)j * M1 + kspec::lam_slot(k, M1, lt)] = (float)(v * (1.0 / kspec::FWD_SCALE));
        }
    }
}

// Store the eigenvalues in ctx->eig_c as setting `slot` of embedding e.
void store_embedding(kry_ctx* ctx, kry_embed* e, int slot) {
    dim3 grid((e->M2 + 31) / 32, (e->M1 + 31) / 32), blk(32, 8);
    const int64_t off = (int64_t)slot * e->M1 * e->M2;
    k_transpose_scale<<<grid, blk, 0, ctx->stream>>>(ctx->eig_c.as<double>(), e->M1, e->M2,
                                                     1.0 / ((double)e->M1 * (double)e->M2), e->lam64T + off,
                                                     e->lam32T ? e->lam32T + off : nullptr,
                                                     e->lam32P ? e->lam32P + off : nullptr,
                                                     e->lam32P ? kspec::transform_threads(e->M1) : 0);
    KRY_CHECK_LAUNCH();
}

// Replace the eigenvalues of FP64 embedding e (one setting, e's grid) by those
// of the circulant extension of d Sigma / d(range) for cov, so that matvecs
// with e apply the range derivative of the covariance (Appendix A, dSigma).
void drange_embedding(kry_ctx* ctx, const kry_cov& cov, kry_embed* e) {
    const int M1 = e->M1, M2 = e->M2;
    ctx->eig_c.ensure((size_t)M1 * M2 * sizeof(double));
    torus_eigs(ctx, true, cov, ctx->dx1, ctx->dx2, M1, M2, ctx->eig_c.as<double>());
    store_embedding(ctx, e, 0);
}


void sample_field(kry_ctx* ctx, const kry_cov& cov, int M1, int M2, const double* xi, double* out) {
    double lo, hi;
    compute_eigs(ctx, cov, ctx->n1, ctx->n2, ctx->dx1, ctx->dx2, M1, M2, &lo, &hi);
    const int n1 = ctx->n1, n2 = ctx->n2;
    double2* z = ctx->eig_z.as<double2>();   // (M1/2 + 1) x n2 of it, n2 <= M2/2
    const double2* tw = ctx->tab64.as<double2>();
    int nb = 0;
    kf64::dispatch<false>(M2, kf64::shape(M2),
                   RunNoise{ctx->eig_c.as<double>(), xi, 1.0 / ((double)M1 * (double)M2), z, M1, n2, tw, ctx->stream});
    kf64::dispatch<false>(M1, kf64::shape(M1), RunCols<1>{z, n2, n2, out, M2, n1, n2, tw, nullptr, &nb, ctx->stream});
}

}  // namespace kry
