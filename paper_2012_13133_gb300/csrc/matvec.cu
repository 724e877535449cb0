// BTTB covariance matvec by circulant embedding (Sec. 3: Sigma is symmetric
// BTTB, stored through one row and applied in O(n log n) with FFTs; the
// embedding's eigenvalues diagonalise it, Appendix A Eq. circ_diag):
//
//   K v = A F^-1 ( Lambda .* F ( A^T v ) ) + tau^2 v
//
// on the M1 x M2 torus, A the observation mask.  Two real vectors travel as
// the real and imaginary parts of one complex field; that is exact because
// Lambda is real and even.  The 2-D transform is split into three kernels:
//
//   pass A  grid rows i < n1: the observed values of a row, zeros elsewhere,
//           forward FFT of length M2 into the intermediate slab (n1 x M2
//           complex per pair);
//   pass B  columns: the n1 nonzero rows of a column, forward FFT of length
//           M1, times Lambda (scaled by 1/(M1 M2)), inverse FFT, the first n1
//           rows back in place;
//   pass C  grid rows: inverse FFT of length M2, the observed columns, plus
//           the nugget term, and (optionally) the partials of the dot product
//           of input and output for the Krylov loops.
//
// The slab is laid out in column tiles, slab[pair][tile][i][c], whose width each
// kind of pass chooses so that the column pass reads and writes whole sectors.
#include <algorithm>
#include <mutex>
#include <string>

#include "dfloat.cuh"
#include "fft.cuh"
#include "mvspec.cuh"
#include "kry_internal.cuh"
#include "mv64.cuh"

namespace kry {

// The specialised FP32 passes (mvspec.cuh) cover torus sides from 64, the FP64
// ones (mv64.cu) every side; the three kernels below run FP32 on tori with a
// shorter side, radix 8 in shared memory (fft.cuh), 8 values per thread.

// ------------------------------------------------------------------ pass A

// One row: the observed values into a zero row in shared memory, forward FFT.
__global__ void __launch_bounds__(1024) k_pass_a(const float* __restrict__ vin, int64_t ld,
                                                 const double* __restrict__ scale, int nvec, int pair0,
                                                 const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                                 int n1, int M2, int C, float2* __restrict__ slab,
                                                 const float2* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    const int L = M2, LT = L / 8, tl = threadIdx.x, row = blockIdx.x;
    const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
    const bool has_b = vb < nvec;

    for (int k = tl; k < L; k += LT) buf[k] = make_float2(0.f, 0.f);
    __syncthreads();
    const float sa = scale ? (float)scale[va] : 1.f;
    const float sb = (scale && has_b) ? (float)scale[vb] : 1.f;
    const float* pa = vin + (int64_t)va * ld;
    const float* pb = vin + (int64_t)vb * ld;
    const int q1 = rowptr[row + 1];
    for (int q = rowptr[row] + tl; q < q1; q += LT) buf[colidx[q]] = make_float2(pa[q] * sa, has_b ? pb[q] * sb : 0.f);
    __syncthreads();
    fft_smem<false>(buf, L, tl, tw);

    // store: slab[pair][tile][row][c]
    float2* out = slab + (int64_t)blockIdx.y * n1 * M2;
    for (int e = tl; e < L; e += LT) {
        const int tile = e / C;
        out[((int64_t)tile * n1 + row) * C + (e - tile * C)] = buf[e];
    }
}

// ------------------------------------------------------------------ pass B

// CC columns, the slab's tile width.
template <int CC>
__global__ void __launch_bounds__(1024) k_pass_b(float2* __restrict__ slab, const float* __restrict__ lamT, int n1,
                                                 int M1, int M2, const float2* __restrict__ tw, int pair0,
                                                 int64_t lam_stride, int vpt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    const int L = M1;
    const int stride = L + 1;
    const int LT = L / 8;
    const int g = threadIdx.x / LT;
    const int tl = threadIdx.x - g * LT;
    const int tile = blockIdx.x;
    float2* blk = slab + (int64_t)blockIdx.y * n1 * M2 + (int64_t)tile * n1 * CC;

    const int nload = n1 * CC;
    for (int e = threadIdx.x; e < nload; e += blockDim.x) {
        const int i = e / CC;
        const int c = e - i * CC;
        buf[c * stride + i] = blk[e];
    }
    for (int e = threadIdx.x; e < (L - n1) * CC; e += blockDim.x) {
        const int c = e / (L - n1);
        const int i = n1 + (e - c * (L - n1));
        buf[c * stride + i] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    float2* cb = buf + g * stride;
    fft_smem<false>(cb, L, tl, tw);
    const int theta = vpt ? (2 * (pair0 + (int)blockIdx.y)) / vpt : 0;
    const float* lam = lamT + theta * lam_stride + (int64_t)(tile * CC + g) * L;
    for (int k = tl; k < L; k += LT) {
        const float l = lam[k];
        float2 z = cb[k];
        cb[k] = make_float2(z.x * l, z.y * l);
    }
    __syncthreads();
    fft_smem<true>(cb, L, tl, tw);
    for (int e = threadIdx.x; e < nload; e += blockDim.x) {
        const int i = e / CC;
        const int c = e - i * CC;
        blk[e] = buf[c * stride + i];
    }
}

// ------------------------------------------------------------------ pass C

// One row: inverse FFT, the observed cells, tau2 * (scaled input), optional dot.
__global__ void __launch_bounds__(1024) k_pass_c(const float2* __restrict__ slab, const float* __restrict__ vin,
                                                 int64_t ld_in, const double* __restrict__ scale,
                                                 float* __restrict__ vout, int64_t ld_out, int nvec, int pair0,
                                                 const int* __restrict__ rowptr, const int* __restrict__ colidx,
                                                 int n1, int M2, int C, double tau2, double* __restrict__ dots,
                                                 int ndot_stride, const float2* __restrict__ tw,
                                                 const double* __restrict__ tau2v, int vpt) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    __shared__ double red[2][32];
    const int L = M2, LT = L / 8, tl = threadIdx.x, row = blockIdx.x;
    const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
    const bool has_b = vb < nvec;

    const float2* in = slab + (int64_t)blockIdx.y * n1 * M2;
    for (int e = tl; e < L; e += LT) {
        const int tile = e / C;
        buf[e] = in[((int64_t)tile * n1 + row) * C + (e - tile * C)];
    }
    __syncthreads();
    fft_smem<true>(buf, L, tl, tw);

    DotAcc<float> acc_a, acc_b;
    {
        const float sa = scale ? (float)scale[va] : 1.f;
        const float sb = (scale && has_b) ? (float)scale[vb] : 1.f;
        const float t2 = (float)(tau2v ? tau2v[vpt ? va / vpt : 0] : tau2);
        const float* pa = vin + (int64_t)va * ld_in;
        const float* pb = vin + (int64_t)vb * ld_in;
        float* oa = vout + (int64_t)va * ld_out;
        float* ob = vout + (int64_t)vb * ld_out;
        const int q1 = rowptr[row + 1];
        for (int q = rowptr[row] + tl; q < q1; q += LT) {
            const float2 z = buf[colidx[q]];
            const float xa = pa[q] * sa;
            const float ya = z.x + t2 * xa;
            oa[q] = ya;
            acc_a.add_prod(xa, ya);
            if (has_b) {
                const float xb = pb[q] * sb;
                const float yb = z.y + t2 * xb;
                ob[q] = yb;
                acc_b.add_prod(xb, yb);
            }
        }
    }
    if (dots != nullptr) {
        double da = acc_a.value(), db = acc_b.value();
        // block reduction of (da, db) in a fixed order; blocks narrower than a
        // warp (short rows) reduce serially through shared memory
        const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (blockDim.x >= 32) {
            for (int o = 16; o > 0; o >>= 1) {
                da += __shfl_down_sync(0xffffffffu, da, o);
                db += __shfl_down_sync(0xffffffffu, db, o);
            }
            if (lane == 0) {
                red[0][w] = da;
                red[1][w] = db;
            }
        } else {
            red[0][threadIdx.x] = da;
            red[1][threadIdx.x] = db;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double sa = 0.0, sb = 0.0;
            const int nw = (blockDim.x >= 32) ? (blockDim.x >> 5) : blockDim.x;
            for (int k = 0; k < nw; ++k) {
                sa += red[0][k];
                sb += red[1][k];
            }
            dots[(int64_t)va * ndot_stride + blockIdx.x] = sa;
            if (has_b) dots[(int64_t)vb * ndot_stride + blockIdx.x] = sb;
        }
    }
}

// ------------------------------------------------------------------ host side

static size_t cx_size(bool dbl) { return dbl ? sizeof(double2) : sizeof(float2); }

// Columns per block (= slab tile width) of the short FP32 column pass: four, fewer
// where their transforms exceed a block's threads.
static int short_cols(int M1) { return M1 <= 2048 ? 4 : M1 == 4096 ? 2 : 1; }

void prof_record(kry_ctx* ctx, cudaEvent_t ev) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    KRY_CUDA(cudaStreamIsCapturing(ctx->stream, &cs));
    if (cs == cudaStreamCaptureStatusActive)
        KRY_CUDA(cudaEventRecordWithFlags(ev, ctx->stream, cudaEventRecordExternal));
    else
        KRY_CUDA(cudaEventRecord(ev, ctx->stream));
}

// FP32 tori that the specialised passes cover.
static bool use_spec(int M1, int M2) { return M1 >= 64 && M2 >= 64 && M1 <= KRY_MAX_M && M2 <= KRY_MAX_M; }

static int ilog2(int x) { return 31 - __builtin_clz((unsigned)x); }

static int batch_bucket(int nvec) {
    int b = 1;
    while (b < nvec && b < 64) b <<= 1;
    return b;
}

uint64_t sched_key(int M1, int M2, bool dbl, int nvec) {
    return (uint64_t)M1 | ((uint64_t)M2 << 16) | ((uint64_t)(dbl ? 1 : 0) << 32) | ((uint64_t)batch_bucket(nvec) << 40);
}

const MvSched& sched_for(kry_ctx* ctx, int M1, int M2, bool dbl, int nvec) {
    auto it = ctx->tuned.find(sched_key(M1, M2, dbl, nvec));
    if (it != ctx->tuned.end()) return it->second;
    return ctx->sched;
}

// Rows per block (passes A and C) and columns per block (pass B) of the
// specialised FP32 passes.  Blocks of 128 threads (four and more per SM, so that
// one block's loads run behind another's butterflies), 256 for the longest
// columns: two of side 4096, or one of side 8192, which alone needs 256 threads
// and reads and writes 8 bytes of each of its tile rows of 32.  Down to
// two warps (one for columns) while the launch has fewer blocks than two per SM
// (128^2, 4 vectors: 11.0 us, with 128 threads 12).  The rows per block group pass
// C's dot partials, so they do not depend on the batch.
static void spec_shape(kry_ctx* ctx, const kry_embed* e, int nvec, int* G, int* C) {
    const int M1 = e->M1, M2 = e->M2, np = (nvec + 1) / 2;
    const MvSched& want = sched_for(ctx, M1, M2, false, nvec);
    const int ltr = kspec::transform_threads(M2), ltc = kspec::transform_threads(M1);
    auto fill = [&](int lt, int th, int least, int64_t transforms) {
        while (th > least && th > lt && transforms * lt / th < 2 * ctx->num_sms) th /= 2;
        return std::max(1, th / lt);
    };
    const int g = want.rows > 0 ? want.rows : fill(ltr, 128, 64, M1 / 2);
    const int c = want.cols > 0 ? want.cols : fill(ltc, M1 >= 4096 ? 256 : 128, 32, (int64_t)M2 * np);
    *G = kspec::block_threads(M2, g, 64) / ltr;
    *C = kspec::block_threads(M1, c, M2) / ltc;
}

// Row and column transforms of the FP64 passes.
static void shape64(kry_ctx* ctx, const kry_embed* e, int nvec, kf64::Shape* row, kf64::Shape* col) {
    const MvSched& want = sched_for(ctx, e->M1, e->M2, true, nvec);
    *row = kf64::shape(e->M2, want.rows);
    *col = kf64::shape(e->M1, want.cols);
}

// Complex pairs per batch: all, unless the schedule says otherwise.
static int batch_pairs(kry_ctx* ctx, const kry_embed* e, bool dbl, int nvec) {
    const int npairs = (nvec + 1) / 2;
    if (!dbl && !use_spec(e->M1, e->M2)) return npairs;
    const MvSched& want = sched_for(ctx, e->M1, e->M2, dbl, nvec);
    return want.pairs_per_batch > 0 ? std::min(want.pairs_per_batch, npairs) : npairs;
}

// The three passes for batches of ppb pairs through the given slab.
template <typename T>
static void run_passes(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale, T* vout,
                       int64_t ld_out, int nvec, double tau2, double* dots, int nds, int mode, void* slab, int ppb,
                       int vpt, const int* skip) {
    const int n1 = e->n1, n2 = e->n2, M1 = e->M1, M2 = e->M2, npairs = (nvec + 1) / 2;
    const double* tau2v = ctx->no_nugget ? nullptr : e->tau2_dev;
    cudaStream_t st = ctx->stream;
    if constexpr (sizeof(T) == 8) {
        kf64::Args a{};
        a.vin = vin; a.ld_in = ld_in; a.scale = scale; a.vout = vout; a.ld_out = ld_out;
        a.nvec = nvec; a.bits = ctx->cellbits.as<uint2>(); a.wpr = (n2 + 31) / 32;
        a.n1 = n1; a.n2 = n2; a.M1 = M1; a.M2 = M2;
        shape64(ctx, e, nvec, &a.row, &a.col);
        a.logC = ilog2(std::min(M2, std::max(2, a.col.NT)));   // tile rows of at least a 32-byte sector
        a.slab = static_cast<double2*>(slab); a.lamT = e->lam64T; a.lam_stride = e->lam_stride; a.vpt = vpt;
        a.tau2 = tau2; a.tau2v = tau2v; a.dots = dots; a.nds = nds;
        a.tw = ctx->tab64.as<double2>(); a.skip = skip; a.mode = mode;
        for (a.pair0 = 0; a.pair0 < npairs; a.pair0 += ppb) {
            a.np = std::min(ppb, npairs - a.pair0);
            kf64::launch(a, st);
        }
        return;
    } else {
        KRY_REQUIRE(mode == 0, KRY_EINVAL, "whole-grid output is FP64 only");
        if (use_spec(M1, M2)) {
            KRY_REQUIRE(e->lam32P != nullptr, KRY_EINVAL, "embedding lacks the permuted eigenvalues");
            kspec::SpecArgs a{};
            a.vin = vin; a.ld_in = ld_in; a.scale = scale; a.vout = vout; a.ld_out = ld_out;
            a.nvec = nvec; a.bits = ctx->cellbits.as<uint2>(); a.wpr = (n2 + 31) / 32;
            a.n1 = n1; a.M1 = M1; a.M2 = M2;
            spec_shape(ctx, e, nvec, &a.G, &a.C);
            a.logCs = ilog2(std::min(32, std::max(4, a.C)));   // tile rows of 1 to 8 32-byte sectors
            a.slab = static_cast<float2*>(slab); a.lamP = e->lam32P; a.lam_stride = e->lam_stride; a.vpt = vpt;
            a.tau2 = tau2; a.tau2v = tau2v; a.dots = dots; a.nds = nds;
            a.twf = ctx->spec_tab.as<float4>();
            a.twi = a.twf + kspec::TWF_WORDS;
            a.post = reinterpret_cast<const float2*>(a.twi + kspec::TWI_WORDS);
            a.tww = a.post + kspec::POST_WORDS;
            a.skip = skip;
            for (a.pair0 = 0; a.pair0 < npairs; a.pair0 += ppb) {
                a.np = std::min(ppb, npairs - a.pair0);
                KRY_REQUIRE(kspec::launch_a(a, st) && kspec::launch_b(a, st) && kspec::launch_c(a, st),
                            KRY_EUNSUPPORTED, "no specialised matvec pass for this shape");
            }
            return;
        }
        const int C = short_cols(M1);
        const int* rowptr = ctx->rowptr.as<int>();
        const int* colidx = ctx->colidx.as<int>();
        const float2* tw = ctx->tw32.as<float2>();
        float2* sl = static_cast<float2*>(slab);
        const size_t smA = (size_t)(M2 + 1) * sizeof(float2), smB = (size_t)C * (M1 + 1) * sizeof(float2);
        auto pass_b = C == 4 ? k_pass_b<4> : C == 2 ? k_pass_b<2> : k_pass_b<1>;
        KRY_ALLOW_MAX_SMEM(k_pass_a);
        KRY_ALLOW_MAX_SMEM(pass_b);
        KRY_ALLOW_MAX_SMEM(k_pass_c);
        for (int pair0 = 0; pair0 < npairs; pair0 += ppb) {
            const int np = std::min(ppb, npairs - pair0);
            const dim3 gA(n1, np), gB(M2 / C, np);
            k_pass_a<<<gA, M2 / 8, smA, st>>>(vin, ld_in, scale, nvec, pair0, rowptr, colidx, n1, M2, C, sl, tw);
            KRY_CHECK_LAUNCH();
            pass_b<<<gB, C * (M1 / 8), smB, st>>>(sl, e->lam32T, n1, M1, M2, tw, pair0, e->lam_stride, vpt);
            KRY_CHECK_LAUNCH();
            k_pass_c<<<gA, M2 / 8, smA, st>>>(sl, vin, ld_in, scale, vout, ld_out, nvec, pair0, rowptr, colidx, n1, M2,
                                              C, tau2, dots, nds, tw, tau2v, vpt);
            KRY_CHECK_LAUNCH();
        }
    }
}

template <typename T>
static void run_matvec(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale, T* vout,
                       int64_t ld_out, int nvec, double tau2, double* dots, int nds, int mode, int vpt = 0,
                       const int* skip = nullptr);

// Irregular sites (sites.cu): A^T by scatter onto the whole grid, sigma^2 Sigma
// on the whole grid by the FFT passes with whole-grid index lists and no
// nugget, then (mode 0) the gather A, nugget and dot partials; in mode 1 the
// whole-grid result is the output.
template <typename T>
static void run_matvec_sites(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale,
                             T* vout, int64_t ld_out, int nvec, double tau2, double* dots, int nds, int mode, int vpt,
                             const int* skip) {
    const int64_t N = (int64_t)e->n1 * e->n2;
    KRY_REQUIRE(ctx->rowptr_full.p && ctx->full_n1 == e->n1 && ctx->full_n2 == e->n2, KRY_EINVAL,
                "the site map's whole-grid index lists are missing");
    DevBuf& gb = sizeof(T) == 8 ? ctx->sites.grid64 : ctx->sites.grid32;
    gb.ensure((size_t)(mode == 0 ? 2 : 1) * nvec * N * sizeof(T));
    T* gin = gb.as<T>();
    T* gout = (mode == 0) ? gin + (size_t)nvec * N : vout;
    site_scatter<T>(ctx, vin, ld_in, scale, nvec, gin, skip);
    struct Scope {   // whole-grid lists in, the site map and the nugget out, for the FFT passes
        kry_ctx* c;
        int64_t p;
        explicit Scope(kry_ctx* x) : c(x), p(x->p) {
            std::swap(c->rowptr, c->rowptr_full);
            std::swap(c->colidx, c->colidx_full);
            std::swap(c->cellbits, c->cellbits_full);
            c->p = (int64_t)c->n1 * c->n2;
            c->sites.active = false;
            c->no_nugget = true;
        }
        ~Scope() {
            std::swap(c->rowptr, c->rowptr_full);
            std::swap(c->colidx, c->colidx_full);
            std::swap(c->cellbits, c->cellbits_full);
            c->p = p;
            c->sites.active = true;
            c->no_nugget = false;
        }
    } scope(ctx);
    run_matvec<T>(ctx, e, gin, N, nullptr, gout, mode == 0 ? N : ld_out, nvec, 0.0, nullptr, 0, 0, vpt, skip);
    if (mode == 0) {
        ctx->p = scope.p;   // the gather runs over the sites
        ctx->sites.active = true;
        site_gather<T>(ctx, gout, vin, ld_in, scale, vout, ld_out, nvec, tau2, e->tau2_dev, vpt, dots, nds, skip);
    }
}

template <typename T>
static void run_matvec(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale, T* vout,
                       int64_t ld_out, int nvec, double tau2, double* dots, int nds, int mode, int vpt,
                       const int* skip) {
    KRY_REQUIRE(vpt == 0 || (vpt % 2 == 0 && nvec % vpt == 0 && nvec / vpt <= e->ntheta), KRY_EINVAL,
                "vectors per theta must be even and divide the batch");
    if (ctx->sites.active) {
        run_matvec_sites<T>(ctx, e, vin, ld_in, scale, vout, ld_out, nvec, tau2, dots, nds, mode, vpt, skip);
        return;
    }
    const bool dbl = sizeof(T) == 8;
    const int ppb = batch_pairs(ctx, e, dbl, nvec);
    DevBuf& sb = dbl ? ctx->slab64 : ctx->slab32;
    sb.ensure((size_t)e->n1 * e->M2 * cx_size(dbl) * ppb);
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (ctx->prof_on) {
        KRY_CUDA(cudaEventCreate(&ev0));
        KRY_CUDA(cudaEventCreate(&ev1));
        prof_record(ctx, ev0);
    }
    run_passes<T>(ctx, e, vin, ld_in, scale, vout, ld_out, nvec, tau2, dots, nds, mode, sb.p, ppb, vpt, skip);
    if (ctx->prof_on) {
        prof_record(ctx, ev1);
        ctx->prof_ev.push_back(ev0);
        ctx->prof_ev.push_back(ev1);
        ctx->prof_nvec.push_back(nvec);
        ctx->prof_dbl.push_back(dbl ? 1 : 0);
    }
}

// Number of per-block dot partials pass C writes per vector for a batch of
// nvec vectors (the Krylov finalisers sum exactly this many).
int matvec_num_partials(kry_ctx* ctx, const kry_embed* e, bool dbl, int nvec) {
    if (ctx->sites.active) return site_num_partials(ctx);
    if (dbl) {
        kf64::Shape row, col;
        shape64(ctx, e, nvec, &row, &col);
        return (e->n1 + row.NT - 1) / row.NT;
    }
    if (use_spec(e->M1, e->M2)) {
        int G, C;
        spec_shape(ctx, e, nvec, &G, &C);
        return (e->n1 + G - 1) / G;
    }
    return e->n1;   // the short passes take a row per block
}

template <typename T>
void matvec_ex(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale, T* vout,
               int64_t ld_out, int nvec, double* dots, int nds, int vpt, const int* skip) {
    run_matvec<T>(ctx, e, vin, ld_in, scale, vout, ld_out, nvec, e->cov.tau2, dots, nds, 0, vpt, skip);
}

template void matvec_ex<float>(kry_ctx*, const kry_embed*, const float*, int64_t, const double*, float*, int64_t, int,
                               double*, int, int, const int*);
template void matvec_ex<double>(kry_ctx*, const kry_embed*, const double*, int64_t, const double*, double*, int64_t,
                                int, double*, int, int, const int*);

template <typename T>
void matvec(kry_ctx* ctx, const kry_embed* e, const T* vin, T* vout, int nvec, int64_t ld, double) {
    run_matvec<T>(ctx, e, vin, ld, nullptr, vout, ld, nvec, e->cov.tau2, nullptr, 0, 0);
}
template void matvec<float>(kry_ctx*, const kry_embed*, const float*, float*, int, int64_t, double);
template void matvec<double>(kry_ctx*, const kry_embed*, const double*, double*, int, int64_t, double);

void sigma_to_grid64(kry_ctx* ctx, const kry_embed* e, const double* vin, double* out_grid, int nvec, int64_t ld,
                     int vpt) {
    run_matvec<double>(ctx, e, vin, ld, nullptr, out_grid, (int64_t)e->n1 * e->n2, nvec, 0.0, nullptr, 0, 1, vpt);
}

// ------------------------------------------------------------------ allocation-free matvec
//
// kry_matvec_noalloc serves callers that cannot allocate device memory when
// they call: applications whose device memory is all owned by their own pool
// or arena (a framework's caching allocator that has reserved the GPU), and
// latency-critical loops that cannot absorb the device-wide synchronisation of
// cudaMalloc / cudaFree.  It runs the same FFT passes as kry_matvec, chosen by
// the same schedule, but its slab lives in a fixed file-scope device array
// instead of context scratch, taking as many complex pairs per batch as the
// array holds.  The array is part of the module, so every GPU that loads this
// library holds it until the process exits.
//
// Set-up: the first call on a device looks up the array's device address
// (cudaGetSymbolAddress, with that device current) and caches it with the
// identity of the device's current CUDA context; a later call under another
// context (after cudaDeviceReset, say) looks it up again.  Make that first call
// before any stream capture.  The context, its mask and the embedding must
// already exist (creating them does allocate).
//
// Sharing: every call on a device uses the same array and it keeps the last
// call's contents.  Nothing needs clearing, because pass A writes every slab
// element that passes B and C read.  Calls whose work overlaps on the GPU
// (other streams, other host threads) race on the array and must be
// serialised by the caller.

#define KRY_NOALLOC_SCRATCH_BYTES (16u << 20)   // 16 MiB: one 1024 x 1024 FP32 complex pair
#define KRY_NOALLOC_MAX_DEVICES 64

static __device__ __align__(256) unsigned char g_noalloc_scratch[KRY_NOALLOC_SCRATCH_BYTES];

struct NoallocSlot {
    void* addr = nullptr;
    unsigned long long ctx_id = 0;
};
static std::mutex g_noalloc_mu;
static NoallocSlot g_noalloc_slot[KRY_NOALLOC_MAX_DEVICES];

// Identity of the calling thread's current CUDA context (driver entry points
// cuCtxGetCurrent / cuCtxGetId, looked up through the runtime), 0 if unknown.
static unsigned long long current_ctx_id() {
    typedef int (*GetCurrentFn)(void**);
    typedef int (*GetIdFn)(void*, unsigned long long*);
    static GetCurrentFn get_current = nullptr;
    static GetIdFn get_id = nullptr;
    static bool looked_up = false;
    if (!looked_up) {   // under g_noalloc_mu
        looked_up = true;
        cudaDriverEntryPointQueryResult q1 = cudaDriverEntryPointSymbolNotFound, q2 = q1;
        void *f1 = nullptr, *f2 = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
            q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
            get_current = reinterpret_cast<GetCurrentFn>(f1);
            get_id = reinterpret_cast<GetIdFn>(f2);
        }
        cudaGetLastError();
    }
    if (!get_current || !get_id) return 0;
    void* c = nullptr;
    unsigned long long id = 0;
    if (get_current(&c) != 0 || c == nullptr || get_id(c, &id) != 0) return 0;
    return id;
}

// Device address of g_noalloc_scratch on the current device (looked up once
// per device and context).
static void* noalloc_scratch(int device) {
    KRY_REQUIRE(device >= 0 && device < KRY_NOALLOC_MAX_DEVICES, KRY_EUNSUPPORTED,
                "device index too large for the allocation-free matvec");
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    NoallocSlot& slot = g_noalloc_slot[device];
    const unsigned long long id = current_ctx_id();
    if (slot.addr == nullptr || slot.ctx_id != id) {
        void* ptr = nullptr;
        cudaError_t err = cudaGetSymbolAddress((void**)&ptr, g_noalloc_scratch);
        if (err != cudaSuccess)
            throw KryError{KRY_ECUDA, std::string("cudaGetSymbolAddress of the static matvec scratch failed: ") +
                                          cudaGetErrorString(err)};
        slot.addr = ptr;
        slot.ctx_id = id;
    }
    return slot.addr;
}

template <typename T>
static void run_matvec_noalloc(kry_ctx* ctx, const kry_embed* e, const T* vin, T* vout, int nvec, int64_t ld,
                               void* scratch) {
    const bool dbl = sizeof(T) == 8;
    const size_t slab_pair = (size_t)e->n1 * e->M2 * cx_size(dbl);
    KRY_REQUIRE(slab_pair <= KRY_NOALLOC_SCRATCH_BYTES, KRY_EUNSUPPORTED,
                "grid too large for the allocation-free matvec: n1 * M2 * sizeof(complex) = " +
                    std::to_string(slab_pair) + " bytes exceeds its 16 MiB static scratch");
    const int cap = std::max(1, (int)(KRY_NOALLOC_SCRATCH_BYTES / slab_pair));
    // the passes and schedule of kry_matvec, with at most `cap` pairs per batch
    run_passes<T>(ctx, e, vin, ld, nullptr, vout, ld, nvec, e->cov.tau2, nullptr, 0, 0, scratch,
                  std::min(batch_pairs(ctx, e, dbl, nvec), cap), 0, nullptr);
}

}  // namespace kry

extern "C" kry_status kry_matvec_noalloc(kry_ctx* ctx, const kry_embed* e, const void* v_dev, void* out_dev,
                                         int32_t nvec, int64_t ld) {
    if (!ctx) return KRY_EINVAL;
    try {
        KRY_CUDA(cudaSetDevice(ctx->device));
        ctx->err.clear();
        KRY_REQUIRE(e != nullptr && e->ctx == ctx, KRY_EINVAL, "embedding is NULL or belongs to another context");
        KRY_REQUIRE(ctx->p > 0 && e->n1 == ctx->n1 && e->n2 == ctx->n2, KRY_EINVAL,
                    "no mask set, or the embedding grid differs from the mask grid");
        KRY_REQUIRE(!ctx->sites.active, KRY_EUNSUPPORTED,
                    "the allocation-free matvec needs an observation mask (kry_set_mask), not sites");
        KRY_REQUIRE(nvec >= 0 && ld >= ctx->p, KRY_EINVAL, "need nvec >= 0 and ld >= p");
        if (nvec == 0) return KRY_OK;
        KRY_REQUIRE(v_dev && out_dev, KRY_EINVAL, "v_dev and out_dev must not be NULL");
        void* scratch = kry::noalloc_scratch(ctx->device);
        if (e->prec == KRY_F64)
            kry::run_matvec_noalloc<double>(ctx, e, static_cast<const double*>(v_dev), static_cast<double*>(out_dev),
                                            nvec, ld, scratch);
        else
            kry::run_matvec_noalloc<float>(ctx, e, static_cast<const float*>(v_dev), static_cast<float*>(out_dev),
                                           nvec, ld, scratch);
        return KRY_OK;
    } catch (const KryError& err) {
        ctx->err = err.msg;
        return err.st;
    } catch (const std::exception& err) {
        ctx->err = err.what();
        return KRY_ECUDA;
    }
}

// ------------------------------------------------------------------ schedule autotuner
//
// Times every feasible schedule (rows per block for the row passes,
// columns per block = slab tile width for the column pass, complex pairs per
// batch: all at once, or chunks whose slab stays within ~32 or ~64 MB of L2)
// on the caller's embedding and batch width, and caches the fastest for
// (M1, M2, precision, batch bucket).

namespace kry {

template <typename T>
__global__ void k_fill_test(T* __restrict__ x, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = (T)(((i * 2654435761ll) & 1023) - 511) * (T)(1.0 / 512.0);
}

template <typename T>
static double time_sched(kry_ctx* ctx, const kry_embed* e, const T* v, T* out, int nvec, int reps) {
    cudaEvent_t a, b;
    KRY_CUDA(cudaEventCreate(&a));
    KRY_CUDA(cudaEventCreate(&b));
    const bool prof = ctx->prof_on;
    ctx->prof_on = false;
    run_matvec<T>(ctx, e, v, ctx->p, nullptr, out, ctx->p, nvec, e->cov.tau2, nullptr, 0, 0);   // warm-up
    KRY_CUDA(cudaEventRecord(a, ctx->stream));
    for (int r = 0; r < reps; ++r)
        run_matvec<T>(ctx, e, v, ctx->p, nullptr, out, ctx->p, nvec, e->cov.tau2, nullptr, 0, 0);
    KRY_CUDA(cudaEventRecord(b, ctx->stream));
    KRY_CUDA(cudaEventSynchronize(b));
    float ms = 0.f;
    KRY_CUDA(cudaEventElapsedTime(&ms, a, b));
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    ctx->prof_on = prof;
    return ms / reps;
}

template <typename T>
static double autotune_t(kry_ctx* ctx, const kry_embed* e, int nvec, MvSched* best_out) {
    const bool dbl = sizeof(T) == 8;
    const int M1 = e->M1, M2 = e->M2;
    const uint64_t key = sched_key(M1, M2, dbl, nvec);
    const size_t n = (size_t)nvec * ctx->p;
    DevBuf tv, to;
    tv.stream = to.stream = ctx->stream;
    tv.ensure(n * sizeof(T));
    to.ensure(n * sizeof(T));
    k_fill_test<T><<<1024, 256, 0, ctx->stream>>>(tv.as<T>(), (int64_t)n);
    KRY_CHECK_LAUNCH();
    const int npairs = (nvec + 1) / 2;
    const size_t slab_pair = (size_t)e->n1 * M2 * cx_size(dbl);
    std::vector<int> ppbs = {0};
    for (size_t budget : {(size_t)32 << 20, (size_t)64 << 20}) {
        const int c = (int)std::max<size_t>(1, budget / slab_pair);
        if (c < npairs && std::find(ppbs.begin(), ppbs.end(), c) == ppbs.end()) ppbs.push_back(c);
    }
    double best = 1e30;
    MvSched bs = ctx->sched;
    const bool had = ctx->tuned.count(key) > 0;
    const MvSched prev = had ? ctx->tuned[key] : bs;
    if (dbl || use_spec(M1, M2)) {
        // blocks that are compiled as asked: others are rounded to one of these
        auto feasible = [&](int M, int nt, int most) {
            return dbl ? kf64::shape(M, nt).NT == nt
                       : kspec::block_threads(M, nt, most) == nt * kspec::transform_threads(M);
        };
        bool any = false;
        for (int g : {0, 1, 2, 4, 8, 16}) {
            if (g && !feasible(M2, g, 64)) continue;
            for (int c : {0, 1, 2, 4, 8, 16}) {
                if (c && !feasible(M1, c, M2)) continue;
                for (int ppb : ppbs) {
                    MvSched cand = bs;
                    cand.rows = g;
                    cand.cols = c;
                    cand.pairs_per_batch = ppb;
                    ctx->tuned[key] = cand;
                    const double ms = time_sched<T>(ctx, e, tv.as<T>(), to.as<T>(), nvec, 3);
                    if (!any || ms < best) {
                        any = true;
                        best = ms;
                        bs = cand;
                    }
                }
            }
        }
        // pin the blocks that run, and report them
        if (dbl) {
            kf64::Shape row, col;
            ctx->tuned[key] = bs;
            shape64(ctx, e, nvec, &row, &col);
            bs.rows = row.NT;
            bs.cols = col.NT;
        } else {
            ctx->tuned[key] = bs;
            spec_shape(ctx, e, nvec, &bs.rows, &bs.cols);
        }
        ctx->tuned[key] = bs;
        // the default blocks of the shortest tori hold more transforms than kry_set_schedule takes:
        // reported as 0, which names the same blocks
        for (int* b : {&bs.rows, &bs.cols})
            if (*b > 16) *b = 0;
    } else {
        if (had) ctx->tuned[key] = prev;
        best = time_sched<T>(ctx, e, tv.as<T>(), to.as<T>(), nvec, 3);
    }
    tv.release();
    to.release();
    if (best_out) *best_out = bs;
    return best;
}

double autotune(kry_ctx* ctx, const kry_embed* e, int nvec, MvSched* best) {
    return e->prec == KRY_F64 ? autotune_t<double>(ctx, e, nvec, best) : autotune_t<float>(ctx, e, nvec, best);
}

}  // namespace kry

extern "C" kry_status kry_autotune(kry_ctx* ctx, const kry_embed* e, int32_t nvec, double* best_ms,
                                   int32_t* rows_per_block, int32_t* cols_per_block, int32_t* pairs_per_batch) {
    if (!ctx) return KRY_EINVAL;
    try {
        KRY_CUDA(cudaSetDevice(ctx->device));
        ctx->err.clear();
        KRY_REQUIRE(e != nullptr && e->ctx == ctx, KRY_EINVAL, "embedding is NULL or belongs to another context");
        KRY_REQUIRE(ctx->p > 0 && e->n1 == ctx->n1 && e->n2 == ctx->n2, KRY_EINVAL,
                    "no mask set, or the embedding grid differs from the mask grid");
        KRY_REQUIRE(nvec >= 1, KRY_EINVAL, "nvec must be >= 1");
        MvSched b;
        const double ms = kry::autotune(ctx, e, nvec, &b);
        if (best_ms) *best_ms = ms;
        if (rows_per_block) *rows_per_block = b.rows;
        if (cols_per_block) *cols_per_block = b.cols;
        if (pairs_per_batch) *pairs_per_batch = b.pairs_per_batch;
        return KRY_OK;
    } catch (const KryError& err) {
        ctx->err = err.msg;
        return err.st;
    } catch (const std::exception& err) {
        ctx->err = err.what();
        return KRY_ECUDA;
    }
}

extern "C" kry_status kry_set_schedule(kry_ctx* ctx, const kry_embed* e, int32_t nvec, int32_t rows_per_block,
                                       int32_t cols_per_block, int32_t pairs_per_batch) {
    if (!ctx) return KRY_EINVAL;
    try {
        KRY_REQUIRE(e != nullptr && e->ctx == ctx, KRY_EINVAL, "embedding is NULL or belongs to another context");
        auto pow2 = [](int x) { return x >= 0 && (x & (x - 1)) == 0; };
        KRY_REQUIRE(nvec >= 1 && pow2(rows_per_block) && pow2(cols_per_block) && rows_per_block <= 16 &&
                        cols_per_block <= 16 && pairs_per_batch >= 0,
                    KRY_EINVAL, "rows/cols per block must be 0 (default) or a power of two <= 16; pairs >= 0");
        const bool dbl = e->prec == KRY_F64;
        MvSched s = ctx->sched;
        s.rows = rows_per_block;
        s.cols = cols_per_block;
        s.pairs_per_batch = pairs_per_batch;
        ctx->tuned[kry::sched_key(e->M1, e->M2, dbl, nvec)] = s;
        return KRY_OK;
    } catch (const KryError& err) {
        ctx->err = err.msg;
        return err.st;
    }
}
