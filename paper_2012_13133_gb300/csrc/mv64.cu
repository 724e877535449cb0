// The FP64 covariance matvec passes (Sec. 3; the three passes of matvec.cu's
// header) for every torus side 8 .. 8192: true residuals, FP64 embeddings, the
// kriging map.  Bound by the FP64 pipe (fft64.cuh): 4 vectors on 1024^2 move 0.2
// GB, 30 us of HBM time, and take 218 + 823 + 243 us (1,940 us before).
#include "fft64.cuh"
#include "mv64.cuh"
#include "mvspec.cuh"

namespace kf64 {

Shape shape(int L, int want_nt) {
    Shape s;
    s.E = L <= 512 ? 4 : 16;
    const int lt = L / s.E;
    if (s.E == 4) {
        s.NT = std::max(1, 32 / lt);
        return s;
    }
    s.NT = std::max(1, (want_nt * lt > 128 ? 256 : 128) / lt);
    if (lt == 512) s.NT = 1;
    return s;
}

// Double-double arithmetic (Dekker, Numer. Math. 1971) for the table: with T from a
// rounded sine a twiddle's imaginary part would carry two roundings (forward
// transforms of 256 points: 7% more error).
struct dd {
    double h, l;
};
__device__ dd dd_norm(double h, double l) {
    const double s = h + l;
    return {s, l - (s - h)};
}
__device__ dd dd_mul(dd a, dd b) {
    const double p = a.h * b.h;
    return dd_norm(p, fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
__device__ dd dd_add(dd a, dd b) {   // |a| >= |b|
    const dd s = dd_norm(a.h, b.h);
    return dd_norm(s.h, s.l + (a.l + b.l));
}
__device__ dd dd_inv(double n) { return {1.0 / n, fma(-n, 1.0 / n, 1.0) / n}; }

// sin and cos of pi z, 0 <= z <= 1/4: Taylor series, the terms past 2^-11 of the
// sum in double.
__device__ void sincospi_dd(double z, dd& s, dd& c) {
    const dd t = dd_mul({3.14159265358979311600, 1.22464679914735317723e-16}, {z, 0.0}), x = dd_mul(t, t);
    const double y = x.h;
    double q = 0.0, r = 0.0;   // sum_{n >= 3} (-y)^(n-3) / (2n + 1)! and / (2n)!
#pragma unroll
    for (int n = 10; n >= 3; --n) {
        double f = 1.0;
#pragma unroll
        for (int m = 2; m <= 2 * n; ++m) f *= m;
        q = fma(-y, q, 1.0 / (f * (2 * n + 1)));
        r = fma(-y, r, 1.0 / f);
    }
    const dd a = dd_mul(t, x), b = dd_mul(a, x), x2 = dd_mul(x, x);
    s = dd_add(dd_mul(a, dd_inv(-6.0)), dd_add(dd_mul(b, dd_inv(120.0)), {-q * t.h * y * y * y, 0.0}));
    s = dd_add(t, s);
    c = dd_add({-0.5 * x.h, -0.5 * x.l}, dd_add(dd_mul(x2, dd_inv(24.0)), {-r * y * y * y, 0.0}));
    c = dd_add({1.0, 0.0}, c);
}

__global__ void k_table(double2* __restrict__ tab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= TW_WORDS) return;
    const int ns = 1 << (31 - __clz(i / 8 + 2));   // sections of 8 ns words from 8 (ns - 2)
    const int r = i - 8 * (ns - 2), e = r / ns, k = r - e * ns;
    const int l = e == 0 ? 1 : 2 + (31 - __clz(e));
    const double turns2 = 2.0 * ((double)k / ns + (e - tw_base(l))) / (double)(1 << l);   // exact, below 1
    const bool neg = turns2 > 0.5;
    const double y = neg ? 1.0 - turns2 : turns2;
    const bool swap = y > 0.25;
    dd s, c;
    sincospi_dd(swap ? 0.5 - y : y, swap ? c : s, swap ? s : c);
    if (neg) c = {-c.h, -c.l};
    const double q = s.h / c.h;   // the tangent that goes with the rounded cosine
    tab[i] = make_double2(c.h, e == 0 ? s.h : q + (fma(-q, c.h, s.h) + s.l) / c.h);
}

void fill_table(double2* tab_dev, cudaStream_t st) {
    k_table<<<(TW_WORDS + 255) / 256, 256, 0, st>>>(tab_dev);
    KRY_CHECK_LAUNCH();
}

// Pass A: row transforms (columns >= n2 are zero: the upper half).
template <int B, int E, int NT>
__global__ void __launch_bounds__(NT * ((1 << B) / E), minb(NT * ((1 << B) / E), E))
    kd_pass_a(const double* __restrict__ vin, int64_t ld, const double* __restrict__ scale, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int logC, double2* __restrict__ slab,
              const double2* __restrict__ tw, const int* __restrict__ skip) {
    using P = Plan<B, E>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int row = blockIdx.x * NT + n;
    const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
    const bool has_b = vb < nvec, live = row < n1;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const double sa = scale ? scale[va] : 1.0, sbv = (scale && has_b) ? scale[vb] : 1.0;
    const double* pa = vin + (int64_t)va * ld;
    const double* pb = has_b ? vin + (int64_t)vb * ld : pa;
    int q[E / 2];
    kspec::cell_indices<P::LT, E / 2>(bits + (int64_t)min(row, n1 - 1) * wpr, wpr, live, t, q);
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E / 2; ++m) v[m] = make_double2(pa[max(q[m], 0)], pb[max(q[m], 0)]);
#pragma unroll
    for (int m = 0; m < E / 2; ++m)
        v[m] = make_double2(q[m] >= 0 ? v[m].x * sa : 0.0, q[m] >= 0 && has_b ? v[m].y * sbv : 0.0);
    transform<P, NT, false, true, false>(reinterpret_cast<double2*>(smem_raw) + n, v, t, tw);
    if (!live) return;
    double2* out = slab + (((int64_t)blockIdx.y * n1) << B);
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const int k = t + s * P::LT;
        out[(((int64_t)(k >> logC) * n1 + row) << logC) + (k & ((1 << logC) - 1))] = v[brev(s, P::LE)];
    }
}

// Pass B: column transforms, x Lambda in registers, inverse, rows < n1 kept.
template <int B, int E, int NT>
__global__ void __launch_bounds__(NT * ((1 << B) / E), minb(NT * ((1 << B) / E), E))
    kd_pass_b(double2* __restrict__ slab, const double* __restrict__ lamT, int n1, int M2, int logC,
              const double2* __restrict__ tw, int pair0, int64_t lam_stride, int vpt, const int* __restrict__ skip,
              int nvec) {
    using P = Plan<B, E>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
    if (skip && skip[va] && (vb >= nvec || skip[vb])) return;
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int col = min((int)blockIdx.x * NT + n, M2 - 1);
    const bool live = (int)blockIdx.x * NT + n < M2;   // (tori narrower than a block)
    double2* sb = reinterpret_cast<double2*>(smem_raw) + n;
    double2* blk = slab + (int64_t)blockIdx.y * n1 * M2 + (((int64_t)(col >> logC) * n1 + t) << logC) +
                   (col & ((1 << logC) - 1));
    double2 v[E], w[E];
#pragma unroll
    for (int m = 0; m < E / 2; ++m)
        v[m] = (t + m * P::LT < n1) ? blk[(int64_t)(m * P::LT) << logC] : make_double2(0.0, 0.0);
    transform<P, NT, false, true, false>(sb, v, t, tw);
    const int theta = vpt ? va / vpt : 0;
    const double* lam = lamT + theta * lam_stride + (int64_t)col * P::L + t;
#pragma unroll
    for (int s = 0; s < E; ++s) {
        const double l = __ldg(lam + s * P::LT);
        const double2 z = v[brev(s, P::LE)];
        w[s] = make_double2(z.x * l, z.y * l);
    }
    __syncthreads();   // every read of the forward transform's last stage is done
    transform<P, NT, true, false, true>(sb, w, t, tw);
#pragma unroll
    for (int s = 0; s < E / 2; ++s)
        if (live && t + s * P::LT < n1) blk[(int64_t)(s * P::LT) << logC] = w[brev(s, P::LE)];
}

// Pass C: inverse row transforms.  MODE 0: the observed cells, nugget and (dots
// != NULL) per-block partials of v . K v; MODE 1: every grid cell, no nugget.
template <int B, int E, int NT, int MODE>
__global__ void __launch_bounds__(NT * ((1 << B) / E), minb(NT * ((1 << B) / E), E))
    kd_pass_c(const double2* __restrict__ slab, const double* __restrict__ vin, int64_t ld_in,
              const double* __restrict__ scale, double* __restrict__ vout, int64_t ld_out, int nvec, int pair0,
              const uint2* __restrict__ bits, int wpr, int n1, int n2, int logC, double tau2,
              double* __restrict__ dots, int ndot_stride, const double2* __restrict__ tw,
              const double* __restrict__ tau2v, int vpt, const int* __restrict__ skip) {
    using P = Plan<B, E>;
    constexpr int TH = NT * P::LT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ double red[2][TH / 32];
    const int n = threadIdx.x & (NT - 1), t = threadIdx.x / NT;
    const int row = blockIdx.x * NT + n;
    const int va = 2 * (pair0 + (int)blockIdx.y), vb = va + 1;
    const bool has_b = vb < nvec, live = row < n1;
    if (skip && skip[va] && (!has_b || skip[vb])) return;   // both columns finished (whole block)
    const double2* in = slab + (((int64_t)blockIdx.y * n1) << B);
    double2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = t + m * P::LT;
        v[m] = in[(((int64_t)(k >> logC) * n1 + min(row, n1 - 1)) << logC) + (k & ((1 << logC) - 1))];
    }
    transform<P, NT, true, false, true>(reinterpret_cast<double2*>(smem_raw) + n, v, t, tw);
    if constexpr (MODE == 1) {
        double* oa = vout + (int64_t)va * ld_out + (int64_t)row * n2;
        double* ob = vout + (int64_t)vb * ld_out + (int64_t)row * n2;
#pragma unroll
        for (int s = 0; s < E / 2; ++s) {
            const int j = t + s * P::LT;
            const double2 z = v[brev(s, P::LE)];
            if (live && j < n2) oa[j] = z.x;
            if (live && j < n2 && has_b) ob[j] = z.y;
        }
        return;
    }
    const double sa = scale ? scale[va] : 1.0, sbv = (scale && has_b) ? scale[vb] : 1.0;
    const double t2 = tau2v ? tau2v[vpt ? va / vpt : 0] : tau2;
    const double* pa = vin + (int64_t)va * ld_in;
    const double* pb = has_b ? vin + (int64_t)vb * ld_in : pa;
    double* oa = vout + (int64_t)va * ld_out;
    double* ob = vout + (int64_t)vb * ld_out;
    int q[E / 2];
    kspec::cell_indices<P::LT, E / 2>(bits + (int64_t)min(row, n1 - 1) * wpr, wpr, live, t, q);
    double2 x[E / 2];
#pragma unroll
    for (int s = 0; s < E / 2; ++s) x[s] = make_double2(pa[max(q[s], 0)], pb[max(q[s], 0)]);
    double da = 0.0, db = 0.0;
#pragma unroll
    for (int s = 0; s < E / 2; ++s) {
        const double2 z = v[brev(s, P::LE)];
        x[s] = make_double2(x[s].x * sa, x[s].y * sbv);
        const double ya = fma(t2, x[s].x, z.x), yb = fma(t2, x[s].y, z.y);
        const bool on = q[s] >= 0;   // what lies in unobserved cells stays out of the sums
        if (on) oa[q[s]] = ya;
        if (on && has_b) ob[q[s]] = yb;
        if (dots && on) {
            da = fma(x[s].x, ya, da);
            db = fma(x[s].y, yb, db);
        }
    }
    if (dots != nullptr) {   // fixed-order block sums
        for (int o = 16; o > 0; o >>= 1) {
            da += __shfl_down_sync(0xffffffffu, da, o);
            db += __shfl_down_sync(0xffffffffu, db, o);
        }
        if ((threadIdx.x & 31) == 0) {
            red[0][threadIdx.x >> 5] = da;
            red[1][threadIdx.x >> 5] = db;
        }
        __syncthreads();
        if (threadIdx.x < 2 && (threadIdx.x == 0 || has_b)) {
            double s = 0.0;
            for (int k = 0; k < TH / 32; ++k) s += red[threadIdx.x][k];
            dots[(int64_t)(threadIdx.x ? vb : va) * ndot_stride + blockIdx.x] = s;
        }
    }
}

namespace {
struct RunA {
    const Args& a;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = Plan<B, E>;
        auto k = kd_pass_a<B, E, NT>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<dim3((a.n1 + NT - 1) / NT, a.np), NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(
            a.vin, a.ld_in, a.scale, a.nvec, a.pair0, a.bits, a.wpr, a.n1, a.logC, a.slab, a.tw, a.skip);
        KRY_CHECK_LAUNCH();
    }
};
struct RunB {
    const Args& a;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = Plan<B, E>;
        auto k = kd_pass_b<B, E, NT>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<dim3((a.M2 + NT - 1) / NT, a.np), NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(
            a.slab, a.lamT, a.n1, a.M2, a.logC, a.tw, a.pair0, a.lam_stride, a.vpt, a.skip, a.nvec);
        KRY_CHECK_LAUNCH();
    }
};
template <int MODE>
struct RunC {
    const Args& a;
    cudaStream_t st;
    template <int B, int E, int NT>
    void run() const {
        using P = Plan<B, E>;
        auto k = kd_pass_c<B, E, NT, MODE>;
        KRY_ALLOW_MAX_SMEM(k);
        k<<<dim3((a.n1 + NT - 1) / NT, a.np), NT * P::LT, (size_t)NT * P::SLOTS * 16, st>>>(
            a.slab, a.vin, a.ld_in, a.scale, a.vout, a.ld_out, a.nvec, a.pair0, a.bits, a.wpr, a.n1, a.n2, a.logC,
            a.tau2, a.dots, a.nds, a.tw, a.tau2v, a.vpt, a.skip);
        KRY_CHECK_LAUNCH();
    }
};
}  // namespace

void launch(const Args& a, cudaStream_t st) {
    dispatch<true>(a.M2, a.row, RunA{a, st});
    dispatch<true>(a.M1, a.col, RunB{a, st});
    if (a.mode == 0) dispatch<true>(a.M2, a.row, RunC<0>{a, st});
    else dispatch<true>(a.M2, a.row, RunC<1>{a, st});
}

}  // namespace kf64
