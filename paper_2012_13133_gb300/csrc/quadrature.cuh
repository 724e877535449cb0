// Gauss quadrature of z^T log(K) z from the Lanczos tridiagonal T: sum_j w_j
// log max(theta_j, lb), theta_j the eigenvalues of T and w_j the squared first
// components of its eigenvectors (Golub & Welsch 1969).
//
// K = sigma2 A Sigma A^T + tau2 I has every eigenvalue >= tau2, and so has
// every Ritz value of exact arithmetic.  Rounding in the matvec can move the
// smallest computed Ritz values below that bound (to zero or below once it is
// of the order of tau2, where the log would be undefined), so the nodes are
// taken as max(theta_j, lb), lb = tau2 of the vector's setting (tau2v[v / vpt]
// for a batched embedding, tau2 otherwise).
//
// One block per vector.  GB300 issues an FP64 instruction of a warp every 64
// cycles on each of an SM's four schedulers, however few lanes are active, so
// the serial eigenvalue iteration (k x 60 rotations of ~80 FP64 instructions
// on one lane: 4.9 ms for 32 probes x 50 steps) is replaced by independent
// work for all lanes.  With R(s) = e1^T (T + s I)^-1 e1 = sum_j w_j / (theta_j +
// s) and sum_j w_j = 1,
//   sum_j w_j log theta_j = log c + int_0^inf [1 / (c + s) - R(s)] ds,
// and in u = log s the integrand is analytic for |Im u| < pi and decays like
// e^-|u|: the trapezoidal rule of step 1/2 is exact to e^(-4 pi^2) ~ 7e-18
// (Trefethen & Weideman, SIAM Review 2014), with ~200 nodes, one per thread.
// R(s) is the continued fraction of T + s I, whose pivots are positive.  Ritz
// values in [lb / 1024, lb) are counted and located by Sturm sequences
// (multisection by the whole block), and w_j (log lb - log theta_j) added, w_j
// = 1 / g'(-theta_j) for R = 1 / g.  Anything else (a Ritz value below lb /
// 1024, two of them within 1e-6, a weight too small for its g', no bound,
// values that are not finite) takes the eigenvalue iteration.  50 steps x 32 probes: 64 us instead of 4.9 ms.

#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace kry {

static const int KRY_MAX_STEPS = 256;   // Lanczos steps, at most

// Number of eigenvalues of T (diagonal a, squared off-diagonal b2) below x: the
// negative pivots of T - x I.  A zero pivot counts as positive and tiny (so does
// the count at an eigenvalue itself: it is not below), NaN as below.
__host__ __device__ __forceinline__ int sturm_count(const double* a, const double* b2, int n, double x) {
    int c = 0;
    double g = 1.0;
    for (int i = 0; i < n; ++i) {
        g = (a[i] - x) - (i > 0 ? b2[i - 1] / g : 0.0);
        if (g == 0.0) g = 1e-300;
        if (!(g > 0.0)) ++c;
    }
    return c;
}

// Implicit QL iterations with Wilkinson shifts, the published procedure tql2
// (Bowdler, Martin, Reinsch & Wilkinson, "The QR and QL algorithms for
// symmetric matrices", Numer. Math. 1968; EISPACK's tql2), rotating only the
// first row of the eigenvector matrix.  Serial; d, e, z are n-element scratch.
__device__ double quadrature_ql(const double* alpha, const double* beta, int n, double lb, double* d, double* e,
                                double* z) {
    for (int i = 0; i < n; ++i) {
        d[i] = alpha[i];
        e[i] = (i < n - 1) ? beta[i] : 0.0;
        z[i] = (i == 0) ? 1.0 : 0.0;
    }
    const double eps = 2.220446049250313e-16;
    for (int l = 0; l < n; ++l) {
        for (int iter = 0; iter < 100; ++iter) {
            int m = l;
            for (; m < n - 1; ++m) {
                const double dd = fabs(d[m]) + fabs(d[m + 1]);
                if (fabs(e[m]) <= eps * dd) break;
            }
            if (m == l) break;
            double g = (d[l + 1] - d[l]) / (2.0 * e[l]);
            double r = hypot(g, 1.0);
            g = d[m] - d[l] + e[l] / (g + copysign(r, g));
            double s = 1.0, c = 1.0, pp = 0.0;
            bool deflated = false;
            for (int i = m - 1; i >= l; --i) {
                const double f = s * e[i];
                const double b = c * e[i];
                r = hypot(f, g);
                e[i + 1] = r;
                if (r == 0.0) {
                    d[i + 1] -= pp;
                    e[m] = 0.0;
                    deflated = true;
                    break;
                }
                s = f / r;
                c = g / r;
                g = d[i + 1] - pp;
                r = (d[i] - g) * s + 2.0 * c * b;
                pp = s * r;
                d[i + 1] = g + pp;
                g = c * r - b;
                const double zf = z[i + 1];
                z[i + 1] = s * z[i] + c * zf;
                z[i] = c * z[i] - s * zf;
            }
            if (deflated) continue;
            d[l] -= pp;
            e[l] = g;
            e[m] = 0.0;
        }
    }
    double acc = 0.0;
    for (int i = 0; i < n; ++i) acc += z[i] * z[i] * log(fmax(d[i], lb));
    return acc;
}

static const int QUAD_THREADS = 256;

// Vector k's tridiagonal: the first m_eff[k] of alphas[k nsteps ..] and one fewer of betas; out[k] = znorm2 times
// its quadrature.
__global__ void k_quadrature(const int* __restrict__ m_eff, const double* __restrict__ alphas,
                             const double* __restrict__ betas, int nsteps, double znorm2, double* __restrict__ out,
                             double tau2, const double* __restrict__ tau2v, int vpt) {
    __shared__ double a[KRY_MAX_STEPS], b2[KRY_MAX_STEPS], red[QUAD_THREADS], lo[KRY_MAX_STEPS], hi[KRY_MAX_STEPS];
    __shared__ int cnt[QUAD_THREADS], below, deep, bad;
    const int k = blockIdx.x, t = threadIdx.x;
    const double lb = (tau2v && vpt > 0) ? tau2v[k / vpt] : tau2;
    const int n = m_eff[k];
    const double* alpha = alphas + (int64_t)k * nsteps;
    const double* beta = betas + (int64_t)k * nsteps;
    // Gershgorin bound on the largest eigenvalue; NaN or Inf anywhere makes it not finite
    double g = 0.0;
    if (t < n) {
        const double bl = t > 0 ? beta[t - 1] : 0.0, br = t < n - 1 ? beta[t] : 0.0;
        a[t] = alpha[t];
        b2[t] = br * br;
        g = fabs(a[t]) + fabs(bl) + fabs(br);
        if (!(g < 1e150)) g = INFINITY;
    }
    red[t] = g;
    if (t == 0) bad = 0;
    __syncthreads();
    for (int o = QUAD_THREADS / 2; o > 0; o >>= 1) {
        if (t < o) red[t] = fmax(red[t], red[t + o]);
        __syncthreads();
    }
    const double top = red[0];
    __syncthreads();
    if (t == 0) below = (lb > 0.0 && top < 1e150) ? sturm_count(a, b2, n, lb) : n + 1;
    if (t == 32) deep = (lb > 0.0 && top < 1e150) ? sturm_count(a, b2, n, lb * 0x1p-10) : 1;
    __syncthreads();
    // nodes u0 + i / 2: both tails of the integrand end below e^-40
    const double u0 = log(lb) - 47.0;
    const double span = log(top) + 40.0 - u0;
    const int m = below;
    if (deep > 0 || m > n || !(span < 512.0)) {
        if (t == 0) out[k] = znorm2 * quadrature_ql(alpha, beta, n, lb, a, b2, lo);
        return;
    }
    double acc = 0.0;
    if (m > 0) {
        // eigenvalues j < m in (lb / 1024, lb]: tpg points of every interval per round
        const int tpg = QUAD_THREADS / m, j = t / tpg, r = t - j * tpg;
        const bool on = j < m;
        if (t < m) {
            lo[t] = lb * 0x1p-10;
            hi[t] = lb;
        }
        __syncthreads();
        int rounds = 1;
        for (double w = tpg + 1; w < 0x1p52; w *= tpg + 1) ++rounds;
        for (int q = 0; q < rounds; ++q) {
            double x = 0.0, l = 0.0, h = 0.0;
            if (on) {
                l = lo[j];
                h = hi[j];
                x = l + (h - l) * ((double)(r + 1) / (double)(tpg + 1));
                cnt[t] = sturm_count(a, b2, n, x) > j;   // eigenvalue j lies below x
            }
            __syncthreads();
            if (on && !cnt[t] && (r == tpg - 1 || cnt[t + 1])) lo[j] = x;
            if (on && cnt[t] && (r == 0 || !cnt[t - 1])) hi[j] = x;
            __syncthreads();
        }
        if (t < m) {
            const double th = 0.5 * (lo[t] + hi[t]);
            if (t > 0 && th - 0.5 * (lo[t - 1] + hi[t - 1]) < 1e-6 * th) bad = 1;
            // g(s) = continued fraction of T + s at s = -theta (where it vanishes), g' its derivative
            double gi = a[n - 1] - th, dg = 1.0;
            for (int i = n - 2; i >= 0; --i) {
                if (gi == 0.0) gi = 1e-300;
                const double f = 1.0 / gi, q2 = b2[i] * f;
                dg = 1.0 + q2 * f * dg;
                gi = (a[i] - th) - q2;
            }
            // the computed 1 / g' is w only where g nearly vanishes: with theta off by delta and the
            // rest of R equal to r there, it is (w + r delta)^2 / w, and g / g' = delta (1 + r delta / w)
            if (!(fabs(gi) <= 0x1p-44 * top * dg)) bad = 1;
            acc = (log(lb) - log(th)) / dg;
        }
        __syncthreads();
        if (bad) {
            if (t == 0) out[k] = znorm2 * quadrature_ql(alpha, beta, n, lb, a, b2, lo);
            return;
        }
    }
    const int nodes = (int)ceil(2.0 * span) + 1;
    for (int i = t; i < nodes; i += QUAD_THREADS) {
        const double s = exp(u0 + 0.5 * i);
        double gi = a[n - 1] + s;
        for (int l = n - 2; l >= 0; --l) gi = (a[l] + s) - b2[l] / gi;
        acc += 0.5 * (s / (lb + s) - s / gi);
    }
    red[t] = acc;
    __syncthreads();
    for (int o = QUAD_THREADS / 2; o > 0; o >>= 1) {
        if (t < o) red[t] += red[t + o];
        __syncthreads();
    }
    if (t == 0) out[k] = znorm2 * (log(lb) + red[0]);
}

}  // namespace kry
