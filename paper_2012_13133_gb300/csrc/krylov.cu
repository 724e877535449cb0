// Krylov loops on the covariance matvec:
//   * stochastic Lanczos quadrature for log det K (Sec. 3.3 names stochastic
//     trace estimation as the alternative to the circulant log-det);
//   * conjugate gradients for K X = B with FP64 residual replacement (the
//     matvec-only solves that replace the O(n^3) inversions of Sec. 3);
//   * GLS beta and the profile log-likelihood; kriging means (the paper's
//     x-hat, Eq. act_xhat, by Woodbury) and simple-kriging variances (the
//     quantity the bootstrap of Sec. 3.5 estimates).
//
// Vectors are FP32 (or FP64 for FP64 embeddings).  Dot products are summed in a
// fixed order, so results do not depend on scheduling: a thread's in double-float
// (FP64 for FP64 vectors), a block's to FP64's precision and range (block_sums),
// the blocks' partials in FP64, by a small kernel or, in FP32 CG, by every block
// of the kernel that needs the sum.
#include <cuda_fp16.h>
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "dfloat.cuh"
#include "kry_internal.cuh"
#include "matern.cuh"
#include "quadrature.cuh"

namespace kry {

template <typename T>
void matvec_ex(kry_ctx* ctx, const kry_embed* e, const T* vin, int64_t ld_in, const double* scale, T* vout,
               int64_t ld_out, int nvec, double* dots, int nds, int vpt = 0, const int* skip = nullptr);
int matvec_num_partials(kry_ctx* ctx, const kry_embed* e, bool dbl, int nvec);

static const int RED_BLOCKS = 128;   // fixed block count of the vector reductions

// ------------------------------------------------------------------ probes

// splitmix64 output function (Steele, Lea & Flood 2014) of state x.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Vector v holds Rademacher probe (v mod nprobe): every covariance setting of a
// batched search sees the same probes.
template <typename T>
__global__ void k_probes(T* __restrict__ W, int64_t p, int64_t ld, int nprobe, uint64_t seed) {
    const int v = blockIdx.y;
    const uint64_t k = (uint64_t)(v % nprobe);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ld; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t key = seed ^ ((k << 32) | (uint64_t)i);
        W[(int64_t)v * ld + i] = i >= p ? (T)0 : (splitmix64(key) >> 63) ? (T)-1 : (T)1;
    }
}

// Run fn() under stream capture on the library's capture stream and replay the
// captured graph once, ordered after earlier work on ctx->stream and before
// later work on it.  Without graphs (ctx->use_graphs false) fn() runs directly.
template <class F>
static void run_captured(kry_ctx* ctx, F&& fn) {
    if (!ctx->use_graphs) {
        fn();
        return;
    }
    if (!ctx->cap_stream) KRY_CUDA(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
    cudaStream_t user = ctx->stream, cap = ctx->cap_stream;
    cudaEvent_t fork, join;
    KRY_CUDA(cudaEventCreateWithFlags(&fork, cudaEventDisableTiming));
    KRY_CUDA(cudaEventCreateWithFlags(&join, cudaEventDisableTiming));
    KRY_CUDA(cudaEventRecord(fork, user));
    KRY_CUDA(cudaStreamWaitEvent(cap, fork, 0));
    cudaGraph_t graph = nullptr;
    ctx->stream = cap;
    KRY_CUDA(cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed));
    try {
        fn();
    } catch (...) {
        cudaStreamEndCapture(cap, &graph);
        if (graph) cudaGraphDestroy(graph);
        ctx->stream = user;
        cudaEventDestroy(fork);
        cudaEventDestroy(join);
        throw;
    }
    ctx->stream = user;
    KRY_CUDA(cudaStreamEndCapture(cap, &graph));
    cudaGraphExec_t exec = nullptr;
    KRY_CUDA(cudaGraphInstantiate(&exec, graph, 0));
    KRY_CUDA(cudaGraphLaunch(exec, cap));
    KRY_CUDA(cudaEventRecord(join, cap));
    KRY_CUDA(cudaStreamWaitEvent(user, join, 0));
    KRY_CUDA(cudaGraphExecDestroy(exec));
    KRY_CUDA(cudaGraphDestroy(graph));
    KRY_CUDA(cudaEventDestroy(fork));
    KRY_CUDA(cudaEventDestroy(join));
}

// A launch sequence captured once into a CUDA graph (on the library's capture
// stream) and replayed on ctx->stream as often as needed.  Replays add the
// captured kernel count to the launch counter.  With profiling on, the matvec
// event pairs recorded during capture are re-recorded by every replay; the
// caller synchronises the stream after a replay and calls harvest(), which adds
// their times to the context's totals.
struct Replay {
    kry_ctx* ctx = nullptr;
    cudaGraphExec_t exec = nullptr;
    unsigned long long kernels = 0;
    std::vector<cudaEvent_t> ev;   // start/stop pairs owned by the graph's profiling nodes
    std::vector<int> nvec, dbl;
    explicit Replay(kry_ctx* c) : ctx(c) {}
    Replay(const Replay&) = delete;
    Replay& operator=(const Replay&) = delete;
    ~Replay() {
        if (exec) cudaGraphExecDestroy(exec);
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
    }
    template <class F>
    void capture(F&& fn) {
        if (!ctx->cap_stream) KRY_CUDA(cudaStreamCreateWithFlags(&ctx->cap_stream, cudaStreamNonBlocking));
        cudaStream_t user = ctx->stream, cap = ctx->cap_stream;
        const unsigned long long n0 = g_kry_launches.load();
        const size_t p0 = ctx->prof_nvec.size();
        cudaGraph_t graph = nullptr;
        ctx->stream = cap;
        KRY_CUDA(cudaStreamBeginCapture(cap, cudaStreamCaptureModeRelaxed));
        try {
            fn();
        } catch (...) {
            cudaStreamEndCapture(cap, &graph);
            if (graph) cudaGraphDestroy(graph);
            ctx->stream = user;
            throw;
        }
        ctx->stream = user;
        // the profiling pairs recorded by the capture belong to the graph from now on
        ev.assign(ctx->prof_ev.begin() + 2 * p0, ctx->prof_ev.end());
        nvec.assign(ctx->prof_nvec.begin() + p0, ctx->prof_nvec.end());
        dbl.assign(ctx->prof_dbl.begin() + p0, ctx->prof_dbl.end());
        ctx->prof_ev.resize(2 * p0);
        ctx->prof_nvec.resize(p0);
        ctx->prof_dbl.resize(p0);
        KRY_CUDA(cudaStreamEndCapture(cap, &graph));
        const cudaError_t err = cudaGraphInstantiate(&exec, graph, 0);
        cudaGraphDestroy(graph);
        KRY_CUDA(err);
        kernels = g_kry_launches.load() - n0;
        g_kry_launches.fetch_sub(kernels);   // counted when replayed
    }
    void launch() {
        KRY_CUDA(cudaGraphLaunch(exec, ctx->stream));
        g_kry_launches.fetch_add(kernels);
    }
    // After the stream has been synchronised following launch().
    void harvest() {
        for (size_t i = 0; i < nvec.size(); ++i) {
            float t = 0.f;
            KRY_CUDA(cudaEventElapsedTime(&t, ev[2 * i], ev[2 * i + 1]));
            ctx->prof_ms_acc[dbl[i]] += t;
            ctx->prof_calls_acc[dbl[i]] += 1;
            ctx->prof_vec_acc[dbl[i]] += nvec[i];
        }
    }
};

// ------------------------------------------------------------------ block reduction helper

template <int N>
__device__ __forceinline__ void block_sum_store(double (&v)[N], double* out, int64_t out_stride) {
    __shared__ double red[N][32];
#pragma unroll
    for (int a = 0; a < N; ++a)
        for (int o = 16; o > 0; o >>= 1) v[a] += __shfl_down_sync(0xffffffffu, v[a], o);
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0)
#pragma unroll
        for (int a = 0; a < N; ++a) red[a][w] = v[a];
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
#pragma unroll
        for (int a = 0; a < N; ++a) {
            double s = 0.0;
            for (int k = 0; k < nw; ++k) s += red[a][k];
            out[a * out_stride] = s;
        }
    }
}

// Sum of part[0..n) by one block in a fixed order (strided per-thread sums,
// then a shuffle tree, then the warp sums in order); the result is valid in
// thread 0.  Deterministic for a given block size.
__device__ __forceinline__ double block_sum(const double* __restrict__ part, int n) {
    __shared__ double ws[32];
    double v = 0.0;
    for (int b = threadIdx.x; b < n; b += blockDim.x) v += part[b];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
    return t;
}

static const int FIN_THREADS = 256;   // block size of the per-vector finalisers

// Four consecutive FP32 values through one 16-byte access (the caller guarantees
// the alignment).
__device__ __forceinline__ void load4(const float* __restrict__ src, float (&out)[4]) {
    const float4 a = *reinterpret_cast<const float4*>(src);
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
}
__device__ __forceinline__ void store4(float* __restrict__ dst, const float (&v)[4]) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}

// Block sum of a running dot product over THREADS threads in a fixed order, valid
// in thread 0.
template <int THREADS>
__device__ __forceinline__ double block_total(const DotAcc<float>& acc) {
    return block_sums<1, THREADS / 32>({acc.a});
}
template <int THREADS>
__device__ __forceinline__ double block_total(const DotAcc<double>& acc) {
    __shared__ double red[THREADS / 32];
    double v = acc.s;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x != 0) return 0.0;
    for (int w = 1; w < THREADS / 32; ++w) v += red[w];
    return v;
}

// Eight consecutive values through 16-byte accesses (the caller guarantees the
// alignment), FP16 ones as FP32.
__device__ __forceinline__ void load8(const float* __restrict__ src, float (&out)[8]) {
    const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
    out[0] = a.x; out[1] = a.y; out[2] = a.z; out[3] = a.w;
    out[4] = b.x; out[5] = b.y; out[6] = b.z; out[7] = b.w;
}
__device__ __forceinline__ void load8(const __half* __restrict__ src, float (&out)[8]) {
    const uint4 q = *reinterpret_cast<const uint4*>(src);
    __half2 h[4];
    memcpy(h, &q, 16);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(h[e]);
        out[2 * e] = f.x;
        out[2 * e + 1] = f.y;
    }
}
__device__ __forceinline__ void load8(const double* __restrict__ src, double (&out)[8]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const double2 d = reinterpret_cast<const double2*>(src)[e];
        out[2 * e] = d.x;
        out[2 * e + 1] = d.y;
    }
}
__device__ __forceinline__ void store8(float* __restrict__ dst, const float (&v)[8]) {
    reinterpret_cast<float4*>(dst)[0] = make_float4(v[0], v[1], v[2], v[3]);
    reinterpret_cast<float4*>(dst)[1] = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(double* __restrict__ dst, const double (&v)[8]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) reinterpret_cast<double2*>(dst)[e] = make_double2(v[2 * e], v[2 * e + 1]);
}
__device__ __forceinline__ void store8(__half* __restrict__ dst, const float (&v)[8]) {
    __half2 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = __floats2half2_rn(v[2 * e], v[2 * e + 1]);
    uint4 q;
    memcpy(&q, h, 16);
    *reinterpret_cast<uint4*>(dst) = q;
}

// ------------------------------------------------------------------ Lanczos

struct LanczosState {
    double* s_cur;    // [nprobe] scale of the current vector: q_j = s_cur * W_cur
    double* s_prev;   // [nprobe]
    double* alpha;    // [nprobe][nsteps]
    double* beta;     // [nprobe][nsteps]
    int* m_eff;       // [nprobe] Lanczos steps kept (early stop on breakdown)
    // partial reorthogonalisation only (all NULL without it)
    double* s_hist;   // [nprobe][nsteps] scale of every stored basis vector: q_i = s_hist[i] * W_i
    double* omega;    // [3][nprobe][nsteps + 1] estimates of q_j^T q_k for j-1, j, j+1 (buffer j mod 3)
    int* flag;        // [nprobe] 1: reorthogonalise the new vector of this step
    int* force;       // [nprobe] 1: the next new vector is reorthogonalised too
    int* again;       // [nprobe] 1: a flagged vector takes a second Gram-Schmidt pass
    double* pre2;     // [nprobe] ||w||^2 before the Gram-Schmidt pass of a flagged vector
};

__global__ void k_lanczos_init(LanczosState S, int nprobe, int nsteps, double s0) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= nprobe) return;
    S.s_cur[k] = s0;
    S.s_prev[k] = 0.0;
    S.m_eff[k] = nsteps;
    if (S.s_hist) {
        S.s_hist[(int64_t)k * nsteps] = s0;
        S.omega[(int64_t)k * (nsteps + 1)] = 1.0;   // omega_{0,0}
        S.flag[k] = 0;
        S.force[k] = 0;
    }
}

// alpha_j = sum of the block partials of q_j^T K q_j (fixed order).
__global__ void k_lanczos_alpha(LanczosState S, const double* __restrict__ part, int nblk, int nprobe, int nsteps,
                                int j) {
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.x;   // one block per vector
    const double a = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x == 0) S.alpha[(int64_t)k * nsteps + j] = a;
}

// The Lanczos vectors keep a leading dimension ld that is a multiple of eight
// and zeros past p (the probes and the zeroed matvec output start them so, and
// the recurrences keep them), so that every access is 16 bytes wide whatever p
// is.

// w_next = U - alpha_j s_cur W_cur - beta_{j-1} s_prev W_prev;  partial ||w_next||^2.
// H (FP32 with reorthogonalisation; else NULL): the current basis vector,
// normalised and scaled to entries of order one, sqrtp s_cur W_cur, for the
// FP16 reorthogonalisation store.
template <typename T>
__global__ void k_lanczos_update(const T* __restrict__ U, const T* __restrict__ Wc, const T* __restrict__ Wp,
                                 T* __restrict__ Wn, int64_t ld, LanczosState S, int nsteps, int j,
                                 double* __restrict__ part, __half* __restrict__ H, double sqrtp) {
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.y;
    const double a = S.alpha[(int64_t)k * nsteps + j], sc = S.s_cur[k];
    const T ca = (T)(a * sc);
    const T cb = (T)((j > 0 ? S.beta[(int64_t)k * nsteps + j - 1] : 0.0) * S.s_prev[k]);
    const T ch = (T)(sc * sqrtp);
    const int64_t off = (int64_t)k * ld;
    DotAcc<T> nrm;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 8; x < ld; x += (int64_t)gridDim.x * blockDim.x * 8) {
        T u[8], wc[8], wp[8];
        load8(U + off + x, u);
        load8(Wc + off + x, wc);
        // at j = 0 there is no previous vector (its buffer is not initialised)
        if (j > 0) {
            load8(Wp + off + x, wp);
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) wp[e] = (T)0;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            u[e] = u[e] - ca * wc[e] - cb * wp[e];
            nrm.add_prod(u[e], u[e]);
        }
        store8(Wn + off + x, u);
        if constexpr (sizeof(T) == 4) {
            if (H) {
#pragma unroll
                for (int e = 0; e < 8; ++e) wc[e] *= ch;
                store8(H + off + x, wc);
            }
        }
    }
    const double s = block_total<256>(nrm);
    if (threadIdx.x == 0) part[(int64_t)k * gridDim.x + blockIdx.x] = s;
}

// beta_j = ||w_next||; early stop when beta_j < 1e-12 |alpha_1|; rescale.
__global__ void k_lanczos_beta(LanczosState S, const double* __restrict__ part, int nblk, int nprobe, int nsteps,
                               int j) {
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.x;   // one block per vector
    const double s = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x != 0) return;
    const double bj = sqrt(s);
    const bool stopped = S.m_eff[k] < nsteps;
    if (!stopped && bj < 1e-12 * fabs(S.alpha[(int64_t)k * nsteps])) S.m_eff[k] = j + 1;
    const bool now_stopped = S.m_eff[k] < nsteps;
    S.beta[(int64_t)k * nsteps + j] = now_stopped ? 0.0 : bj;
    S.s_prev[k] = S.s_cur[k];
    S.s_cur[k] = now_stopped ? 0.0 : 1.0 / bj;
    if (S.s_hist && j + 1 < nsteps) S.s_hist[(int64_t)k * nsteps + j + 1] = S.s_cur[k];
}

// ------------------------------------------------------------------ partial reorthogonalisation
//
// The basis may lose orthogonality (Sec. 3.2, which leaves a reorthogonalisation
// scheme to the user); in FP32 the loss reaches the Gauss quadrature within a
// few tens of steps.  Partial reorthogonalisation (H. D. Simon, "The Lanczos
// algorithm with partial reorthogonalization", Math. Comp. 42, 1984) tracks
// estimates omega_{j,k} of q_j^T q_k by a scalar recurrence derived from the
// three-term recurrences of q_j and q_k, with a rounding term of size
// eps_round (beta_k + beta_j); when the largest estimate for the new vector
// exceeds sqrt(eps) (eps = unit roundoff of the vectors), the new vector and
// the one after it are orthogonalised against every stored basis vector
// (classical Gram-Schmidt, repeated once when it cancels most of the vector)
// and their estimates reset to what the pass leaves: eps, or for FP32 vectors,
// whose basis is stored in FP16 (2^-11 relative rounding, half the traffic of
// an FP32 store), the FP16 rounding of a removed component of size sqrt(eps),
// about 2 eps.  The rounding term uses
// eps_round = eps log2(M1 M2): the local error of a step is that of the FFT
// matvec, which grows with the log of the transform size.  With eps alone,
// FP32 runs on smooth long-range covariances (512^2 grid, range >= 0.1)
// lost orthogonality unnoticed: per-probe values up to 3% off the FP64 run,
// some NaN; with eps_round they agree to 2e-5 at 5% more time.  Semi-orthogonality
// (|q_j^T q_k| <= sqrt(eps)) keeps the tridiagonal equal to the projection of K
// on the Krylov space up to O(eps ||K||) (Simon 1984).  Decisions are per
// vector, on the device, so the launch sequence is fixed and graph-capturable.

// A running sum: double-float (hi, lo) for FP32 vectors, (sum, 0) in FP64.
template <typename T>
struct Pair {
    T hi, lo;
};
__device__ __forceinline__ void pair_add(Pair<float>& a, Pair<float> b) { df_add(a.hi, a.lo, b.hi, b.lo); }
__device__ __forceinline__ void pair_add(Pair<double>& a, Pair<double> b) { a.hi += b.hi; }
// a += x y: the product rounded to T, FP32 sums kept exactly but for the last bits of lo.
__device__ __forceinline__ void pair_add_prod(Pair<float>& a, float x, float y) {
    float s, t;
    two_sum(a.hi, __fmul_rn(x, y), s, t);
    a = {s, __fadd_rn(a.lo, t)};
}
__device__ __forceinline__ void pair_add_prod(Pair<double>& a, double x, double y) { a.hi = fma(x, y, a.hi); }
__device__ __forceinline__ double pair_value(Pair<float> a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double pair_value(Pair<double> a) { return a.hi; }
template <typename T>
__device__ __forceinline__ Pair<T> pair_xor(Pair<T> a, int o) {
    Pair<T> b;
    b.hi = __shfl_xor_sync(0xffffffffu, a.hi, o);
    b.lo = sizeof(T) == 4 ? __shfl_xor_sync(0xffffffffu, a.lo, o) : (T)0;
    return b;
}

// Sums of eight values over a warp: lanes 4a .. 4a + 3 return the sum of s[a].
// Each of the first three exchanges hands half of the values over, so that it
// takes 9 exchanges instead of 40.
template <typename T>
__device__ __forceinline__ Pair<T> warp_sum8(Pair<T> (&s)[8], int lane) {
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        const bool up = lane & (4 * h);
#pragma unroll
        for (int a = 0; a < h; ++a) {
            const Pair<T> keep = up ? s[a + h] : s[a], give = up ? s[a] : s[a + h];
            s[a] = keep;
            pair_add(s[a], pair_xor(give, 4 * h));
        }
    }
    pair_add(s[0], pair_xor(s[0], 2));
    pair_add(s[0], pair_xor(s[0], 1));
    return s[0];
}

// Estimates for q_{j+1} from ||w||^2 partials (before any reorthogonalisation);
// sets flag[k] when w is to be reorthogonalised.  One block per vector, one
// thread per estimate (the recurrence over i < j reads the two previous
// vectors' estimates only; j < nsteps <= KRY_MAX_STEPS = FIN_THREADS).  Only as
// many warps as there are estimates: every FP64 instruction of an idle warp
// holds a pipe for 64 cycles too (32 probes x 50 steps on 512^2: 11.36 -> 11.15 ms).
__global__ void k_pro_omega(LanczosState S, const double* __restrict__ part, int nblk, int nsteps, int j,
                            double eps, double eps_round, double omega_reset) {
    pdl_wait();
    pdl_launch_dependents();
    __shared__ double sh_s, sh_t[8], sh_w[8];
    const int k = blockIdx.x, i = threadIdx.x;
    const double s0 = block_sum(part + (int64_t)k * nblk, nblk);
    if (i == 0) sh_s = s0;
    __syncthreads();
    const double s = sh_s;
    const int64_t ostride = (int64_t)gridDim.x * (nsteps + 1);
    double* on = S.omega + ((j + 1) % 3) * ostride + (int64_t)k * (nsteps + 1);   // omega_{j+1, .}
    const double* oc = S.omega + (j % 3) * ostride + (int64_t)k * (nsteps + 1);   // omega_{j, .}
    const double* op = S.omega + ((j + 2) % 3) * ostride + (int64_t)k * (nsteps + 1);   // omega_{j-1, .}
    const double* al = S.alpha + (int64_t)k * nsteps;
    const double* be = S.beta + (int64_t)k * nsteps;
    const double bj = sqrt(s);
    if (S.m_eff[k] < nsteps || !(bj > 0.0)) {   // stopped: nothing to keep orthogonal
        if (i == 0) S.flag[k] = 0;
        return;
    }
    const double aj = al[j];
    double tnorm = fabs(aj) + bj, worst = 0.0;
    if (i < j) {
        tnorm = fmax(tnorm, fabs(al[i]) + be[i]);
        double t = be[i] * oc[i + 1] + (al[i] - aj) * oc[i] - be[j - 1] * op[i];
        if (i > 0) t += be[i - 1] * oc[i - 1];
        t += copysign(eps_round * (be[i] + bj), t);
        t /= bj;
        on[i] = t;
        worst = fabs(t);
    }
    for (int o = 16; o > 0; o >>= 1) {
        tnorm = fmax(tnorm, __shfl_xor_sync(0xffffffffu, tnorm, o));
        worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    }
    if ((i & 31) == 0) {
        sh_t[i >> 5] = tnorm;
        sh_w[i >> 5] = worst;
    }
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        tnorm = fmax(tnorm, sh_t[w]);
        worst = fmax(worst, sh_w[w]);
    }
    const double last = eps_round * tnorm / bj;   // omega_{j+1, j}
    worst = fmax(worst, last);
    const int force = S.force[k];
    const int f = (force || worst > sqrt(eps)) ? 1 : 0;
    __syncthreads();   // force is read by every thread before thread 0 replaces it
    if (i == 0) {
        on[j] = f ? omega_reset : last;
        on[j + 1] = 1.0;
        S.flag[k] = f;
        S.pre2[k] = s;
        S.force[k] = f && !force;   // the vector after a reorthogonalised one is reorthogonalised too
    }
    if (f && i < j) on[i] = omega_reset;
}

// Whether vector k takes the Gram-Schmidt pass: its flag in the first pass.  In
// the second, "twice is enough" (Kahan; Parlett, The Symmetric Eigenvalue
// Problem, 1980, Sec. 6-9): a flagged vector whose norm fell below 1/sqrt(2) of
// its norm before the first pass lost most of itself to cancellation, and its
// rounding errors are then large relative to what is left.  Every block of
// the vector decides alike from the same partials; block 0 records it for the
// update that follows.
__device__ __forceinline__ bool reorth_now(const LanczosState& S, int k, int pass, const double* __restrict__ part,
                                           int nblk) {
    const bool first = S.flag[k] != 0;
    if (pass == 0) return first;
    if (!first) {
        if (blockIdx.x == 0 && threadIdx.x == 0) S.again[k] = 0;
        return false;
    }
    __shared__ double s;
    const double t = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x == 0) s = t;
    __syncthreads();
    const bool yes = s < 0.5 * S.pre2[k];
    if (blockIdx.x == 0 && threadIdx.x == 0) S.again[k] = yes ? 1 : 0;
    return yes;
}

// Partial dot products W_i^T w (i = 0..j) of each flagged vector against the
// basis store Q (T, or FP16 for FP32 vectors).  A block holds its 8192 values of
// w (FP64: 2048) in registers and sweeps the basis eight vectors at a time, so
// every thread has 32 (FP64: 8 times four) independent 16-byte loads in flight.
// Products are in the vector precision T (a coefficient only needs a few correct
// digits: it removes a component of size <= sqrt(eps)), FP32 ones added in
// double-float throughout, so that the coefficient is as exact as its products
// are; FP64 ones in FP64.  dpart rows are
// [nvec][nsteps + 8][gridDim.x] (hi, lo) pairs: a sweep's rows past j (zeros)
// stay in the vector's padding.  What held the pass before: one FP64 shuffle
// tree of eight values per block and sweep (64 cycles an instruction) for 2 to
// 6 values a thread, and 2-byte loads where p is odd (32 vectors of 183,501
// values, 50 steps: 6.4 ms -> 2.1 ms).
template <typename T, typename Sq>
__global__ void __launch_bounds__(256) k_reorth_dots(const Sq* __restrict__ Q, const T* __restrict__ Wn, int nvec,
                                                     int64_t ld, int j, LanczosState S, int pass,
                                                     const double* __restrict__ part, int nblk, int nsteps,
                                                     Pair<T>* __restrict__ dpart) {
    pdl_wait();
    pdl_launch_dependents();
    constexpr int NC = sizeof(T) == 4 ? 4 : 1;   // groups of eight values a thread holds
    __shared__ Pair<T> red[2][8][8];
    const int k = blockIdx.y;
    if (!reorth_now(S, k, pass, part, nblk)) return;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t vs = (int64_t)nvec * ld;   // distance of consecutive basis vectors
    for (int64_t base = 0, chunk = 0; base < ld; base += (int64_t)gridDim.x * NC * 2048, ++chunk) {
        int64_t x[NC];
        bool in[NC];
        T w[NC][8];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int64_t y = base + ((int64_t)blockIdx.x * NC + c) * 2048 + threadIdx.x * 8;
            in[c] = y < ld;
            x[c] = (int64_t)k * ld + (in[c] ? y : 0);
            load8(Wn + x[c], w[c]);
#pragma unroll
            for (int e = 0; e < 8; ++e) w[c][e] = in[c] ? w[c][e] : (T)0;
        }
        for (int i0 = 0, sweep = 0; i0 <= j; i0 += 8, ++sweep) {
            Pair<T> acc[8];
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                acc[a] = {(T)0, (T)0};
                const Sq* q = Q + (int64_t)min(i0 + a, j) * vs;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    T qv[8];
                    load8(q + x[c], qv);
#pragma unroll
                    for (int e = 0; e < 8; ++e) pair_add_prod(acc[a], qv[e], w[c][e]);
                }
            }
            Pair<T> tot = warp_sum8<T>(acc, lane);   // of acc[lane >> 2] over the warp
            if ((lane & 3) == 0) red[sweep & 1][wp][lane >> 2] = tot;
            __syncthreads();
            if (threadIdx.x < 8) {
                tot = red[sweep & 1][0][threadIdx.x];
#pragma unroll
                for (int u = 1; u < 8; ++u) pair_add(tot, red[sweep & 1][u][threadIdx.x]);
                Pair<T>* out = dpart + ((int64_t)k * (nsteps + 8) + i0 + threadIdx.x) * gridDim.x + blockIdx.x;
                if (i0 + (int)threadIdx.x > j) tot = {(T)0, (T)0};
                if (chunk) pair_add(tot, *out);
                *out = tot;
            }
        }
        __syncthreads();
    }
}

// w -= sum_i coef_i W_i (in the basis precision) for flagged vectors; partial
// ||w||^2 replaces the update's so that beta_j is the norm after
// reorthogonalisation.  Every block sums the dot partials itself (one warp per
// basis vector, fixed order): coef_i = s_i (q_i^T w) = s_i^2 (W_i^T w) for a
// store of the unnormalised W_i, or (q_i^T w) / sqrt(p) = (H_i^T w) / p for the
// FP16 store H_i = sqrt(p) q_i (hscale = 1 / p, else 0).
template <typename T, typename Sq>
__global__ void __launch_bounds__(256) k_reorth_apply(const Sq* __restrict__ Q, T* __restrict__ Wn, int nvec,
                                                      int64_t ld, int j, LanczosState S, int pass, int nsteps,
                                                      const Pair<T>* __restrict__ dpart, int nd, double hscale,
                                                      double* __restrict__ part) {
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.y;
    if (pass == 0 ? !S.flag[k] : !S.again[k]) return;
    __shared__ Pair<T> tot[KRY_MAX_STEPS];
    __shared__ T c[KRY_MAX_STEPS];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    for (int i = wp; i <= j; i += 8) {
        const Pair<T>* d = dpart + ((int64_t)k * (nsteps + 8) + i) * nd;
        Pair<T> s = {(T)0, (T)0};
        for (int b = lane; b < nd; b += 32) pair_add(s, d[b]);
        for (int o = 16; o > 0; o >>= 1) pair_add(s, pair_xor(s, o));
        if (lane == 0) tot[i] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
        const double d = pair_value(tot[i]), si = S.s_hist[(int64_t)k * nsteps + i];
        c[i] = (T)(hscale > 0.0 ? hscale * d : si * si * d);
    }
    __syncthreads();
    T* w = Wn + (int64_t)k * ld;
    DotAcc<T> nrm;
    for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 8; x < ld; x += (int64_t)gridDim.x * blockDim.x * 8) {
        T proj[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) proj[e] = 0;
#pragma unroll 4
        for (int i = 0; i <= j; ++i) {
            T qv[8];
            load8(Q + ((int64_t)i * nvec + k) * ld + x, qv);
#pragma unroll
            for (int e = 0; e < 8; ++e) proj[e] += c[i] * qv[e];
        }
        T r[8];
        load8(w + x, r);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            r[e] -= proj[e];
            nrm.add_prod(r[e], r[e]);
        }
        store8(w + x, r);
    }
    const double s = block_total<256>(nrm);
    if (threadIdx.x == 0) part[(int64_t)k * gridDim.x + blockIdx.x] = s;
}

// Lanczos over nvec vectors (vector v holds probe v mod nprobe; vpt consecutive
// vectors share one covariance setting of a batched embedding, 0 = one
// setting).  Step 0 runs directly (it sizes every buffer); steps 1.. are
// captured into one CUDA graph and replayed as one launch.  Without
// reorthogonalisation three basis vectors rotate through three buffers; with it
// every basis vector is kept ([nsteps][nvec][p]) for the Gram-Schmidt passes.
template <typename T>
static void lanczos_logdet(kry_ctx* ctx, const kry_embed* e, int nvec, int nprobe, int nsteps, uint64_t seed,
                           double* per_vec, int vpt, bool reorth) {
    const bool dbl = sizeof(T) == 8;
    const int64_t p = ctx->p;
    const int64_t ld = (p + 7) & ~(int64_t)7;   // leading dimension of every Lanczos vector (zeros past p)
    const int nblkC = matvec_num_partials(ctx, e, dbl, nvec);
    const size_t vbytes = (size_t)nvec * ld * sizeof(T);
    ctx->work[0].ensure(vbytes);
    T* U = ctx->work[0].as<T>();
    if (ld > p)
        KRY_CUDA(cudaMemset2DAsync(U + p, ld * sizeof(T), 0, (ld - p) * sizeof(T), nvec, ctx->stream));
    T* Q = nullptr;   // FP64 basis store with reorthogonalisation
    T* W[3] = {nullptr, nullptr, nullptr};
    // FP32 with reorthogonalisation: the three-term recurrence runs on three
    // rotating FP32 vectors, and every basis vector is also kept, normalised,
    // in an FP16 store for the Gram-Schmidt passes (half the traffic and memory
    // of an FP32 store; k_lanczos_update)
    const bool hstore = reorth && !dbl;
    __half* H = nullptr;
    if (reorth && dbl) {
        ctx->work[1].ensure(vbytes * nsteps);
        Q = ctx->work[1].as<T>();
    } else if (hstore) {
        ctx->work[1].ensure((size_t)nvec * ld * sizeof(__half) * nsteps);
        H = ctx->work[1].as<__half>();
        ctx->work[2].ensure(3 * vbytes);
        for (int b = 0; b < 3; ++b) W[b] = ctx->work[2].as<T>() + (size_t)b * nvec * ld;
    } else {
        for (int b = 1; b < 4; ++b) ctx->work[b].ensure(vbytes);
        for (int b = 0; b < 3; ++b) W[b] = ctx->work[b + 1].as<T>();
    }
    auto basis = [&](int i) -> T* { return Q ? Q + (size_t)i * nvec * ld : W[i % 3]; };
    // blocks per vector of the streaming kernels: 16 values a thread and more
    const int nrb = (int)std::max<int64_t>(1, std::min<int64_t>(RED_BLOCKS, (ld + 4095) / 4096));
    const int ndot = (int)std::max<int64_t>(1, std::min<int64_t>(RED_BLOCKS, (ld + (dbl ? 2047 : 8191)) / (dbl ? 2048 : 8192)));
    const int nred = std::max(nblkC, nrb);
    ctx->work[4].ensure((size_t)nvec * nred * sizeof(double));
    double* part = ctx->work[4].as<double>();
    const size_t nsc = (size_t)nvec * (2 * nsteps + 4) + nvec;
    const size_t npro = reorth ? (size_t)nvec * (nsteps + 3 * (nsteps + 1) + 1) : 0;
    ctx->scal.ensure((nsc + npro) * sizeof(double));
    double* sc = ctx->scal.as<double>();
    LanczosState S;
    S.s_cur = sc;
    S.s_prev = sc + nvec;
    S.alpha = sc + 2 * nvec;
    S.beta = S.alpha + (size_t)nvec * nsteps;
    double* res = S.beta + (size_t)nvec * nsteps;
    ctx->work[5].ensure((size_t)nvec * 4 * sizeof(int));
    S.m_eff = ctx->work[5].as<int>();
    S.s_hist = S.omega = S.pre2 = nullptr;
    S.flag = S.force = S.again = nullptr;
    Pair<T>* dpart = nullptr;
    if (reorth) {
        S.s_hist = sc + nsc;
        S.omega = S.s_hist + (size_t)nvec * nsteps;
        S.pre2 = S.omega + (size_t)3 * nvec * (nsteps + 1);
        S.flag = S.m_eff + nvec;
        S.force = S.flag + nvec;
        S.again = S.force + nvec;
        ctx->work[6].ensure((size_t)nvec * (nsteps + 8) * ndot * sizeof(Pair<T>));
        dpart = ctx->work[6].as<Pair<T>>();
    }
    const double eps = dbl ? 1.1102230246251565e-16 : 5.9604644775390625e-08;   // unit roundoff of T
    // rounding term of the omega recurrence: the local error of one Lanczos step
    // is dominated by the FFT matvec, whose error grows like log2 of the
    // transform size (eps log2(M1 M2) ||K||, not eps ||K||)
    const double eps_round = eps * std::log2((double)e->M1 * (double)e->M2);
    // what a Gram-Schmidt pass leaves of q_i^T w: rounding of order eps, or, with
    // the FP16 store, the FP16 rounding (2^-11) of a removed component of size
    // up to sqrt(eps)
    const double omega_reset = hstore ? std::max(eps, std::sqrt(eps) * 4.8828125e-4) : eps;

    const int tb = 256;
    k_lanczos_init<<<(nvec + tb - 1) / tb, tb, 0, ctx->stream>>>(S, nvec, nsteps, 1.0 / sqrt((double)p));
    KRY_CHECK_LAUNCH();
    dim3 gp((unsigned)std::min<int64_t>((ld + 255) / 256, 1024), nvec);
    k_probes<T><<<gp, 256, 0, ctx->stream>>>(basis(0), p, ld, nprobe, seed);
    KRY_CHECK_LAUNCH();
    const dim3 gu(nrb, nvec), gd(ndot, nvec);
    const double sqrtp = sqrt((double)p), hscale = hstore ? 1.0 / (double)p : 0.0;
    // launches of one step, back to back with programmatic dependent launch
    auto step = [&](int j) {
        cudaStream_t st = ctx->stream;
        T* Wc = basis(j);
        T* Wp = basis(j > 0 ? j - 1 : 0);
        matvec_ex<T>(ctx, e, Wc, ld, S.s_cur, U, ld, nvec, part, nblkC, vpt);
        launch_pdl(k_lanczos_alpha, dim3(nvec), dim3(FIN_THREADS), 0, st, S, part, nblkC, nvec, nsteps, j);
        if (j == nsteps - 1) return;
        T* Wn = basis(j + 1);
        launch_pdl(k_lanczos_update<T>, gu, dim3(256), 0, st, U, Wc, Wp, Wn, ld, S, nsteps, j, part,
                   hstore ? H + (size_t)j * nvec * ld : nullptr, sqrtp);
        if (reorth) {
            launch_pdl(k_pro_omega, dim3(nvec), dim3(std::min(FIN_THREADS, std::max(64, (j + 31) / 32 * 32))), 0, st, S, part, nrb, nsteps, j, eps, eps_round,
                       omega_reset);
            for (int pass = 0; pass < 2; ++pass) {   // the second for vectors that lost most of their norm
                if constexpr (sizeof(T) == 4) {
                    launch_pdl(k_reorth_dots<T, __half>, gd, dim3(256), 0, st, H, Wn, nvec, ld, j, S, pass, part, nrb,
                               nsteps, dpart);
                    launch_pdl(k_reorth_apply<T, __half>, gu, dim3(256), 0, st, H, Wn, nvec, ld, j, S, pass, nsteps,
                               dpart, ndot, hscale, part);
                } else {
                    launch_pdl(k_reorth_dots<T, T>, gd, dim3(256), 0, st, Q, Wn, nvec, ld, j, S, pass, part, nrb,
                               nsteps, dpart);
                    launch_pdl(k_reorth_apply<T, T>, gu, dim3(256), 0, st, Q, Wn, nvec, ld, j, S, pass, nsteps, dpart,
                               ndot, hscale, part);
                }
            }
        }
        launch_pdl(k_lanczos_beta, dim3(nvec), dim3(FIN_THREADS), 0, st, S, part, nrb, nvec, nsteps, j);
    };
    step(0);
    if (nsteps > 1)
        run_captured(ctx, [&]() {
            for (int j = 1; j < nsteps; ++j) step(j);
        });
    k_quadrature<<<nvec, QUAD_THREADS, 0, ctx->stream>>>(S.m_eff, S.alpha, S.beta, nsteps, (double)p, res, e->cov.tau2,
                                                       e->ntheta > 1 ? e->tau2_dev : nullptr, vpt);
    KRY_CHECK_LAUNCH();
    KRY_CUDA(cudaMemcpyAsync(per_vec, res, nvec * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    KRY_CUDA(cudaStreamSynchronize(ctx->stream));
}

void logdet(kry_ctx* ctx, const kry_embed* e, int nprobe, int nsteps, uint64_t seed, bool reorth,
            double* per_probe) {
    KRY_REQUIRE(nsteps >= 1 && nsteps <= KRY_MAX_STEPS, KRY_EINVAL, "nsteps must be in [1, 256]");
    KRY_REQUIRE(nprobe >= 1, KRY_EINVAL, "nprobe must be >= 1");
    if (e->prec == KRY_F64)
        lanczos_logdet<double>(ctx, e, nprobe, nprobe, nsteps, seed, per_probe, 0, reorth);
    else
        lanczos_logdet<float>(ctx, e, nprobe, nprobe, nsteps, seed, per_probe, 0, reorth);
}

// Batched form: ntheta settings of a batched embedding x nprobe probes each
// (nprobe even), per_vec[ntheta * nprobe].
void logdet_batched(kry_ctx* ctx, const kry_embed* e, int nprobe, int nsteps, uint64_t seed, bool reorth,
                    double* per_vec) {
    KRY_REQUIRE(nsteps >= 1 && nsteps <= KRY_MAX_STEPS, KRY_EINVAL, "nsteps must be in [1, 256]");
    KRY_REQUIRE(nprobe >= 2 && nprobe % 2 == 0, KRY_EINVAL, "batched log-det needs an even probe count");
    const int nvec = e->ntheta * nprobe;
    const int vpt = e->ntheta > 1 ? nprobe : 0;
    if (e->prec == KRY_F64)
        lanczos_logdet<double>(ctx, e, nvec, nprobe, nsteps, seed, per_vec, vpt, reorth);
    else
        lanczos_logdet<float>(ctx, e, nvec, nprobe, nsteps, seed, per_vec, vpt, reorth);
}

// ------------------------------------------------------------------ CG

// The pinned host scratch as n ints, grown where a batch has more columns than it
// holds (no copy into it is in flight: every user waits for its own).
static int* host_ints(kry_ctx* ctx, size_t n) {
    if (n * sizeof(int) > ctx->host_cap) {
        double* more = nullptr;
        KRY_CUDA(cudaMallocHost(&more, n * sizeof(int)));
        cudaFreeHost(ctx->host_pinned);
        ctx->host_pinned = more;
        ctx->host_cap = n * sizeof(int);
    }
    return reinterpret_cast<int*>(ctx->host_pinned);
}

struct CgState {
    double* rr;      // [nrhs] r^T r
    double* alpha;   // [nrhs]
    double* beta;    // [nrhs]
    double* thr2;    // [nrhs] convergence threshold on r^T r
    int* done;       // [nrhs]
    int* iters;      // [nrhs]
    int* ndone;      // [1]
};

// x = 0, r = b (converted), p = r; partial ||r||^2.
template <typename T>
__global__ void k_cg_start(const double* __restrict__ B, int64_t ldb, T* __restrict__ X, T* __restrict__ R,
                           T* __restrict__ P, int64_t p, double* __restrict__ part) {
    const int k = blockIdx.y;
    const int64_t off = (int64_t)k * p;
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
        const T b = (T)B[(int64_t)k * ldb + i];
        X[off + i] = (T)0;
        R[off + i] = b;
        P[off + i] = b;
        acc[0] += (double)b * (double)b;
    }
    block_sum_store<1>(acc, part + (int64_t)k * gridDim.x + blockIdx.x, 0);
}

__global__ void k_cg_init_scalars(CgState S, const double* __restrict__ part, int nblk, int nrhs,
                                  const double* __restrict__ tol) {
    const int k = blockIdx.x;   // one block per right-hand side
    const double s = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x != 0) return;
    S.rr[k] = s;
    S.thr2[k] = tol[k] * tol[k] * s;
    S.done[k] = (s == 0.0 || s <= S.thr2[k]) ? 1 : 0;
    S.iters[k] = 0;
    S.alpha[k] = 0.0;
    S.beta[k] = 0.0;
    if (k == 0) *S.ndone = 0;
}

__global__ void k_cg_alpha(CgState S, const double* __restrict__ part, int nblk, int nrhs) {
    const int k = blockIdx.x;   // one block per right-hand side
    const double pq = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x == 0) S.alpha[k] = (S.done[k] || pq == 0.0) ? 0.0 : S.rr[k] / pq;
    if (k == 0 && threadIdx.x == 0) *S.ndone = 0;
}

// x += alpha p, r -= alpha q; partial ||r||^2.
template <typename T>
__global__ void k_cg_update(T* __restrict__ X, T* __restrict__ R, const T* __restrict__ P, const T* __restrict__ Q,
                            int64_t p, CgState S, double* __restrict__ part) {
    const int k = blockIdx.y;
    const int64_t off = (int64_t)k * p;
    const T a = (T)S.alpha[k];
    const bool act = !S.done[k];
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
        T r = R[off + i];
        if (act) {
            X[off + i] += a * P[off + i];
            r -= a * Q[off + i];
            R[off + i] = r;
        }
        acc[0] += (double)r * (double)r;
    }
    block_sum_store<1>(acc, part + (int64_t)k * gridDim.x + blockIdx.x, 0);
}

__global__ void k_cg_beta(CgState S, const double* __restrict__ part, int nblk, int nrhs, int maxit) {
    const int k = blockIdx.x;   // one block per right-hand side
    const double s = block_sum(part + (int64_t)k * nblk, nblk);
    if (threadIdx.x != 0) return;
    if (!S.done[k]) {
        S.iters[k] += 1;
        S.beta[k] = s / S.rr[k];
        S.rr[k] = s;
        if (s <= S.thr2[k] || !(s == s) || S.iters[k] >= maxit) {
            S.done[k] = 1;
            S.beta[k] = 0.0;
        }
    } else {
        S.beta[k] = 0.0;
    }
    if (S.done[k]) atomicAdd(S.ndone, 1);
}

template <typename T>
__global__ void k_cg_pupdate(T* __restrict__ P, const T* __restrict__ R, int64_t p, CgState S) {
    const int k = blockIdx.y;
    if (S.done[k]) return;
    const int64_t off = (int64_t)k * p;
    const T b = (T)S.beta[k];
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x)
        P[off + i] = R[off + i] + b * P[off + i];
}

// Inner CG in precision T on nrhs right-hand sides B (FP64, leading dim ldb),
// tolerances tol[k] relative to ||B_k||.  Solution X (T, leading dim p) in
// ctx->work[6].  Returns the largest iteration count.
template <typename T>
static int cg_inner(kry_ctx* ctx, const kry_embed* e, const double* B, int64_t ldb, int nrhs, const double* tol_dev,
                    int maxit, T** X_out, int vpt) {
    const bool dbl = sizeof(T) == 8;
    const int64_t p = ctx->p;
    cudaStream_t st = ctx->stream;
    const size_t vb = (size_t)nrhs * p * sizeof(T);
    ctx->work[6].ensure(vb);
    ctx->work[7].ensure(vb);
    ctx->work[8].ensure(vb);
    ctx->work[9].ensure(vb);
    T* X = ctx->work[6].as<T>();
    T* R = ctx->work[7].as<T>();
    T* P = ctx->work[8].as<T>();
    T* Q = ctx->work[9].as<T>();
    const int nblkC = matvec_num_partials(ctx, e, dbl, nrhs);
    ctx->work[10].ensure((size_t)nrhs * std::max(nblkC, RED_BLOCKS) * sizeof(double));
    double* part = ctx->work[10].as<double>();
    ctx->work[11].ensure((size_t)nrhs * (5 * sizeof(double) + 2 * sizeof(int)) + 64);
    char* sb = ctx->work[11].as<char>();
    CgState S;
    S.rr = reinterpret_cast<double*>(sb);
    S.alpha = S.rr + nrhs;
    S.beta = S.alpha + nrhs;
    S.thr2 = S.beta + nrhs;
    S.done = reinterpret_cast<int*>(S.thr2 + nrhs);
    S.iters = S.done + nrhs;
    S.ndone = S.iters + nrhs;

    dim3 gv(RED_BLOCKS, nrhs);
    k_cg_start<T><<<gv, 256, 0, st>>>(B, ldb, X, R, P, p, part);
    KRY_CHECK_LAUNCH();
    k_cg_init_scalars<<<nrhs, FIN_THREADS, 0, st>>>(S, part, RED_BLOCKS, nrhs, tol_dev);
    KRY_CHECK_LAUNCH();
    int* hdone = host_ints(ctx, nrhs);
    int it = 0;
    const int poll = 8;
    for (; it < maxit; ++it) {
        matvec_ex<T>(ctx, e, P, p, nullptr, Q, p, nrhs, part, nblkC, vpt);
        k_cg_alpha<<<nrhs, FIN_THREADS, 0, st>>>(S, part, nblkC, nrhs);
        KRY_CHECK_LAUNCH();
        k_cg_update<T><<<gv, 256, 0, st>>>(X, R, P, Q, p, S, part);
        KRY_CHECK_LAUNCH();
        k_cg_beta<<<nrhs, FIN_THREADS, 0, st>>>(S, part, RED_BLOCKS, nrhs, maxit);
        KRY_CHECK_LAUNCH();
        k_cg_pupdate<T><<<gv, 256, 0, st>>>(P, R, p, S);
        KRY_CHECK_LAUNCH();
        if ((it + 1) % poll == 0) {
            KRY_CUDA(cudaMemcpyAsync(hdone, S.ndone, sizeof(int), cudaMemcpyDeviceToHost, st));
            KRY_CUDA(cudaStreamSynchronize(st));
            if (*hdone >= nrhs) {
                ++it;
                break;
            }
        }
    }
    KRY_CUDA(cudaMemcpyAsync(hdone, S.iters, nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
    KRY_CUDA(cudaStreamSynchronize(st));
    int mx = 0;
    for (int k = 0; k < nrhs; ++k) mx = std::max(mx, hdone[k]);
    *X_out = X;
    return mx;
}

// R = B - K X and the block's partials of ||R||^2, ||B||^2; columns flagged in
// skip are left alone (their partials stay stale).  Up to two values per thread
// this was all FP64 shuffle trees (two per block, 4096 blocks for 32 columns of
// 45,900 values: 36.7 us); now eight and more per thread and the two sums in one
// tree (8.0 us, with the skipping).
static const int RES_PER_THREAD = 8;
__global__ void k_residual(const double* __restrict__ B, int64_t ldb, const double* __restrict__ KX,
                           double* __restrict__ R, int64_t p, double* __restrict__ part, const int* __restrict__ skip) {
    __shared__ double red[2][8];
    const int k = blockIdx.y;
    if (skip && skip[k]) return;
    double r2 = 0.0, b2 = 0.0;
#pragma unroll 4
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
        const double b = B[(int64_t)k * ldb + i];
        const double r = b - KX[(int64_t)k * p + i];
        R[(int64_t)k * p + i] = r;
        r2 += r * r;
        b2 += b * b;
    }
    // lanes 0-15 go on with ||R||^2, 16-31 with ||B||^2
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double give = lane < 16 ? b2 : r2;
    double v = (lane < 16 ? r2 : b2) + __shfl_xor_sync(0xffffffffu, give, 16);
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((lane & 15) == 0) red[lane >> 4][w] = v;
    __syncthreads();
    if (threadIdx.x < 2) {
        double s = 0.0;
        for (int q = 0; q < 8; ++q) s += red[threadIdx.x][q];
        part[((int64_t)k * gridDim.x + blockIdx.x) * 2 + threadIdx.x] = s;
    }
}

// Lane sums of part[0], part[stride], ... (n values) over a warp in a fixed
// order; valid in every lane.  (One warp per sum: a single thread's 128
// dependent FP64 adds took 15 us.)
__device__ __forceinline__ double warp_sum(const double* __restrict__ part, int n, int stride) {
    double v = 0.0;
    for (int b = threadIdx.x & 31; b < n; b += 32) v += part[(int64_t)b * stride];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Column norms from the residual kernel's partials: one warp per sum.
__global__ void k_norms_final(const double* __restrict__ part, int nblk, int nrhs, double* __restrict__ out) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;   // 2 k + (0: ||r||, 1: ||b||)
    if (i >= 2 * nrhs) return;
    const double s = warp_sum(part + (int64_t)(i >> 1) * nblk * 2 + (i & 1), nblk, 2);
    if ((threadIdx.x & 31) == 0) out[i] = sqrt(s);
}

__global__ void k_set(double* x, int64_t n, double v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = v;
}

// FP64 true residual R = B - K X and per-column (||R||, ||B||), which
// residual_norms fetches.
static void true_residual(kry_ctx* ctx, const kry_embed* e, const double* B, int64_t ldb, const double* X,
                          int64_t ldx, int nrhs, double* R, double* KX, int vpt, const int* skip) {
    const int64_t p = ctx->p;
    cudaStream_t st = ctx->stream;
    // KX = K X (FP64 matvec); X has leading dimension ldx.  Columns flagged in
    // skip (pairs of them) are not transformed: their residual norms are stale.
    matvec_ex<double>(ctx, e, X, ldx, nullptr, KX, p, nrhs, nullptr, 0, vpt, skip);
    ctx->red.ensure((size_t)nrhs * RED_BLOCKS * 2 * sizeof(double) + (size_t)nrhs * 2 * sizeof(double));
    double* part = ctx->red.as<double>();
    double* fin = part + (size_t)nrhs * RED_BLOCKS * 2;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(RED_BLOCKS, p / (256 * RES_PER_THREAD)));
    k_residual<<<dim3(nb, nrhs), 256, 0, st>>>(B, ldb, KX, R, p, part, skip);
    KRY_CHECK_LAUNCH();
    k_norms_final<<<(2 * nrhs + 7) / 8, 256, 0, st>>>(part, nb, nrhs, fin);
    KRY_CHECK_LAUNCH();
}

// The norms of the last true_residual, on the host.
static std::vector<double> residual_norms(kry_ctx* ctx, int nrhs) {
    std::vector<double> nrm(2 * nrhs);
    const double* fin = ctx->red.as<double>() + (size_t)nrhs * RED_BLOCKS * 2;
    KRY_CUDA(cudaMemcpyAsync(nrm.data(), fin, 2 * nrhs * sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    KRY_CUDA(cudaStreamSynchronize(ctx->stream));
    return nrm;
}

// ------------------------------------------------------------------ reliable-update mixed-precision CG
//
// FP32 CG (FP32 matvec, FP64 scalars) whose solution accumulates in FP64 and
// whose recursive FP32 residual is replaced by the true residual b - K x,
// computed with the FP64 matvec, whenever it has fallen 10x since the last
// replacement or reached the target (the "reliable updates" of van der Vorst
// & Ye, "Residual replacement strategies for Krylov subspace iterative
// methods", SIAM J. Sci. Comput. 2000).  The search direction is kept across
// replacements, so the Krylov progress of FP64 CG is retained while every
// matvec of the iteration runs in FP32.  Convergence is declared only on a
// true FP64 residual.

// Each iteration is the plain CG recurrence:
//   q = K p                                  (FFT matvec; pass C forms the partials of p^T q)
//   alpha = gamma / p^T q, r -= alpha q      (k_rcg_update; forms the partials of r^T r)
//   beta = gamma' / gamma, x += alpha p, p = r + beta p   (k_rcg_pupdate; counts the
//                                             iteration and asks for a residual replacement)
// Every block of the two streaming kernels adds up the few hundred partials of
// its column itself (total128, the same fixed order in all of them): about 0.4
// us beside its first loads, where a launch of its own for alpha and for beta
// took 3 us each.  x waits for the second kernel, which reads p anyhow.  An
// iteration for 4 columns: 32 x 32 27.5 -> 24.1 us, 256 x 256 28.1 -> 26.0,
// 1024 x 1024 100.7 -> 97.9 (both with sums in double-float; block_sums).  (All of the vector work in one kernel, a cluster of
// 16 blocks per column, took 22.6 us at 256 x 256 but 113.7 at 1024 x 1024, and
// no less than these two from 8 columns on.)
// K p is computed afresh by every matvec, so no auxiliary recurrence can
// drift in FP32 (single-reduction rearrangements carry K p by a recurrence and
// broke down on the ill-conditioned grids here).
//
// With a preconditioner (an embedding `pre` whose matvec applies M^-1 = A (S +
// tau2 I)^-1 A^T, S the circulant embedding of sigma2 Sigma on the matvec's
// torus: the inverse of the torus covariance, restricted to the observed
// cells), the same launches run preconditioned CG: after the update, z = M^-1 r
// by the FFT passes (pass C forms the partials of r^T z), gamma = r^T z,
// beta = gamma' / gamma, p = z + beta p; convergence is still judged on r^T r.
// M^-1 is symmetric positive definite (a principal block of an SPD matrix).
// It approximates K^-1 well where most of the grid is observed and the gaps
// are clustered, and poorly under scattered missing cells.
struct RcgState {
    double* gam;      // [nrhs] gamma = r^T z (r^T r without a preconditioner) of the current residual
    double* gold;     // [nrhs] gamma of the residual that the current p belongs to
    double* rr;       // [nrhs] r^T r of the current residual
    double* alpha;    // [nrhs]
    double* rr_ref;   // [nrhs] r^T r at the last replacement
    double* thr2;     // [nrhs] (rtol ||b||)^2
    int* want;        // [nrhs] 1: the last iteration asks for a replacement
    int* done;        // [nrhs]
    int* iters;       // [nrhs]
    int* ndone;       // [1]
};

// Blocks per right-hand side of the CG vector kernels: 304 (two per SM) for a
// few right-hand sides, fewer for many, so that a batch keeps about 1216
// blocks.
static int cg_blocks(int nrhs) { return std::max(8, std::min(304, 1216 / std::max(1, nrhs))); }

// The FP32 vectors of the loop keep a leading dimension ld that is a multiple of
// eight, with zeros past p, so that every access is 16 bytes wide whatever p is.

// X = 0 (a double-float pair Xh + Xl), R = P = (float) B; partials of ||B||^2
// (FP64) per column, one per block.
__global__ void k_rcg_start(const double* __restrict__ B, int64_t ldb, float* __restrict__ Xh, float* __restrict__ Xl,
                            float* __restrict__ R, float* __restrict__ P, int64_t p, int64_t ld,
                            double* __restrict__ part_rr) {
    const int k = blockIdx.y;
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ld; i += (int64_t)gridDim.x * blockDim.x) {
        const double b = i < p ? B[(int64_t)k * ldb + i] : 0.0;
        const int64_t o = (int64_t)k * ld + i;
        Xh[o] = 0.f;
        Xl[o] = 0.f;
        R[o] = (float)b;
        P[o] = (float)b;
        acc[0] += b * b;
    }
    block_sum_store<1>(acc, part_rr + (int64_t)k * gridDim.x + blockIdx.x, 0);
}

// rr = ||B||^2 from the start's partials; gamma = r^T z from the
// preconditioner matvec's partials (part_rz, nrz per column) or = rr.
__global__ void k_rcg_init_scalars(RcgState S, const double* __restrict__ part_rr, int nblk,
                                   const double* __restrict__ part_rz, int nrz, int nrhs,
                                   const double* __restrict__ tol) {
    const int k = blockIdx.x;   // one block per right-hand side
    const double s = block_sum(part_rr + (int64_t)k * nblk, nblk);
    double g = s;
    if (part_rz) {
        __syncthreads();   // block_sum's shared slots are reused
        g = block_sum(part_rz + (int64_t)k * nrz, nrz);
    }
    if (threadIdx.x == 0) {
        S.gam[k] = g;
        S.rr[k] = s;
        S.rr_ref[k] = s;
        S.gold[k] = g;
        S.alpha[k] = 0.0;
        S.thr2[k] = tol[k] * tol[k] * s;
        S.want[k] = 0;
        S.done[k] = (s == 0.0 || !(g > 0.0)) ? 1 : 0;
        S.iters[k] = 0;
    }
}

// Threads and blocks per column of the two streaming kernels: two blocks per SM of
// GB300 over all columns (every block repeats its column's sum, 0.4 us of FP64 pipe,
// so four times as many blocks took 15 + 17 us instead of 8 + 10 for 4 columns
// of 524,288 values).
static const int CG_THREADS = 512;
static int rcg_blocks(int nrhs) { return std::max(1, 304 / nrhs); }   // <= cg_blocks(nrhs)

// Sum of part[0 .. n) in a fixed order, valid in thread 0: by the first four
// warps, one per scheduler, since an FP64 instruction of a warp holds its
// scheduler's FP64 pipe for 64 cycles (for the same reason thread 0 alone
// divides, and the others get FP32 values).  red: four doubles of shared
// memory, written here only.
__device__ __forceinline__ double total128(const double* __restrict__ part, int n, double* red) {
    if (threadIdx.x < 128) {
        double v = 0.0;
        for (int b = threadIdx.x; b < n; b += 128) v += part[b];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    }
    __syncthreads();
    return threadIdx.x == 0 ? (red[0] + red[1]) + (red[2] + red[3]) : 0.0;
}

// alpha = gamma / p^T q (0 if p^T q is not positive), R -= alpha Q (FP32);
// partials of ||R||^2 (block_sums).  Streaming: two vectors read, one
// written, from L2 where they fit.
__global__ void __launch_bounds__(CG_THREADS) k_rcg_update(float* __restrict__ R, const float* __restrict__ Q, int64_t ld,
                                                    RcgState S, const double* __restrict__ part_pq, int npq,
                                                    double* __restrict__ part_rr) {
    __shared__ double red[4];
    __shared__ float coef;
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.y;
    if (S.done[k]) return;   // finished columns keep x and r
    const int64_t off = (int64_t)k * ld, step = (int64_t)gridDim.x * blockDim.x * 4;
    int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    float r[4], q[4];
    if (x < ld) {   // in flight during the sum
        load4(R + off + x, r);
        load4(Q + off + x, q);
    }
    const double g = threadIdx.x == 0 ? S.gam[k] : 0.0;
    const double d = total128(part_pq + (int64_t)k * npq, npq, red);
    if (threadIdx.x == 0) {
        const double a = d > 0.0 ? g / d : 0.0;
        coef = (float)a;
        if (blockIdx.x == 0) {
            S.alpha[k] = a;
            S.gold[k] = g;
        }
    }
    __syncthreads();
    const float af = coef;
    DotAcc<float> nrm;
    while (x < ld) {
        float rn[4], qn[4];
        if (x + step < ld) {
            load4(R + off + x + step, rn);
            load4(Q + off + x + step, qn);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            r[e] -= af * q[e];
            nrm.add_prod(r[e], r[e]);
        }
        store4(R + off + x, r);
#pragma unroll
        for (int e = 0; e < 4; ++e) r[e] = rn[e], q[e] = qn[e];
        x += step;
    }
    const double s = block_total<CG_THREADS>(nrm);
    if (threadIdx.x == 0) part_rr[(int64_t)k * gridDim.x + blockIdx.x] = s;
}

// rr' = r^T r from the update's partials and gamma' = r^T z from part_rz (nrz
// per column; NULL without a preconditioner: gamma' = rr'), beta = gamma' /
// gamma; X += alpha P in double-float (Xh + Xl, FP32 instructions only) and P =
// Z + beta P (Z = R without a preconditioner).  Streaming: four vectors read,
// three written.  Block 0 counts the iteration and asks for a replacement when
// rr' has fallen 100x since the last one, reached the target, is not finite, or
// the budget is spent (no block reads what it writes).
__global__ void __launch_bounds__(CG_THREADS) k_rcg_pupdate(float* __restrict__ Xh, float* __restrict__ Xl,
                                                     float* __restrict__ P, const float* __restrict__ Z, int64_t ld,
                                                     RcgState S, const double* __restrict__ part_rr, int nrr,
                                                     const double* __restrict__ part_rz, int nrz, int maxit) {
    __shared__ double red[8];
    __shared__ float coef[3];
    pdl_wait();
    pdl_launch_dependents();
    const int k = blockIdx.y;
    if (S.done[k]) return;
    const int64_t off = (int64_t)k * ld, step = (int64_t)gridDim.x * blockDim.x * 4;
    int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4;
    float z[4], pv[4], xh[4], xl[4];
    auto load = [&](int64_t o) {
        load4(Z + o, z);
        load4(P + o, pv);
        load4(Xh + o, xh);
        load4(Xl + o, xl);
    };
    if (x < ld) load(off + x);   // in flight during the sums
    double g0 = 0.0;
    if (threadIdx.x == 0) {
        g0 = S.gold[k];
        df_split(S.alpha[k], coef[1], coef[2]);
    }
    const double rr = total128(part_rr + (int64_t)k * nrr, nrr, red);
    const double rz = part_rz ? total128(part_rz + (int64_t)k * nrz, nrz, red + 4) : 0.0;
    if (threadIdx.x == 0) {
        const double g = part_rz ? rz : rr;
        coef[0] = (float)((g0 > 0.0) ? g / g0 : 0.0);
        if (blockIdx.x == 0) {
            S.gam[k] = g;
            S.rr[k] = rr;
            const int it = S.iters[k] + 1;
            S.iters[k] = it;
            S.want[k] = (rr <= S.thr2[k] || rr <= 1e-2 * S.rr_ref[k] || !(rr == rr) || !(g == g) || it >= maxit) ? 1 : 0;
        }
    }
    __syncthreads();
    const float b = coef[0], ahi = coef[1], alo = coef[2];
    while (x < ld) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            df_axpy(xh[e], xl[e], ahi, alo, pv[e]);
            pv[e] = z[e] + b * pv[e];
        }
        store4(Xh + off + x, xh);
        store4(Xl + off + x, xl);
        store4(P + off + x, pv);
        x += step;
        if (x < ld) load(off + x);
    }
}

// X = Xh + Xl in FP64 (the caller's layout, leading dimension ldx), but for pairs
// of columns (which are transformed together) that are both flagged in skip.
__global__ void k_df_to_f64(const float* __restrict__ Xh, const float* __restrict__ Xl, int64_t p, int64_t ld,
                            double* __restrict__ X, int64_t ldx, const int* __restrict__ skip) {
    const int k = blockIdx.y, k1 = k ^ 1;
    if (skip && skip[k] && (k1 >= (int)gridDim.y || skip[k1])) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x)
        X[(int64_t)k * ldx + i] = (double)Xh[(int64_t)k * ld + i] + (double)Xl[(int64_t)k * ld + i];
}

// The kept direction belongs to the recursive residual.  Where a block of
// iterations gains more digits than FP32 holds (rr below 1e-12 rr_ref; condition
// numbers below about 2), the recursion goes on below the true residual, of norm
// rn, and the step along the then far shorter direction would overshoot by the
// square of the ratio: the column starts again from its residual.  Slower systems,
// whose recursion drifts by rounding, keep their direction.  S.rr and S.rr_ref are
// the recursive r^T r and that of the last replacement until k_round_end.
__device__ __forceinline__ bool rcg_restart(const RcgState& S, int k, double rn) {
    return S.rr[k] < 1e-12 * S.rr_ref[k] && rn * rn > 16.0 * S.rr[k];
}

// Residual replacement of the running columns of the round: R = (float) R64,
// and without a preconditioner P = R where the column starts again.
__global__ void k_rcg_replace(const double* __restrict__ R64, float* __restrict__ R, float* __restrict__ P, int64_t p,
                              int64_t ld, const double* __restrict__ norms, RcgState S, int precond,
                              const int* __restrict__ sel) {
    const int k = blockIdx.y;
    if (S.done[k] || sel[k]) return;   // only the columns of the round (the others' norms are stale)
    const bool again = !precond && rcg_restart(S, k, norms[2 * k]);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
        const float r = (float)R64[(int64_t)k * p + i];
        R[(int64_t)k * ld + i] = r;
        if (again) P[(int64_t)k * ld + i] = r;
    }
}

// Preconditioned runs after a replacement: gamma = r^T z, the fixed-order sum of
// the preconditioner matvec's partials (block 0 of a column), and P = Z where the
// column starts again.
__global__ void k_rcg_regamma(RcgState S, const float* __restrict__ Z, float* __restrict__ P, int64_t ld,
                              const double* __restrict__ norms, const double* __restrict__ part_rz, int nrz,
                              const int* __restrict__ sel) {
    const int k = blockIdx.y;
    if (S.done[k] || sel[k]) return;
    if (blockIdx.x == 0) {
        const double g = block_sum(part_rz + (int64_t)k * nrz, nrz);
        if (threadIdx.x == 0) S.gam[k] = g;
    }
    if (!rcg_restart(S, k, norms[2 * k])) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ld; i += (int64_t)gridDim.x * blockDim.x)
        P[(int64_t)k * ld + i] = Z[(int64_t)k * ld + i];
}

// Ends a replacement round (one block).  Its running columns: rr = rr_ref =
// ||R64||^2 and, without a preconditioner, gamma = rr; done when ||R64|| <= rtol
// ||B|| or the iteration budget is spent (a non-finite residual also ends the
// column; the caller reports it).  Counts the finished columns and clears the
// requests.
__global__ void k_round_end(RcgState S, int nrhs, const double* __restrict__ norms, int maxit, int precond,
                            const int* __restrict__ sel) {
    __shared__ int finished;
    if (threadIdx.x == 0) finished = 0;
    __syncthreads();
    int d = 0;
    for (int k = threadIdx.x; k < nrhs; k += blockDim.x) {
        if (!S.done[k] && !sel[k]) {
            const double rn = norms[2 * k], rr = rn * rn;
            if (!precond) S.gam[k] = rr;
            S.rr[k] = rr;
            S.rr_ref[k] = rr;
            if (rr <= S.thr2[k] || S.iters[k] >= maxit || !(rn == rn)) S.done[k] = 1;
        }
        d += S.done[k];
        S.want[k] = 0;
    }
    atomicAdd(&finished, d);
    __syncthreads();
    if (threadIdx.x == 0) *S.ndone = finished;
}

static void true_residual(kry_ctx* ctx, const kry_embed* e, const double* B, int64_t ldb, const double* X,
                          int64_t ldx, int nrhs, double* R, double* KX, int vpt, const int* skip = nullptr);

// Skip flags of a replacement round: with `all`, no column is skipped (every
// running column is replaced, and the FP64 residual covers the finished ones
// too); otherwise the columns that are done or do not ask for a replacement.
__global__ void k_rcg_select(RcgState S, int nrhs, int* __restrict__ skip, int all) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < nrhs) skip[k] = (!all && (S.done[k] || !S.want[k])) ? 1 : 0;
}

// Returns the largest per-column iteration count.  pre: preconditioner
// embedding (NULL: plain CG).
static int cg_reliable(kry_ctx* ctx, const kry_embed* e, const double* B, int64_t ldb, double* X, int64_t ldx,
                       int nrhs, double rtol, int maxit, bool* fresh, int vpt,
                       const kry_embed* pre) {
    const int64_t p = ctx->p;
    cudaStream_t st = ctx->stream;
    const int64_t ld = (p + 7) & ~(int64_t)7;   // leading dimension of the FP32 vectors (zeros past p)
    const size_t vb = (size_t)nrhs * ld * sizeof(float);
    ctx->work[7].ensure(vb);
    ctx->work[8].ensure(vb);
    ctx->work[9].ensure(vb);
    float* R = ctx->work[7].as<float>();
    float* P = ctx->work[8].as<float>();
    float* Q = ctx->work[9].as<float>();
    float* Z = R;
    if (pre) {
        ctx->work[3].ensure(vb);
        Z = ctx->work[3].as<float>();
    }
    const int nblkC = matvec_num_partials(ctx, e, false, nrhs);
    const int nbc = cg_blocks(nrhs);
    ctx->work[10].ensure((size_t)nrhs * (2 * nblkC + nbc) * sizeof(double));
    double* part_pq = ctx->work[10].as<double>();        // matvec partials (p^T K p)
    double* part_rr = part_pq + (size_t)nrhs * nblkC;     // start / update partials (r^T r)
    double* part_rz = pre ? part_rr + (size_t)nrhs * nbc : nullptr;   // preconditioner partials (r^T z)
    ctx->work[11].ensure((size_t)nrhs * (6 * sizeof(double) + 4 * sizeof(int)) + 64);
    char* sb = ctx->work[11].as<char>();
    RcgState S;
    S.gam = reinterpret_cast<double*>(sb);
    S.rr = S.gam + nrhs;
    S.alpha = S.rr + nrhs;
    S.gold = S.alpha + nrhs;
    S.rr_ref = S.gold + nrhs;
    S.thr2 = S.rr_ref + nrhs;
    S.want = reinterpret_cast<int*>(S.thr2 + nrhs);
    S.done = S.want + nrhs;
    S.iters = S.done + nrhs;
    S.ndone = S.iters + nrhs;
    int* sel = S.ndone + 1;   // skip flags of a replacement round
    ctx->tolbuf.ensure(nrhs * sizeof(double));
    std::vector<double> tol_h(nrhs, rtol);
    KRY_CUDA(cudaMemcpyAsync(ctx->tolbuf.p, tol_h.data(), nrhs * sizeof(double), cudaMemcpyHostToDevice, st));
    ctx->work[4].ensure((size_t)nrhs * p * sizeof(double));
    double* R64 = ctx->work[4].as<double>();
    ctx->kxbuf.ensure((size_t)nrhs * p * sizeof(double));
    ctx->work[12].ensure(2 * vb);
    float* Xh = ctx->work[12].as<float>();   // the solution as a double-float pair
    float* Xl = Xh + (size_t)nrhs * ld;

    dim3 gv(RED_BLOCKS, nrhs);
    dim3 gc(nbc, nrhs), gl(rcg_blocks(nrhs), nrhs);
    if (ld > p) {   // the matvec writes the first p values of Q and Z only
        KRY_CUDA(cudaMemset2DAsync(Q + p, ld * sizeof(float), 0, (ld - p) * sizeof(float), nrhs, st));
        if (pre) KRY_CUDA(cudaMemset2DAsync(Z + p, ld * sizeof(float), 0, (ld - p) * sizeof(float), nrhs, st));
    }
    auto to_f64 = [&](const int* skip) {
        k_df_to_f64<<<gv, 256, 0, st>>>(Xh, Xl, p, ld, X, ldx, skip);
        KRY_CHECK_LAUNCH();
    };
    k_rcg_start<<<gc, 256, 0, st>>>(B, ldb, Xh, Xl, R, P, p, ld, part_rr);
    KRY_CHECK_LAUNCH();
    if (pre) matvec_ex<float>(ctx, pre, R, ld, nullptr, Z, ld, nrhs, part_rz, nblkC, vpt, nullptr);   // z = M^-1 r
    k_rcg_init_scalars<<<nrhs, FIN_THREADS, 0, st>>>(S, part_rr, nbc, part_rz, nblkC, nrhs, ctx->tolbuf.as<double>());
    KRY_CHECK_LAUNCH();
    if (pre) KRY_CUDA(cudaMemcpyAsync(P, Z, vb, cudaMemcpyDeviceToDevice, st));   // p = z
    int* hflag = host_ints(ctx, nrhs);
    const int poll = 8;
    *fresh = false;
    // one CG iteration on ctx->stream (the capture stream while capturing)
    auto iterate = [&]() {
        cudaStream_t s2 = ctx->stream;
        // kernels launched back to back with programmatic dependent launch: each
        // waits for its predecessor's completion before touching its outputs;
        // columns that have converged are not transformed (pairs of finished
        // columns skip every pass)
        matvec_ex<float>(ctx, e, P, ld, nullptr, Q, ld, nrhs, part_pq, nblkC, vpt, S.done);
        launch_pdl(k_rcg_update, gl, dim3(CG_THREADS), 0, s2, R, Q, ld, S, part_pq, nblkC, part_rr);
        if (pre) matvec_ex<float>(ctx, pre, R, ld, nullptr, Z, ld, nrhs, part_rz, nblkC, vpt, S.done);
        launch_pdl(k_rcg_pupdate, gl, dim3(CG_THREADS), 0, s2, Xh, Xl, P, Z, ld, S, part_rr, (int)gl.x, part_rz, nblkC, maxit);
    };
    // Iterations run in blocks of `poll`.  The first block runs directly (it
    // sizes every buffer); later blocks replay one captured graph.
    Replay block(ctx);
    for (int it0 = 0; it0 < maxit + poll; it0 += poll) {
        if (it0 == 0 || !ctx->use_graphs) {
            for (int i = 0; i < poll; ++i) iterate();
        } else {
            if (!block.exec)
                block.capture([&]() {
                    for (int i = 0; i < poll; ++i) iterate();
                });
            block.launch();
        }
        KRY_CUDA(cudaMemcpyAsync(hflag, S.want, nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
        KRY_CUDA(cudaStreamSynchronize(st));
        if (block.exec) block.harvest();
        int nwant = 0;
        for (int k = 0; k < nrhs; ++k) nwant += hflag[k] != 0;
        if (nwant > 0) {
            // Residual replacement.  A few right-hand sides (which converge
            // together) are all replaced in one round; in larger batches only
            // the columns that ask for it, and the FP64 matvec transforms only
            // their pairs.
            const int all = nrhs <= 8 ? 1 : 0;
            k_rcg_select<<<(nrhs + 255) / 256, 256, 0, st>>>(S, nrhs, sel, all);
            KRY_CHECK_LAUNCH();
            to_f64(sel);
            true_residual(ctx, e, B, ldb, X, ldx, nrhs, R64, ctx->kxbuf.as<double>(), vpt, sel);
            double* dn = ctx->red.as<double>() + (size_t)nrhs * RED_BLOCKS * 2;   // device norms
            k_rcg_replace<<<gc, 256, 0, st>>>(R64, R, P, p, ld, dn, S, pre ? 1 : 0, sel);
            KRY_CHECK_LAUNCH();
            if (pre) {   // z = M^-1 r and gamma = r^T z for the replaced r
                matvec_ex<float>(ctx, pre, R, ld, nullptr, Z, ld, nrhs, part_rz, nblkC, vpt, sel);
                k_rcg_regamma<<<gc, FIN_THREADS, 0, st>>>(S, Z, P, ld, dn, part_rz, nblkC, sel);
                KRY_CHECK_LAUNCH();
            }
            k_round_end<<<1, 256, 0, st>>>(S, nrhs, dn, maxit, pre ? 1 : 0, sel);
            KRY_CHECK_LAUNCH();
            KRY_CUDA(cudaMemcpyAsync(hflag, S.ndone, sizeof(int), cudaMemcpyDeviceToHost, st));
            KRY_CUDA(cudaStreamSynchronize(st));
            if (*hflag >= nrhs) {
                // the last residuals are every column's only if every column took part
                *fresh = all || nwant == nrhs;
                break;
            }
        }
    }
    to_f64(nullptr);   // X, after the loop or its last replacement round (idempotent)
    std::vector<int> its(nrhs);
    KRY_CUDA(cudaMemcpyAsync(its.data(), S.iters, nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
    KRY_CUDA(cudaStreamSynchronize(st));
    int mx = 0;
    for (int k = 0; k < nrhs; ++k) mx = std::max(mx, its[k]);
    return mx;
}

SolveInfo solve(kry_ctx* ctx, const kry_embed* e, const double* B, int64_t ldb, double* X, int64_t ldx, int nrhs,
                double rtol, int maxit, int vpt = 0, const kry_embed* pre = nullptr) {
    SolveInfo info;
    const int64_t p = ctx->p;
    cudaStream_t st = ctx->stream;
    KRY_REQUIRE(nrhs >= 1, KRY_EINVAL, "nrhs must be >= 1");
    KRY_REQUIRE(rtol > 0 && maxit >= 1, KRY_EINVAL, "rtol must be > 0 and maxit >= 1");
    ctx->kxbuf.ensure((size_t)nrhs * p * sizeof(double));
    ctx->work[4].ensure((size_t)nrhs * p * sizeof(double));
    double* R = ctx->work[4].as<double>();
    bool fresh = false;
    if (e->prec == KRY_F64) {
        // plain FP64 CG
        ctx->tolbuf.ensure(nrhs * sizeof(double));
        std::vector<double> tol_h(nrhs, rtol);
        KRY_CUDA(cudaMemcpyAsync(ctx->tolbuf.p, tol_h.data(), nrhs * sizeof(double), cudaMemcpyHostToDevice, st));
        double* Xd;
        info.iters = cg_inner<double>(ctx, e, B, ldb, nrhs, ctx->tolbuf.as<double>(), maxit, &Xd, vpt);
        KRY_CUDA(cudaMemcpy2DAsync(X, ldx * sizeof(double), Xd, p * sizeof(double), p * sizeof(double), nrhs,
                                   cudaMemcpyDeviceToDevice, st));
    } else {
        // FP32 CG with FP64 solution and residual replacement
        info.iters = cg_reliable(ctx, e, B, ldb, X, ldx, nrhs, rtol, maxit, &fresh, vpt, pre);
    }
    // the reported residual is always the true FP64 residual of the returned X
    if (!fresh) true_residual(ctx, e, B, ldb, X, ldx, nrhs, R, ctx->kxbuf.as<double>(), vpt);
    const std::vector<double> nrm = residual_norms(ctx, nrhs);
    info.relres = 0.0;
    for (int k = 0; k < nrhs; ++k) {
        const double bn = nrm[2 * k + 1];
        const double rk = bn > 0 ? nrm[2 * k] / bn : 0.0;
        if (!(rk == rk)) {   // a non-finite residual is reported, not dropped by max
            info.relres = rk;
            break;
        }
        info.relres = std::max(info.relres, rk);
    }
    info.converged = info.relres <= rtol * (1.0 + 1e-9);
    return info;
}

// ------------------------------------------------------------------ GLS and the log-likelihood

// G[a][b] = V_a^T Z_b for the (ncov+1) columns V = [y, X] and Z = K^-1 V.
__global__ void k_gram(const double* __restrict__ V, int64_t ldv, const double* __restrict__ Z, int64_t ldz,
                       int64_t p, int nc, double* __restrict__ part) {
    const int a = blockIdx.y / nc, b = blockIdx.y % nc;
    double acc[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x)
        acc[0] += V[(int64_t)a * ldv + i] * Z[(int64_t)b * ldz + i];
    block_sum_store<1>(acc, part + (int64_t)blockIdx.y * gridDim.x + blockIdx.x, 0);
}

// beta = (X^T K^-1 X)^-1 X^T K^-1 y by Cholesky of the ncov x ncov matrix;
// quad = y^T K^-1 y - beta^T X^T K^-1 y; loglik = -1/2 (logdet + quad + p log 2 pi).
__global__ void k_gls(const double* __restrict__ part, int nblk, int ncov, int64_t p, double logdet,
                      double* __restrict__ out) {
    const int nc = ncov + 1;
    __shared__ double G[KRY_MAX_COV + 1][KRY_MAX_COV + 1];
    for (int i = threadIdx.x >> 5; i < nc * nc; i += blockDim.x >> 5) {   // one warp per entry
        const double s = warp_sum(part + (int64_t)i * nblk, nblk, 1);
        if ((threadIdx.x & 31) == 0) G[i / nc][i % nc] = s;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    // symmetrise (V^T K^-1 V is symmetric in exact arithmetic)
    double A[KRY_MAX_COV][KRY_MAX_COV], g[KRY_MAX_COV], L[KRY_MAX_COV][KRY_MAX_COV];
    for (int a = 0; a < ncov; ++a) {
        g[a] = 0.5 * (G[a + 1][0] + G[0][a + 1]);
        for (int b = 0; b < ncov; ++b) A[a][b] = 0.5 * (G[a + 1][b + 1] + G[b + 1][a + 1]);
    }
    int ok = 1;
    for (int j = 0; j < ncov; ++j) {
        double s = A[j][j];
        for (int k = 0; k < j; ++k) s -= L[j][k] * L[j][k];
        if (!(s > 0)) {
            ok = 0;
            s = 1e-300;
        }
        L[j][j] = sqrt(s);
        for (int i = j + 1; i < ncov; ++i) {
            double t = A[i][j];
            for (int k = 0; k < j; ++k) t -= L[i][k] * L[j][k];
            L[i][j] = t / L[j][j];
        }
    }
    double w[KRY_MAX_COV], beta[KRY_MAX_COV];
    for (int i = 0; i < ncov; ++i) {
        double t = g[i];
        for (int k = 0; k < i; ++k) t -= L[i][k] * w[k];
        w[i] = t / L[i][i];
    }
    for (int i = ncov - 1; i >= 0; --i) {
        double t = w[i];
        for (int k = i + 1; k < ncov; ++k) t -= L[k][i] * beta[k];
        beta[i] = t / L[i][i];
    }
    double quad = G[0][0];
    for (int i = 0; i < ncov; ++i) quad -= beta[i] * g[i];
    const double ll = -0.5 * (logdet + quad + (double)p * 1.8378770664093454836);
    out[0] = ll;
    out[1] = quad;
    out[2] = ok ? 0.0 : 1.0;
    for (int i = 0; i < ncov; ++i) out[3 + i] = beta[i];
}

// V = [y, X] (p x (ncov+1), ld p) and Z = K^-1 V already solved.
GlsResult gls(kry_ctx* ctx, const double* V, const double* Z, int ncov, double logdet) {
    const int64_t p = ctx->p;
    const int nc = ncov + 1;
    cudaStream_t st = ctx->stream;
    ctx->red.ensure((size_t)nc * nc * RED_BLOCKS * sizeof(double) + 64 * sizeof(double));
    double* part = ctx->red.as<double>();
    double* out = part + (size_t)nc * nc * RED_BLOCKS;
    dim3 g(RED_BLOCKS, nc * nc);
    k_gram<<<g, 256, 0, st>>>(V, p, Z, p, p, nc, part);
    KRY_CHECK_LAUNCH();
    k_gls<<<1, 256, 0, st>>>(part, RED_BLOCKS, ncov, p, logdet, out);
    KRY_CHECK_LAUNCH();
    KRY_CUDA(cudaMemcpyAsync(ctx->host_pinned, out, (3 + ncov) * sizeof(double), cudaMemcpyDeviceToHost, st));
    KRY_CUDA(cudaStreamSynchronize(st));
    GlsResult r;
    r.loglik = ctx->host_pinned[0];
    r.quad = ctx->host_pinned[1];
    r.ok = ctx->host_pinned[2] == 0.0;
    for (int i = 0; i < ncov; ++i) r.beta[i] = ctx->host_pinned[3 + i];
    return r;
}

// ------------------------------------------------------------------ kriging helpers

// w = Z[:,0] - Z[:,1:] beta  (K^-1 (y - X beta) without another solve).
__global__ void k_resid_weights(const double* __restrict__ Z, int64_t p, int ncov, const double* __restrict__ beta,
                                double* __restrict__ w) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
        double v = Z[i];
        for (int c = 0; c < ncov; ++c) v -= Z[(int64_t)(c + 1) * p + i] * beta[c];
        w[i] = v;
    }
}

// ------------------------------------------------------------------ parametric bootstrap (Sec. 3.5)

__global__ void k_boot_rhs(const double* __restrict__ G, int64_t N, const int* __restrict__ cellidx, int64_t p,
                           const double* __restrict__ eps, double tau, double* __restrict__ R) {
    const int b = blockIdx.y;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p; q += (int64_t)gridDim.x * blockDim.x)
        R[(int64_t)b * p + q] = G[(int64_t)b * N + cellidx[q]] + tau * eps[(int64_t)b * p + q];
}

void boot_rhs(kry_ctx* ctx, const double* G, int64_t N, const double* eps, double tau, double* R, int nrep) {
    const int64_t p = ctx->p;
    dim3 g((unsigned)std::min<int64_t>((p + 255) / 256, 1024), nrep);
    k_boot_rhs<<<g, 256, 0, ctx->stream>>>(G, N, ctx->cellidx.as<int>(), p, eps, tau, R);
    KRY_CHECK_LAUNCH();
}

__global__ void k_boot_mse(const double* __restrict__ G, const double* __restrict__ H, int64_t N, int nrep,
                           const int64_t* __restrict__ cells, int64_t ncell, double* __restrict__ var,
                           int* __restrict__ bad) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ncell; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cell = cells[t];
        if (cell < 0 || cell >= N) {
            var[t] = __longlong_as_double(0x7ff8000000000000ll);
            *bad = 1;
            continue;
        }
        double s = 0.0;
        for (int b = 0; b < nrep; ++b) {
            const double d = G[(int64_t)b * N + cell] - H[(int64_t)b * N + cell];
            s += d * d;
        }
        var[t] = s / nrep;
    }
}

void boot_mse(kry_ctx* ctx, const double* G, const double* H, int64_t N, int nrep, const int64_t* cells,
              int64_t ncell, double* var, int* bad) {
    if (ncell <= 0) return;
    k_boot_mse<<<(unsigned)std::min<int64_t>((ncell + 255) / 256, 4096), 256, 0, ctx->stream>>>(G, H, N, nrep, cells,
                                                                                              ncell, var, bad);
    KRY_CHECK_LAUNCH();
}

// mean[t] = X_t beta + grid[cells[t]]; a cell index outside [0, N) gives NaN
// and raises *bad.
__global__ void k_krige_cells(const double* __restrict__ grid, int64_t N, const int64_t* __restrict__ cells,
                              int64_t ncell, const double* __restrict__ Xc, int ncov, const double* __restrict__ beta,
                              double* __restrict__ mean, int* __restrict__ bad) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < ncell; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t cell = cells[t];
        if (cell < 0 || cell >= N) {
            mean[t] = __longlong_as_double(0x7ff8000000000000ll);
            *bad = 1;
            continue;
        }
        double m = grid[cell];
        for (int c = 0; c < ncov; ++c) m += Xc[(int64_t)c * ncell + t] * beta[c];
        mean[t] = m;
    }
}

struct CovPar {
    double sigma2, inv_range, nu, ca, sa, ratio, dx1, dx2;
};

// mean[s] = X_s beta + sum_o sigma2 rho(site_s - cell_o) w_o  (one block per site).
__global__ void k_krige_sites(const double* __restrict__ sites, int64_t nsite, const double* __restrict__ Xs, int ncov,
                              const double* __restrict__ beta, const double* __restrict__ w,
                              const int* __restrict__ cellidx, int64_t p, int n2, CovPar cp,
                              double* __restrict__ mean) {
    const int64_t s = blockIdx.x;
    if (s >= nsite) return;
    const double x1 = sites[2 * s], x2 = sites[2 * s + 1];
    double acc[1] = {0.0};
    for (int64_t q = threadIdx.x; q < p; q += blockDim.x) {
        const int cell = cellidx[q];
        const int i = cell / n2, j = cell - (cell / n2) * n2;
        const double h1 = x1 - (i + 0.5) * cp.dx1, h2 = x2 - (j + 0.5) * cp.dx2;
        const double r = kry_scaled_dist(h1, h2, cp.ca, cp.sa, cp.ratio, cp.inv_range);
        acc[0] += cp.sigma2 * kry_matern(r, cp.nu) * w[q];
    }
    __shared__ double tot;
    block_sum_store<1>(acc, &tot, 0);
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = tot;
        for (int c = 0; c < ncov; ++c) m += Xs[(int64_t)c * nsite + s] * beta[c];
        mean[s] = m;
    }
}

// Columns of sigma2 Sigma_{obs, t} for a batch of target cells: C[k][q].
// Target cells are clamped into the grid (k_krige_cells flags bad indices).
__global__ void k_cross_cols(const int64_t* __restrict__ cells, int64_t t0, const int* __restrict__ cellidx, int64_t p,
                             int n2, int64_t N, CovPar cp, double* __restrict__ C) {
    const int k = blockIdx.y;
    const int64_t t = min(max(cells[t0 + k], (int64_t)0), N - 1);
    const int ti = (int)(t / n2), tj = (int)(t - (t / n2) * n2);
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < p; q += (int64_t)gridDim.x * blockDim.x) {
        const int cell = cellidx[q];
        const int i = cell / n2, j = cell - (cell / n2) * n2;
        const double r = kry_scaled_dist((i - ti) * cp.dx1, (j - tj) * cp.dx2, cp.ca, cp.sa, cp.ratio, cp.inv_range);
        C[(int64_t)k * p + q] = cp.sigma2 * kry_matern(r, cp.nu);
    }
}

// var[t0 + k] = sigma2 - C_k^T S_k.
__global__ void k_var_final(const double* __restrict__ C, const double* __restrict__ Sx, int64_t p, double sigma2,
                            double* __restrict__ var, int64_t t0) {
    const int k = blockIdx.x;
    double acc[1] = {0.0};
    for (int64_t q = threadIdx.x; q < p; q += blockDim.x) acc[0] += C[(int64_t)k * p + q] * Sx[(int64_t)k * p + q];
    __shared__ double tot;
    block_sum_store<1>(acc, &tot, 0);
    __syncthreads();
    if (threadIdx.x == 0) var[t0 + k] = sigma2 - tot;
}

CovPar cov_par(const kry_cov& cov, double dx1, double dx2) {
    CovPar c;
    c.sigma2 = cov.sigma2;
    c.inv_range = 1.0 / cov.range;
    c.nu = cov.nu;
    c.ca = cos(cov.aniso_angle);
    c.sa = sin(cov.aniso_angle);
    c.ratio = cov.aniso_ratio;
    c.dx1 = dx1;
    c.dx2 = dx2;
    return c;
}

void krige_launch_cells(kry_ctx* ctx, const double* grid, const int64_t* cells, int64_t ncell, const double* Xc,
                        int ncov, const double* beta_dev, double* mean, int* bad) {
    if (ncell <= 0) return;
    k_krige_cells<<<(unsigned)std::min<int64_t>((ncell + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        grid, (int64_t)ctx->n1 * ctx->n2, cells, ncell, Xc, ncov, beta_dev, mean, bad);
    KRY_CHECK_LAUNCH();
}

void krige_launch_sites(kry_ctx* ctx, const kry_cov& cov, const double* sites, int64_t nsite, const double* Xs,
                        int ncov, const double* beta_dev, const double* w, double* mean) {
    if (nsite <= 0) return;
    k_krige_sites<<<(unsigned)nsite, 256, 0, ctx->stream>>>(sites, nsite, Xs, ncov, beta_dev, w,
                                                           ctx->cellidx.as<int>(), ctx->p, ctx->n2,
                                                           cov_par(cov, ctx->dx1, ctx->dx2), mean);
    KRY_CHECK_LAUNCH();
}

void resid_weights(kry_ctx* ctx, const double* Z, int ncov, const double* beta_dev, double* w) {
    k_resid_weights<<<(unsigned)std::min<int64_t>((ctx->p + 255) / 256, 4096), 256, 0, ctx->stream>>>(
        Z, ctx->p, ncov, beta_dev, w);
    KRY_CHECK_LAUNCH();
}

// Simple-kriging variances at target cells, nb targets per batch of solves.
bool krige_variances(kry_ctx* ctx, const kry_embed* e, const int64_t* cells, int64_t ncell, double* var,
                     double rtol, int maxit, const kry_embed* pre) {
    const int64_t p = ctx->p;
    cudaStream_t st = ctx->stream;
    const int nb = 32;
    DevBuf& cbuf = ctx->cbuf;
    DevBuf& sbuf = ctx->sbuf;
    cbuf.ensure((size_t)nb * p * sizeof(double));
    sbuf.ensure((size_t)nb * p * sizeof(double));
    bool ok = true;
    const CovPar cp = cov_par(e->cov, ctx->dx1, ctx->dx2);
    for (int64_t t0 = 0; t0 < ncell; t0 += nb) {
        const int k = (int)std::min<int64_t>(nb, ncell - t0);
        dim3 g((unsigned)std::min<int64_t>((p + 255) / 256, 1024), k);
        k_cross_cols<<<g, 256, 0, st>>>(cells, t0, ctx->cellidx.as<int>(), p, ctx->n2, (int64_t)ctx->n1 * ctx->n2, cp,
                                         cbuf.as<double>());
        KRY_CHECK_LAUNCH();
        SolveInfo si = solve(ctx, e, cbuf.as<double>(), p, sbuf.as<double>(), p, k, rtol, maxit, 0, pre);
        ok = ok && si.converged;
        k_var_final<<<k, 256, 0, st>>>(cbuf.as<double>(), sbuf.as<double>(), p, e->cov.sigma2, var, t0);
        KRY_CHECK_LAUNCH();
    }
    return ok;
}

}  // namespace kry
