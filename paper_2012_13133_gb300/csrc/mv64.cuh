// FP64 matvec passes (mv64.cu) on transforms of fft64.cuh, and the launch shapes
// that the FP64 covariance embedding (embed.cu) shares.
#pragma once

#include <algorithm>

#include "kry_internal.cuh"

namespace kf64 {

// Values per thread and transforms per block of transforms of length L.  The
// values per thread decide the rounding (radix 4 or 16 stages), so they depend on
// L alone: a vector's result must not depend on the batch it is in (without
// reorthogonalisation FP64 Lanczos amplifies rounding to the seventh digit).  Up
// to 512 points, four values: one pair on 256^2 would otherwise occupy 256 of the
// 608 schedulers, and an FP64 instruction costs a scheduler 64 cycles.
struct Shape {
    int E, NT;
    int threads(int L) const { return NT * (L / E); }
};
Shape shape(int L, int want_nt = 0);

void fill_table(double2* tab_dev, cudaStream_t st);

// Arguments of one batch of complex pairs (see kspec::SpecArgs).
struct Args {
    const double* vin;
    int64_t ld_in;
    const double* scale;
    double* vout;
    int64_t ld_out;
    int nvec, pair0, np;
    const uint2* bits;
    int wpr;
    int n1, n2, M1, M2;
    Shape row, col;
    int logC;   // log2 of the slab tile width
    double2* slab;
    const double* lamT;   // [M2][M1], scaled by 1 / (M1 M2)
    int64_t lam_stride;
    int vpt;
    double tau2;
    const double* tau2v;
    double* dots;
    int nds;
    const double2* tw;
    const int* skip;
    int mode;   // 0: observed cells, nugget, dots; 1: every grid cell
};
void launch(const Args& a, cudaStream_t st);

// f.template run<B, E, NT>() for L = 2^B and shape s (throws if not compiled).
// E = 16: 1024 <= L <= 8192 in blocks of 128 or 256 threads (one transform where
// it has more; 256 only with WIDE); E = 4: 8 <= L <= 512 in the smallest blocks
// of at least a warp.
template <int B, bool WIDE, class F>
void dispatch16(const Shape& s, const F& f) {
    constexpr int LT = (1 << B) / 16, N1 = LT >= 128 ? 1 : 128 / LT, N2 = LT >= 256 ? 1 : 256 / LT;
    if (s.NT == N1) return f.template run<B, 16, N1>();
    if constexpr (WIDE && N2 != N1)
        if (s.NT == N2) return f.template run<B, 16, N2>();
    throw KryError{KRY_EUNSUPPORTED, "no FP64 pass for this block"};
}
template <int B, class F>
void dispatch4(const Shape& s, const F& f) {
    constexpr int LT = (1 << B) / 4, NT = LT >= 32 ? 1 : 32 / LT;
    if (s.NT != NT) throw KryError{KRY_EUNSUPPORTED, "no FP64 pass for this block"};
    f.template run<B, 4, NT>();
}
template <bool WIDE, class F>
void dispatch(int L, const Shape& s, const F& f) {
    if (s.E == 16) switch (L) {
        case 1024: return dispatch16<10, WIDE>(s, f);
        case 2048: return dispatch16<11, WIDE>(s, f);
        case 4096: return dispatch16<12, WIDE>(s, f);
        case 8192: return dispatch16<13, WIDE>(s, f);
    }
    else switch (L) {
        case 8: return dispatch4<3>(s, f);
        case 16: return dispatch4<4>(s, f);
        case 32: return dispatch4<5>(s, f);
        case 64: return dispatch4<6>(s, f);
        case 128: return dispatch4<7>(s, f);
        case 256: return dispatch4<8>(s, f);
        case 512: return dispatch4<9>(s, f);
    }
    throw KryError{KRY_EUNSUPPORTED, "no FP64 pass for this length"};
}

// Blocks per SM that leave a 16-value thread 128 registers (64 hold the
// transform, 32 the twiddles of a stage).
constexpr int minb(int th, int E) { return E == 4 ? 1 : th >= 512 ? 1 : 512 / th; }

}  // namespace kf64
