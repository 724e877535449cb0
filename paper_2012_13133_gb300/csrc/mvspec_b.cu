// Pass B of the specialised FP32 matvec (mvspec.cuh) for every supported
// (log2 M1, threads per block).
#include "kry_internal.cuh"
#include "mvspec.cuh"
#include "mvwide.cuh"

namespace kspec {

namespace {
struct RunB {
    const SpecArgs& a;
    cudaStream_t st;
    template <int B, int TH>
    bool run() const {
        dim3 grid(a.M2 / nt_of(B, TH), a.np);
        if constexpr (is_wide(B)) {
            auto k = kw_pass_b<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), wide_smem(B, TH), st, a.slab, a.lamP, a.n1, a.M2, a.logCs, a.tww, a.post,
                       a.pair0, a.lam_stride, a.vpt, a.skip, a.nvec);
        } else {
            auto k = ks_pass_b<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), smem_bytes(B, TH), st, a.slab, a.lamP, a.n1, a.M2, a.logCs, a.twf, a.twi, a.post,
                       a.pair0, a.lam_stride, a.vpt, a.skip, a.nvec);
        }
        return true;
    }
};
}  // namespace

bool launch_b(const SpecArgs& a, cudaStream_t st) { return dispatch(ilog2i(a.M1), a.C * transform_threads(a.M1), RunB{a, st}); }

}  // namespace kspec
