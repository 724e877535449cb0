// Pass C of the specialised FP32 matvec (mvspec.cuh) for every supported
// (log2 M2, threads per block).
#include "kry_internal.cuh"
#include "mvspec.cuh"
#include "mvwide.cuh"

namespace kspec {

namespace {
struct RunC {
    const SpecArgs& a;
    cudaStream_t st;
    template <int B, int TH>
    bool run() const {
        constexpr int NT = nt_of(B, TH);
        dim3 grid((a.n1 + NT - 1) / NT, a.np);
        if constexpr (is_wide(B)) {
            auto k = kw_pass_c<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), wide_smem(B, TH), st, a.slab, a.vin, a.ld_in, a.scale, a.vout, a.ld_out, a.nvec,
                       a.pair0, a.bits, a.wpr, a.n1, a.logCs, a.tau2, a.dots, a.nds, a.tww, a.post, a.tau2v, a.vpt, a.skip);
        } else {
            auto k = ks_pass_c<B, TH>;
            KRY_ALLOW_MAX_SMEM(k);
            launch_pdl(k, grid, dim3(TH), smem_bytes(B, TH), st, reinterpret_cast<const float4*>(a.slab), a.vin, a.ld_in,
                       a.scale, a.vout, a.ld_out, a.nvec, a.pair0, a.bits, a.wpr, a.n1, a.logCs, a.tau2, a.dots,
                       a.nds, a.twi, a.post, a.tau2v, a.vpt, a.skip);
        }
        return true;
    }
};
}  // namespace

bool launch_c(const SpecArgs& a, cudaStream_t st) { return dispatch(ilog2i(a.M2), a.G * transform_threads(a.M2), RunC{a, st}); }

}  // namespace kspec
