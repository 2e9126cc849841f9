// Walk kernel instantiations with the level-1 codebook in FP32, and their dispatch
// (compiled apart from lc_search.cu so the instantiations build in parallel).
#include "lc_walk.cuh"

namespace lc {

cudaError_t walk_config_f32(int variant, int M1, bool fq, const WalkArgs &wa, size_t per_warp, int sms, int want,
                            int *wpc, int *grid, size_t *smem)
{
    return by_shape<float>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        const auto fn = wa.team > 1 ? (wa.beam > 1 ? launch_walk<T::M1, T::D1, float, T::FQ, false, true, true>
                                                   : launch_walk<T::M1, T::D1, float, T::FQ, false, false, true>)
                                    : (wa.beam > 1 ? launch_walk<T::M1, T::D1, float, T::FQ, false, true, false>
                                                   : launch_walk<T::M1, T::D1, float, T::FQ, false, false, false>);
        return fn(wa, per_warp, sms, want, wpc, grid, smem);
    });
}

cudaError_t walk_run_f32(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                         cudaStream_t st, bool pdl)
{
    return by_shape<float>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        const auto fn = wa.team > 1 ? (wa.beam > 1 ? run_walk<T::M1, T::D1, float, T::FQ, false, true, true>
                                                   : run_walk<T::M1, T::D1, float, T::FQ, false, false, true>)
                                    : (wa.beam > 1 ? run_walk<T::M1, T::D1, float, T::FQ, false, true, false>
                                                   : run_walk<T::M1, T::D1, float, T::FQ, false, false, false>);
        return fn(wa, smem, wpc, grid, st, pdl);
    });
}

// The walk instantiation a plan launches (for finding its node in a captured graph).
const void *walk_fn_f32(int variant, int M1, bool fq, bool batch, bool team)
{
    const void *fn = nullptr;
    by_shape<float>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        fn = team ? (batch ? (const void *)walk_kernel<T::M1, T::D1, float, T::FQ, false, true, true>
                           : (const void *)walk_kernel<T::M1, T::D1, float, T::FQ, false, false, true>)
                  : (batch ? (const void *)walk_kernel<T::M1, T::D1, float, T::FQ, false, true, false>
                           : (const void *)walk_kernel<T::M1, T::D1, float, T::FQ, false, false, false>);
        return cudaSuccess;
    });
    return fn;
}

cudaError_t descent_config_f32(int variant, int M1, bool fq, const WalkArgs &wa, int sms, int *wpc, int *grid,
                               size_t *smem)
{
    return by_shape<float>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        return launch_descent<T::M1, T::D1, float, T::FQ>(wa, sms, wpc, grid, smem);
    });
}

cudaError_t descent_run_f32(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                            cudaStream_t st, bool pdl)
{
    return by_shape<float>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        return run_descent<T::M1, T::D1, float, T::FQ>(wa, smem, wpc, grid, st, pdl);
    });
}

}  // namespace lc
