// Walk kernel instantiations with the level-1 codebook in FP16, and their dispatch
// (compiled apart from lc_search.cu so the instantiations build in parallel).
#include "lc_walk.cuh"

namespace lc {

cudaError_t walk_config_f16(int variant, int M1, bool fq, const WalkArgs &wa, size_t per_warp, int sms, int want,
                            int *wpc, int *grid, size_t *smem)
{
    return by_shape<__half>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        const auto fn = wa.team > 1 ? (wa.beam > 1 ? launch_walk<T::M1, T::D1, __half, T::FQ, false, true, true>
                                                   : launch_walk<T::M1, T::D1, __half, T::FQ, false, false, true>)
                                    : (wa.beam > 1 ? launch_walk<T::M1, T::D1, __half, T::FQ, false, true, false>
                                                   : launch_walk<T::M1, T::D1, __half, T::FQ, false, false, false>);
        return fn(wa, per_warp, sms, want, wpc, grid, smem);
    });
}

cudaError_t walk_run_f16(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                         cudaStream_t st, bool pdl)
{
    return by_shape<__half>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        const auto fn = wa.team > 1 ? (wa.beam > 1 ? run_walk<T::M1, T::D1, __half, T::FQ, false, true, true>
                                                   : run_walk<T::M1, T::D1, __half, T::FQ, false, false, true>)
                                    : (wa.beam > 1 ? run_walk<T::M1, T::D1, __half, T::FQ, false, true, false>
                                                   : run_walk<T::M1, T::D1, __half, T::FQ, false, false, false>);
        return fn(wa, smem, wpc, grid, st, pdl);
    });
}

// The walk instantiation a plan launches (for finding its node in a captured graph).
const void *walk_fn_f16(int variant, int M1, bool fq, bool batch, bool team)
{
    const void *fn = nullptr;
    by_shape<__half>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        fn = team ? (batch ? (const void *)walk_kernel<T::M1, T::D1, __half, T::FQ, false, true, true>
                           : (const void *)walk_kernel<T::M1, T::D1, __half, T::FQ, false, false, true>)
                  : (batch ? (const void *)walk_kernel<T::M1, T::D1, __half, T::FQ, false, true, false>
                           : (const void *)walk_kernel<T::M1, T::D1, __half, T::FQ, false, false, false>);
        return cudaSuccess;
    });
    return fn;
}

cudaError_t descent_config_f16(int variant, int M1, bool fq, const WalkArgs &wa, int sms, int *wpc, int *grid,
                               size_t *smem)
{
    return by_shape<__half>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        return launch_descent<T::M1, T::D1, __half, T::FQ>(wa, sms, wpc, grid, smem);
    });
}

cudaError_t descent_run_f16(int variant, int M1, bool fq, const WalkArgs &wa, size_t smem, int wpc, int grid,
                            cudaStream_t st, bool pdl)
{
    return by_shape<__half>(variant, M1, fq, [&](auto t) {
        using T = decltype(t);
        return run_descent<T::M1, T::D1, __half, T::FQ>(wa, smem, wpc, grid, st, pdl);
    });
}

// The table form: 32 sub-spaces of 3 coordinates.
cudaError_t walk_config_tab(int, int, bool, const WalkArgs &wa, size_t per_warp, int sms, int want, int *wpc, int *grid,
                            size_t *smem)
{
    return wa.beam > 1 ? launch_walk<32, 3, __half, false, true, true, false>(wa, per_warp, sms, want, wpc, grid, smem)
                       : launch_walk<32, 3, __half, false, true, false, false>(wa, per_warp, sms, want, wpc, grid, smem);
}

cudaError_t walk_run_tab(int, int, bool, const WalkArgs &wa, size_t smem, int wpc, int grid, cudaStream_t st, bool pdl)
{
    return wa.beam > 1 ? run_walk<32, 3, __half, false, true, true, false>(wa, smem, wpc, grid, st, pdl)
                       : run_walk<32, 3, __half, false, true, false, false>(wa, smem, wpc, grid, st, pdl);
}

const void *walk_fn_tab(int, int, bool, bool batch, bool)
{
    return batch ? (const void *)walk_kernel<32, 3, __half, false, true, true, false>
                 : (const void *)walk_kernel<32, 3, __half, false, true, false, false>;
}

cudaError_t descent_config_tab(int, int, bool, const WalkArgs &wa, int sms, int *wpc, int *grid, size_t *smem)
{
    return launch_descent<32, 3, __half, false, true>(wa, sms, wpc, grid, smem);
}

cudaError_t descent_run_tab(int, int, bool, const WalkArgs &wa, size_t smem, int wpc, int grid, cudaStream_t st, bool pdl)
{
    return run_descent<32, 3, __half, false, true>(wa, smem, wpc, grid, st, pdl);
}

}  // namespace lc
