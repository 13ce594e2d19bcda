// FP32 3D register-accumulator collide kernels for clusters of kRgAsync and more CTAs (scatter by
// st.async): instantiations and launch entry points, variants 1 - 4.
#include "ef_cluster_launch.h"
#include "ef_collide_rg.cuh"
#include "ef_launch.h"

namespace ef {

namespace {

template <int N, int V>
constexpr auto rg_kernel()
{
    return collide_kernel_rg<3, N, rg_rpt<V>(), (rg_bound<N, V>() > 0 ? rg_bound<N, V>() : 32), V == 4, true>;
}

// f(kernel) for variant v of size N, or cudaErrorInvalidValue where it is not built
template <int N, typename Fn>
cudaError_t rg_with(int v, Fn f)
{
    if (v == 1) return f(rg_kernel<N, 1>());
    if (v == 2) return f(rg_kernel<N, 2>());
    if constexpr (rg_bound<N, 3>() > 0) {
        if (v == 3) return f(rg_kernel<N, 3>());
    }
    if (v == 4) return f(rg_kernel<N, 4>());
    return cudaErrorInvalidValue;
}

}  // namespace

#define EF_RG_SIZES(X) X(16) X(24) X(32) X(40) X(48) X(64)

cudaError_t rg_async_setup_f32(int N, int v, size_t smem, int cluster, int tpb, int *max_clusters)
{
    auto f = [&](auto k) { return setup_kernel(k, smem, cluster, tpb, max_clusters); };
    switch (N) {
#define EF_CASE(n) case n: return rg_with<n>(v, f);
        EF_RG_SIZES(EF_CASE)
#undef EF_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t rg_async_launch_f32(int N, int v, const CollideArgs &a, int grid_clusters, int tpb, size_t smem, cudaStream_t s)
{
    auto f = [&](auto k) { return launch_kernel(k, a, grid_clusters, tpb, smem, s); };
    switch (N) {
#define EF_CASE(n) case n: return rg_with<n>(v, f);
        EF_RG_SIZES(EF_CASE)
#undef EF_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ef
