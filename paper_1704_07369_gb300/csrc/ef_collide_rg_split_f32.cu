// FP32 3D register-accumulator collide kernels, split instantiations (parts of a cell's ops on several
// clusters, ef_split.cu): variants 1 and 2 of ef_collide_rg_f32.cu, apart from them so that the split's
// branches cost the unsplit kernels no registers.
#include "ef_cluster_launch.h"
#include "ef_collide_rg.cuh"
#include "ef_launch.h"

namespace ef {

namespace {

template <int N, int V, bool ASYNC>
constexpr auto rg_split_kernel()
{
    return collide_kernel_rg<3, N, rg_rpt<V>(), rg_bound<N, V>(), false, ASYNC, true>;
}

// f(kernel) for variant v and cluster size of size N (only N <= 32 fits fewer than kRgAsync CTAs)
template <int N, typename Fn>
cudaError_t rg_split_with(int v, int cluster, Fn f)
{
    if (v != 1 && v != 2) return cudaErrorInvalidValue;
    if (cluster >= kRgAsync) return v == 1 ? f(rg_split_kernel<N, 1, true>()) : f(rg_split_kernel<N, 2, true>());
    if constexpr (N <= 32) return v == 1 ? f(rg_split_kernel<N, 1, false>()) : f(rg_split_kernel<N, 2, false>());
    return cudaErrorInvalidValue;
}

}  // namespace

#define EF_RG_SIZES(X) X(16) X(24) X(32) X(40) X(48) X(64)

cudaError_t rg_split_setup_f32(int N, int v, size_t smem, int cluster, int tpb, int *max_clusters)
{
    auto f = [&](auto k) { return setup_kernel(k, smem, cluster, tpb, max_clusters); };
    switch (N) {
#define EF_CASE(n) case n: return rg_split_with<n>(v, cluster, f);
        EF_RG_SIZES(EF_CASE)
#undef EF_CASE
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t rg_split_launch_f32(int N, int v, const CollideArgs &a, int grid_clusters, int tpb, size_t smem, cudaStream_t s)
{
    auto f = [&](auto k) { return launch_kernel(k, a, grid_clusters, tpb, smem, s); };
    switch (N) {
#define EF_CASE(n) case n: return rg_split_with<n>(v, a.cluster, f);
        EF_RG_SIZES(EF_CASE)
#undef EF_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace ef
