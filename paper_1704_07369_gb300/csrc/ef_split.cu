// ef_split.cu -- the finishing kernel of collide launches whose cells are split into parts: sums the
// parts' gains, forms Q = G - F nu and writes Q or F + dt Q with the status checks and diagnostics of
// the collide kernels' last op (ef_collide_impl.cuh, emit_row).
//
// A batch with fewer cells than the device holds clusters leaves SMs idle while each cluster works
// through all of its cell's ops; split, the ops of one cell run on several clusters at once, each
// repeating the forward transform, and their partial gains meet here.  The parts are read back from
// L2 (a part is N^d values, all parts of a launch at most the clusters' worth of cells), eight loads
// in flight a thread, in part order, so the result does not depend on timing.  One cluster of CTAs per
// cell: the diagnostics meet in distributed shared memory.
//
// Measured, unsplit against split with the shape that pick_shape chooses (ef_plan.cpp): Q of one FP32
// cell of N = 32 (Maxwell, 49 ops) 427 -> 31 us; 100 Euler steps with diagnostics of one FP64 2D cell of
// N = 16 16.8 -> 4.7 ms; two such steps of one FP64 cell of N = 32 14.0 -> 1.11 ms; two SSP-RK3 steps of
// four FP64 2D cells of N = 64 5.3 -> 1.17 ms.
#include <type_traits>

#include "ef_collide_impl.cuh"
#include "ef_launch.h"

namespace ef {
namespace {

constexpr int kFinThreads = 256;

template <typename T>
struct FinVec;
template <>
struct FinVec<float> {
    using type = float4;
    static constexpr int W = 4;
};
template <>
struct FinVec<double> {
    using type = double2;
    static constexpr int W = 2;
};

template <typename T, int D>
__global__ void __launch_bounds__(kFinThreads) finish_kernel(const CollideArgs a, int N)
{
    using V = typename FinVec<T>::type;
    constexpr int W = FinVec<T>::W;
    constexpr bool FFD = sizeof(T) == 4 && D == 3;
    constexpr bool ROWS = sizeof(T) == 4;    // sums over F row by row
    using DG = std::conditional_t<FFD, DiagF, Diag>;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int64_t c = blockIdx.x / C;
    const int S = a.nsplit;
    const int cell = (D == 3 ? N * N : N) * N;
    const int64_t coff = a.cell_off ? a.cell_off[c] : c * (int64_t)cell;
    const int64_t cglob = a.cell_id ? a.cell_id[c] : c;
    const T *part = reinterpret_cast<const T *>(a.part) + c * (S + 1) * (int64_t)cell;
    const T *F = reinterpret_cast<const T *>(a.F) + coff;
    T *Out = reinterpret_cast<T *>(a.Q) + coff;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ double red[kFinThreads / 32 + 1][kDiag];

    DG dg;
    dg.reset();
    bool bad = false, neg = false;
    if (ROWS && a.diag) {
        // FP32: the sums over F by rows, in the order of emit_row, so that a cell's moments do not
        // depend on whether its launch was split
        for (int r = rank * kFinThreads + tid; r < (D == 3 ? N * N : N); r += C * kFinThreads) {
            T s_m = 0, s_mx = 0, s_e2 = 0, s_eta = 0, mn_f = F[r * N];
#pragma unroll 4
            for (int n0 = 0; n0 < N; n0 += W) {
                T f[W];
                *reinterpret_cast<V *>(f) = *reinterpret_cast<const V *>(F + r * N + n0);
#pragma unroll
                for (int j = 0; j < W; ++j) {
                    const T jx = T(n0 + j - N / 2);
                    s_m += f[j];
                    s_mx += f[j] * jx;
                    s_e2 += f[j] * jx * jx;
                    if (f[j] > T(0)) s_eta += f[j] * log_t<T>(f[j]);
                    mn_f = f[j] < mn_f ? f[j] : mn_f;
                }
            }
            dg.template add_row<D, T>(s_m, s_mx, s_e2, s_eta, T(0), (D == 3 ? r / N : r) - N / 2, D == 3 ? r % N - N / 2 : 0, mn_f,
                                       T(3.0e38));
        }
        cl.sync();                           // an Euler step in place: every row of F read before any is written
    }
    for (int i0 = (rank * kFinThreads + tid) * W; i0 < cell; i0 += C * kFinThreads * W) {
        T f[W], q[W], nu[W];
        *reinterpret_cast<V *>(f) = *reinterpret_cast<const V *>(F + i0);
        *reinterpret_cast<V *>(nu) = __ldcg(reinterpret_cast<const V *>(part + (int64_t)S * cell + i0));
#pragma unroll
        for (int j = 0; j < W; ++j) q[j] = T(0);
        for (int p0 = 0; p0 < S; p0 += 8) {
            T g[8][W];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (p0 + u < S) *reinterpret_cast<V *>(g[u]) = __ldcg(reinterpret_cast<const V *>(part + (int64_t)(p0 + u) * cell + i0));
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                if (p0 + u >= S) break;
#pragma unroll
                for (int j = 0; j < W; ++j) q[j] += g[u][j];
            }
        }
        const int row = i0 / N, x0 = i0 - row * N;
        const int jz = (D == 3 ? row / N : row) - N / 2, jy = D == 3 ? row % N - N / 2 : 0;
        T s_m = 0, s_mx = 0, s_e2 = 0, s_eta = 0, s_prod = 0, mn_f = f[0], mx_nu = nu[0], mn_out = T(3.0e38);
#pragma unroll
        for (int j = 0; j < W; ++j) {
            const T qv = q[j] - f[j] * nu[j];
            T o = qv;
            if (a.out_mode == OUT_EULER) {
                o = f[j] + T(a.dt) * qv;
                if (o < T(0) && T(a.dt) * nu[j] > T(1)) neg = true;
            }
            if (!isfinite(o)) bad = true;
            if (a.diag) {
                if constexpr (!ROWS) {
                    const T jx = T(x0 + j - N / 2);
                    s_m += f[j];
                    s_mx += f[j] * jx;
                    s_e2 += f[j] * jx * jx;
                    mn_f = f[j] < mn_f ? f[j] : mn_f;
                }
                if (f[j] > T(0)) {
                    const T lf = log_t<T>(f[j]);
                    if constexpr (!ROWS) s_eta += f[j] * lf;
                    s_prod += qv * lf;
                }
                mx_nu = nu[j] > mx_nu ? nu[j] : mx_nu;
                mn_out = o < mn_out ? o : mn_out;
            }
            q[j] = o;
        }
        *reinterpret_cast<V *>(Out + i0) = *reinterpret_cast<V *>(q);
        if (a.diag) {
            if constexpr (FFD) {
                ff_add(dg.sum[6], s_prod);
                dg.min_out = fminf(dg.min_out, mn_out);
            } else if constexpr (ROWS) {
                dg.sum[6] += (double)s_prod;
                dg.min_out = fmin(dg.min_out, (double)mn_out);
            } else {
                dg.template add_row<D, T>(s_m, s_mx, s_e2, s_eta, s_prod, jz, jy, mn_f, mn_out);
            }
            dg.max_nu = mx_nu > dg.max_nu ? mx_nu : dg.max_nu;
        }
    }
    if (bad) record_status(a.status, 7);     // EF_ERR_NOT_FINITE
    if (neg) record_status(a.status, 6);     // EF_ERR_POSITIVITY
    if (!a.diag) return;

    auto merge = [](int k, double v, double u) { return (k == 7 || k == 9) ? fmin(v, u) : (k == 8 ? fmax(v, u) : v + u); };
#pragma unroll
    for (int k = 0; k < kDiag; ++k) {
        double v;
        if constexpr (FFD) {
            if (k < 7) {
                FF x = dg.sum[k];
#pragma unroll
                for (int sh = 16; sh > 0; sh >>= 1)
                    x = ff_merge(x, FF{__shfl_xor_sync(0xffffffffu, x.hi, sh), __shfl_xor_sync(0xffffffffu, x.lo, sh)});
                v = ff_value(x);
            } else {
                float x = k == 7 ? dg.min_f : k == 8 ? dg.max_nu : dg.min_out;
#pragma unroll
                for (int sh = 16; sh > 0; sh >>= 1) {
                    const float u = __shfl_xor_sync(0xffffffffu, x, sh);
                    x = k == 8 ? fmaxf(x, u) : fminf(x, u);
                }
                v = x;
            }
        } else {
            v = k < 7 ? dg.sum[k] : k == 7 ? dg.min_f : k == 8 ? dg.max_nu : dg.min_out;
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) v = merge(k, v, __shfl_xor_sync(0xffffffffu, v, sh));
        }
        if (lane == 0) red[warp][k] = v;
    }
    __syncthreads();
    if (tid < kDiag) {
        double v = red[0][tid];
        for (int w = 1; w < kFinThreads / 32; ++w) v = merge(tid, v, red[w][tid]);
        red[kFinThreads / 32][tid] = v;
    }
    cl.sync();
    if (rank == 0 && tid < kDiag) {
        const int k = tid;
        double v = red[kFinThreads / 32][k];
        for (int r = 1; r < C; ++r) v = merge(k, v, cl.map_shared_rank(&red[0][0], r)[(kFinThreads / 32) * kDiag + k]);
        const double hd = (D == 3) ? a.h * a.h * a.h : a.h * a.h;
        if (k == 0 || k == 5) v *= hd;
        else if (k >= 1 && k <= 3) v *= hd * a.h;
        else if (k == 4) v *= 0.5 * hd * a.h * a.h;
        if (D == 2 && k == 3) v = 0.0;
        a.diag[cglob * kDiag + k] = v;
    }
    cl.sync();                               // no CTA leaves before rank 0 has read its sums
}

template <typename T, int D>
cudaError_t finish_td(int N, const CollideArgs &a, cudaStream_t s)
{
    // CTAs per cell: about four vectors a thread, at most 8 (a portable cluster)
    const int64_t nv = (int64_t)(D == 3 ? N * N : N) * N / FinVec<T>::W;
    int C = 1;
    while (C < 8 && nv > (int64_t)C * kFinThreads * 4) C *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.ncells * C), 1, 1);
    cfg.blockDim = dim3(kFinThreads, 1, 1);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, finish_kernel<T, D>, a, N);
}

}  // namespace

// loads the finishing kernel (a plan-time call: a first launch under capture could not)
cudaError_t split_finish_setup(int prec, int d)
{
    cudaFuncAttributes fa;
    if (prec == 0) return d == 3 ? cudaFuncGetAttributes(&fa, finish_kernel<float, 3>) : cudaFuncGetAttributes(&fa, finish_kernel<float, 2>);
    return d == 3 ? cudaFuncGetAttributes(&fa, finish_kernel<double, 3>) : cudaFuncGetAttributes(&fa, finish_kernel<double, 2>);
}

cudaError_t split_finish_launch(int prec, int d, int N, const CollideArgs &a, cudaStream_t s)
{
    if (prec == 0) return d == 3 ? finish_td<float, 3>(N, a, s) : finish_td<float, 2>(N, a, s);
    return d == 3 ? finish_td<double, 3>(N, a, s) : finish_td<double, 2>(N, a, s);
}

}  // namespace ef
