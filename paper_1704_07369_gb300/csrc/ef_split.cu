// ef_split.cu -- the finishing kernel of collide launches whose cells are split into parts: sums the
// parts' gains, forms Q = G - F nu and writes Q or F + dt Q with the status checks and diagnostics of
// the collide kernels' last op (ef_collide_impl.cuh, emit_row).
//
// A batch with fewer cells than the device holds clusters leaves SMs idle while each cluster works
// through all of its cell's ops; split, the ops of one cell run on several clusters at once, each
// repeating the forward transform, and their partial gains meet here.  The parts are read back from
// L2 (a part is N^d values, all parts of a launch at most the clusters' worth of cells), eight loads
// in flight a thread, in part order, so the result does not depend on timing.  A cell's rows are spread
// over as many CTAs as fill the device (split_finish_ctas): an FP64 warp instruction takes a
// sub-partition 64 cycles, and a point's logarithm and sums are about 65 of them.  A CTA owns whole
// rows, so that a step in place may write them behind its own reads alone; the diagnostics of the
// CTAs meet in global memory, summed in CTA order by whichever CTA arrives last.
// One cluster of at most eight CTAs per cell, the diagnostics in distributed shared memory, took 88 us
// for an FP64 cell of N = 32, 13 us for an FP64 2D cell of N = 16 and 17 us for the 49 parts of an FP32
// cell of N = 32.
//
// Measured, unsplit one-line-per-thread kernels against split with the shape that pick_shape chooses
// (ef_plan.cpp) and the present kernels: Q of one FP32 cell of N = 32 (Maxwell, 49 ops) 427 -> 25 us; 100
// Euler steps with diagnostics of one FP64 2D cell of N = 16 16.8 -> 2.46 ms; two such steps of one FP64
// cell of N = 32 14.0 -> 0.79 ms; two SSP-RK3 steps of four FP64 2D cells of N = 64 5.3 -> 0.80 ms.
#include <algorithm>
#include <type_traits>

#include "ef_collide_impl.cuh"
#include "ef_launch.h"

namespace ef {
namespace {

constexpr int kFinThreads = 128;     // one warp per sub-partition

// values per thread and pass (split_finish_ctas has them too): 2D FP64 cells are small, so one
template <typename T, int D>
struct FinVec {
    using type = float4;
    static constexpr int W = 4;
};
template <>
struct FinVec<double, 3> {
    using type = double2;
    static constexpr int W = 2;
};
template <>
struct FinVec<double, 2> {
    using type = double;
    static constexpr int W = 1;
};

// v[k] of all lanes summed, k < 8, with 9 additions a lane in place of 40: lanes 4 k .. 4 k + 3 return sum k
__device__ __forceinline__ double warp_sum8(double (&v)[8], int lane)
{
#pragma unroll
    for (int h = 4, sh = 16; h >= 1; h >>= 1, sh >>= 1) {
#pragma unroll
        for (int j = 0; j < h; ++j) {
            const bool up = lane & sh;
            const double keep = up ? v[j + h] : v[j], send = up ? v[j] : v[j + h];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, send, sh);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    return v[0];
}

template <typename T, int D>
__global__ void __launch_bounds__(kFinThreads) finish_kernel(const CollideArgs a, int N)
{
    using V = typename FinVec<T, D>::type;
    constexpr int W = FinVec<T, D>::W;
    constexpr bool FFD = sizeof(T) == 4 && D == 3;
    constexpr bool ROWS = sizeof(T) == 4;    // sums over F row by row
    using DG = std::conditional_t<FFD, DiagF, Diag>;
    const int C = a.fin_ctas, rank = (int)(blockIdx.x % C);
    const int64_t c = blockIdx.x / C;
    const int nrow = D == 3 ? N * N : N, rpc = (nrow + C - 1) / C;
    const int r0 = min(rank * rpc, nrow), r1 = min(r0 + rpc, nrow);     // rows of this CTA
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
    bool bad = false, neg = false;           // an updated value below zero
    // dt nu > 1 somewhere in the cell: the part with the loss has left it (ef_collide_impl.cuh, fin_flags).
    // Loaded here, beside F, and not where it is used: its latency would end the launch
    unsigned big;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(big) : "l"(fin_flags(a) + c));
    if (ROWS && a.diag) {
        // FP32: the sums over F by rows, in the order of emit_row, so that a cell's moments do not
        // depend on whether its launch was split
        for (int r = r0 + tid; r < r1; r += kFinThreads) {
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
        __syncthreads();                     // an Euler step in place: the CTA's rows of F read before any is written
    }
    for (int i0 = r0 * N + tid * W; i0 < r1 * N; i0 += kFinThreads * W) {
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
                if (o < T(0)) neg = true;
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
    if (a.out_mode == OUT_EULER && neg && big) record_status(a.status, 6);     // EF_ERR_POSITIVITY
    if (!a.diag) return;

    auto merge = [](int k, double v, double u) { return (k == 7 || k == 9) ? fmin(v, u) : (k == 8 ? fmax(v, u) : v + u); };
    auto extreme = [](int k, auto x) {
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1) {
            const auto u = __shfl_xor_sync(0xffffffffu, x, sh);
            x = k == 8 ? fmax(x, u) : fmin(x, u);
        }
        return x;
    };
    if constexpr (FFD) {
#pragma unroll
        for (int k = 0; k < 7; ++k) {
            FF x = dg.sum[k];
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1)
                x = ff_merge(x, FF{__shfl_xor_sync(0xffffffffu, x.hi, sh), __shfl_xor_sync(0xffffffffu, x.lo, sh)});
            if (lane == 0) red[warp][k] = ff_value(x);
        }
    } else {
        double v[8];
#pragma unroll
        for (int k = 0; k < 7; ++k) v[k] = dg.sum[k];
        v[7] = 0.0;
        const double t = warp_sum8(v, lane);
        if ((lane & 3) == 0 && lane < 28) red[warp][lane >> 2] = t;
    }
    {
        const double mf = extreme(7, dg.min_f), mx = extreme(8, dg.max_nu), mo = extreme(9, dg.min_out);
        if (lane == 0) {
            red[warp][7] = mf;
            red[warp][8] = mx;
            red[warp][9] = mo;
        }
    }
    __syncthreads();
    auto finish = [&](int k, double v) {
        const double hd = (D == 3) ? a.h * a.h * a.h : a.h * a.h;
        if (k == 0 || k == 5) v *= hd;
        else if (k >= 1 && k <= 3) v *= hd * a.h;
        else if (k == 4) v *= 0.5 * hd * a.h * a.h;
        if (D == 2 && k == 3) v = 0.0;
        a.diag[cglob * kDiag + k] = v;
    };
    double *cta = reinterpret_cast<double *>(static_cast<unsigned char *>(a.fin) + a.fin_off) + c * C * kDiag;   // [C][kDiag]
    if (tid < kDiag) {
        double v = red[0][tid];
        for (int w = 1; w < kFinThreads / 32; ++w) v = merge(tid, v, red[w][tid]);
        if (C == 1) finish(tid, v);
        else cta[rank * kDiag + tid] = v;
    }
    if (C == 1) return;
    // the CTA that arrives last sums the cell's CTAs in order, and leaves the arrival count at zero
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (tid == 0) {
        int *count = static_cast<int *>(a.fin) + c;
        last = atomicAdd(count, 1) == C - 1;
        if (last) *count = 0;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (C <= 8) {
        if (tid < kDiag) {
            double v = __ldcg(cta + tid);
            for (int r = 1; r < C; ++r) v = merge(tid, v, __ldcg(cta + r * kDiag + tid));
            finish(tid, v);
        }
        return;
    }
    // warp-uniform k: one FP64 instruction a step, not the three of merge
    for (int k = warp; k < kDiag; k += kFinThreads / 32) {
        double v;
        if (k < 7) {
            v = 0.0;
            for (int r = lane; r < C; r += 32) v += __ldcg(cta + r * kDiag + k);
#pragma unroll
            for (int sh = 16; sh > 0; sh >>= 1) v += __shfl_xor_sync(0xffffffffu, v, sh);
        } else {
            v = k == 8 ? -1.0e300 : 1.0e300;
            for (int r = lane; r < C; r += 32) v = merge(k, v, __ldcg(cta + r * kDiag + k));
            v = extreme(k, v);
        }
        if (lane == 0) finish(k, v);
    }
}

template <typename T, int D>
cudaError_t finish_td(int N, const CollideArgs &a, cudaStream_t s)
{
    finish_kernel<T, D><<<(unsigned)(a.ncells * a.fin_ctas), kFinThreads, 0, s>>>(a, N);
    return cudaGetLastError();
}

}  // namespace

// CTAs per cell of the finishing launch: rows enough for a pass of every thread, at most four CTAs per
// SM in all (one where the cells alone are more)
int split_finish_ctas(int prec, int d, int N, int64_t n, int sms)
{
    const int W = prec == 0 ? 4 : d == 3 ? 2 : 1, rows = d == 3 ? N * N : N;
    const int64_t most = std::max<int64_t>(1, (int64_t)4 * sms / std::max<int64_t>(n, 1));
    const int rpc = (int)std::max<int64_t>((kFinThreads * W + N - 1) / N, (rows + most - 1) / most);
    return (rows + rpc - 1) / rpc;
}

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
