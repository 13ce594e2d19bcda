// ef_mlp.cu -- the learned surrogate's multilayer perceptron: bf16 weights and activations, FP32
// accumulation, hand-written training (forward, MSE loss, backward, Adam) and inference.
//
// Layer l: pre_l = A_{l-1} W_l^T + b_l, A_l = relu(pre_l) (no activation on the last layer).
// Every product is one "TN" GEMM C[M,N] = A[M,K] B[N,K]^T with both operands K-contiguous bf16
// and an FP32 accumulator on the tensor cores: tcgen05.mma fed by TMA, with the accumulator in
// tensor memory, for the shapes it tiles (M a multiple of 128), else mma.sync m16n8k16 with 64 x 64
// tiles.  Backward products use the transposed
// copies the forward pass and the optimizer write alongside (activations^T, W^T).
// Split precision: every layer input a (the features and each hidden activation) is stored as two
// bf16 halves, hi = bf16(a) and lo = bf16(a - hi), side by side, and multiplied against the weights
// duplicated [bf16(W) | bf16(W)], so that a forward product sees a to about 16 mantissa bits while
// both tensor-core operands stay bf16.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <string>
#include <vector>

#include "ef.h"
#include "ef_launch.h"

namespace {

using bf16 = __nv_bfloat16;

// mma.sync kernel: 64 x 64 tiles, K in blocks of 64, four cp.async stages; a shared-memory row of 72 bf16
// (144 bytes) keeps ldmatrix and the staged epilogue rows free of bank conflicts
constexpr int BM = 64, BN = 64, BK = 64, LDS = BK + 8, NSTAGE = 4;
constexpr size_t kSyncSmem = (size_t)NSTAGE * (BM + BN) * LDS * 2;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(smem)), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N)); }

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const void *p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_u32(p)));
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

struct GemmArgs {
    const bf16 *A;      // [M][lda], K contiguous
    const bf16 *B;      // [N][ldb], K contiguous
    int M, N, K, lda, ldb;
    const float *bias;  // nullable [N]
    int relu;
    float *Cf;          // nullable fp32 out [M][ldcf]  (pre-activation)
    int ldcf;
    bf16 *Cb;           // nullable bf16 out [M][ldcb]  (post-activation)
    int ldcb;
    bf16 *CbT;          // nullable bf16 transposed out [N][ldcbt]
    int ldcbt;
    int lo_off;         // > 0: also write the low halves a - bf16(a) at column / row + lo_off
    int *status;        // nullable: device status word, EF_ERR_TIMEOUT (5) when a bounded wait gives up
    const float *pre;   // EPI_DA: [M][ldpre] pre-activations whose sign masks the result
    int ldpre;
    float *db;          // EPI_DW: nullable [M] sums of A's rows
};

// What the mma.sync kernel does with its product:
//   EPI_FWD  bias, optional FP32 copy, relu, bf16 halves and their transposes (GemmArgs above)
//   EPI_DW   weight gradient of the tied hi / lo halves: B holds [hi rows | lo rows], N counts both; the
//            two products of a column are added and stored in Cf [M][ldcf], and A's row sums in db
//   EPI_DA   gradient at the layer below: masked by pre > 0, as bf16 in Cb and transposed in CbT
enum Epilogue { EPI_FWD = 0, EPI_DW = 1, EPI_DA = 2 };

// 4 warps in 2 x 2, each 32 x 32 (2 m16 x 4 n8 tiles).  M % 64 == N % 64 == K % 64 == 0.  The training
// batch's products (64 - 240 tiles) leave one or two CTAs per SM, so a tile's time is its serial chain
// of K blocks: three blocks are in flight ahead of the one being multiplied.  Every product is summed
// in K order by one accumulator chain, whatever the tile or stage count.  Results leave through
// shared memory as 16-byte pieces of rows, for the transposed copies too; the element-wise passes that
// followed a product (fold of the halves, relu mask, row sums) are its epilogue.  Loss and gradients of
// a 1024-row batch (928 - 512 x 3 - 926): 300 -> 169 us, 27 launches -> 15.
template <int MODE>
__global__ void __launch_bounds__(128) gemm_sync_kernel(const GemmArgs g)
{
    extern __shared__ __align__(16) unsigned char sync_raw[];
    bf16 *sA = reinterpret_cast<bf16 *>(sync_raw);             // [NSTAGE][BM][LDS]
    bf16 *sB = sA + NSTAGE * BM * LDS;                         // [NSTAGE][BN][LDS]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int wm = warp >> 1, wn = warp & 1;
    const int m0 = blockIdx.y * BM;
    const int n0 = blockIdx.x * (MODE == EPI_DW ? BN / 2 : BN);
    const int nk = g.K / BK;

    auto load_tile = [&](int kt) {
        if (kt < nk) {
            bf16 *a = sA + (kt % NSTAGE) * BM * LDS, *b = sB + (kt % NSTAGE) * BN * LDS;
            // A: 64 rows x 64 bf16 = 512 chunks of 16 B; B likewise: 4 + 4 chunks per thread
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = tid + i * 128;
                const int r = c >> 3, k8 = (c & 7) * 8;
                // EPI_DW: 32 rows of the hi halves, then the same 32 of the lo halves
                const int rb = MODE == EPI_DW ? (r < BN / 2 ? n0 + r : g.N / 2 + n0 + r - BN / 2) : n0 + r;
                cp_async16(a + r * LDS + k8, g.A + (size_t)(m0 + r) * g.lda + kt * BK + k8);
                cp_async16(b + r * LDS + k8, g.B + (size_t)rb * g.ldb + kt * BK + k8);
            }
        }
        cp_async_commit();
    };

    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.f;
    // EPI_DW: sums of A's rows, two threads a row, as an unevaluated pair (Knuth's TwoSum): the 64 values
    // of a K block in a tree, the blocks without rounding.  (320 sums of 16384 values of one sign over
    // eight binary orders: largest relative error 7e-7 with one FP32 chain, 4e-8 so.)
    [[maybe_unused]] float rs_hi = 0.f, rs_lo = 0.f;

    for (int kt = 0; kt < NSTAGE - 1; ++kt) load_tile(kt);
    for (int kt = 0; kt < nk; ++kt) {
        cp_async_wait<NSTAGE - 2>();
        __syncthreads();                                       // block kt has landed; block kt - 1 is read
        load_tile(kt + NSTAGE - 1);
        const bf16 *a = sA + (kt % NSTAGE) * BM * LDS, *b = sB + (kt % NSTAGE) * BN * LDS;
        if constexpr (MODE == EPI_DW) {
            if (blockIdx.x == 0 && g.db) {
                float t[8] = {};
#pragma unroll
                for (int k8 = 0; k8 < BK / 2; k8 += 8) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(a + (tid >> 1) * LDS + (tid & 1) * (BK / 2) + k8);
                    const bf16 *e = reinterpret_cast<const bf16 *>(&w);
#pragma unroll
                    for (int j = 0; j < 8; ++j) t[j] += __bfloat162float(e[j]);
                }
#pragma unroll
                for (int h = 4; h > 0; h >>= 1)
#pragma unroll
                    for (int j = 0; j < h; ++j) t[j] += t[j + h];
                const float b = t[0] + __shfl_xor_sync(0xffffffffu, t[0], 1);
                const float sum = rs_hi + b, bb = sum - rs_hi;
                rs_lo += (rs_hi - (sum - bb)) + (b - bb);
                rs_hi = sum;
            }
        }
#pragma unroll
        for (int kk = 0; kk < BK; kk += 16) {
            uint32_t af[2][4];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = wm * 32 + i * 16 + (lane & 7) + ((lane >> 3) & 1) * 8;
                ldmatrix_x4(af[i], a + r * LDS + kk + (lane >> 4) * 8);
            }
            uint32_t bfr[4][2];
#pragma unroll
            for (int j2 = 0; j2 < 2; ++j2) {      // two n8 tiles per ldmatrix.x4
                uint32_t t[4];
                const int n = wn * 32 + j2 * 16 + (lane & 7) + (lane >> 4) * 8;
                ldmatrix_x4(t, b + n * LDS + kk + ((lane >> 3) & 1) * 8);
                bfr[2 * j2][0] = t[0];
                bfr[2 * j2][1] = t[1];
                bfr[2 * j2 + 1][0] = t[2];
                bfr[2 * j2 + 1][1] = t[3];
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], af[i], bfr[j][0], bfr[j][1]);
        }
    }
    cp_async_wait<0>();
    __syncthreads();                                           // the stages are free: epilogue staging
    // fragment: c0,c1 at (row, col..col+1), c2,c3 at (row + 8, ...)
    if constexpr (MODE == EPI_DW) {
        float *sf = reinterpret_cast<float *>(sync_raw);       // [64][34] products with the lo halves
        constexpr int LF = BN / 2 + 2;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            if (wn == 1 - half) {
#pragma unroll
                for (int i = 0; i < 2; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int row = wm * 32 + i * 16 + (lane >> 2) + h * 8, col = j * 8 + (lane & 3) * 2;
                            float2 *q = reinterpret_cast<float2 *>(sf + row * LF + col);
                            if (half == 0) {
                                *q = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
                            } else {
                                const float2 lo = *q;
                                *reinterpret_cast<float2 *>(g.Cf + (size_t)(m0 + row) * g.ldcf + n0 + col) =
                                    make_float2(acc[i][j][2 * h] + lo.x, acc[i][j][2 * h + 1] + lo.y);
                            }
                        }
            }
            __syncthreads();
        }
        // an overflowed sum stays infinite (its low part is a NaN)
        if (blockIdx.x == 0 && g.db && !(tid & 1)) g.db[m0 + (tid >> 1)] = isinf(rs_hi) ? rs_hi : rs_hi + rs_lo;
        return;
    } else {
        bf16 *st = reinterpret_cast<bf16 *>(sync_raw);         // [hi, hi^T, lo, lo^T][64][LDS]
        const bool lo_out = MODE == EPI_FWD && g.lo_off > 0;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int row = wm * 32 + i * 16 + (lane >> 2) + h * 8, col = wn * 32 + j * 8 + (lane & 3) * 2;
                    float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
                    if constexpr (MODE == EPI_FWD) {
                        if (g.bias) {
                            v0 += g.bias[n0 + col];
                            v1 += g.bias[n0 + col + 1];
                        }
                        if (g.Cf) *reinterpret_cast<float2 *>(g.Cf + (size_t)(m0 + row) * g.ldcf + n0 + col) = make_float2(v0, v1);
                        if (g.relu) {
                            v0 = fmaxf(v0, 0.f);
                            v1 = fmaxf(v1, 0.f);
                        }
                    } else {
                        const float2 p = *reinterpret_cast<const float2 *>(g.pre + (size_t)(m0 + row) * g.ldpre + n0 + col);
                        v0 = p.x > 0.f ? v0 : 0.f;
                        v1 = p.y > 0.f ? v1 : 0.f;
                    }
                    if (!g.Cb && !g.CbT) continue;
                    const bf16 h0 = __float2bfloat16(v0), h1 = __float2bfloat16(v1);
                    *reinterpret_cast<__nv_bfloat162 *>(st + row * LDS + col) = __halves2bfloat162(h0, h1);
                    st[(BM + col) * LDS + row] = h0;
                    st[(BM + col + 1) * LDS + row] = h1;
                    if (lo_out) {
                        const bf16 l0 = __float2bfloat16(v0 - __bfloat162float(h0)), l1 = __float2bfloat16(v1 - __bfloat162float(h1));
                        *reinterpret_cast<__nv_bfloat162 *>(st + (2 * BM + row) * LDS + col) = __halves2bfloat162(l0, l1);
                        st[(3 * BM + col) * LDS + row] = l0;
                        st[(3 * BM + col + 1) * LDS + row] = l1;
                    }
                }
        if (!g.Cb && !g.CbT) return;
        __syncthreads();
        for (int half = 0; half < (lo_out ? 2 : 1); ++half) {
            const bf16 *q = st + half * 2 * BM * LDS;
            const int off = half ? g.lo_off : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int c = tid + i * 128, r = c >> 3, k8 = (c & 7) * 8;
                if (g.Cb) *reinterpret_cast<uint4 *>(g.Cb + (size_t)(m0 + r) * g.ldcb + off + n0 + k8) = *reinterpret_cast<const uint4 *>(q + r * LDS + k8);
                if (g.CbT) *reinterpret_cast<uint4 *>(g.CbT + (size_t)(off + n0 + r) * g.ldcbt + m0 + k8) = *reinterpret_cast<const uint4 *>(q + (BM + r) * LDS + k8);
            }
        }
    }
}

template <int MODE>
cudaError_t gemm_sync(const GemmArgs &g, cudaStream_t s)
{
    if (g.M % BM || g.N % BN || g.K % BK) return cudaErrorInvalidValue;
    static unsigned long long set_on = 0;    // devices on which the attribute has been raised
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(__atomic_load_n(&set_on, __ATOMIC_ACQUIRE) & bit)) {
        e = cudaFuncSetAttribute(gemm_sync_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSyncSmem);
        if (e != cudaSuccess) return e;
        __atomic_fetch_or(&set_on, bit, __ATOMIC_ACQ_REL);
    }
    gemm_sync_kernel<MODE><<<dim3(g.N / BN, g.M / BM), 128, kSyncSmem, s>>>(g);
    return cudaGetLastError();
}

// ------------------------------------------------------------ tcgen05 GEMM ---------------
// The same product and epilogue on the 5th-generation tensor cores, persistent: one CTA per SM works
// through 128 x TN tiles of C (columns fastest, so that a row block of A is read from L2), K in blocks of
// 64.  Six warps: a producer thread (TMA loads with 128-byte swizzle into a ring of shared-memory
// stages), an MMA thread (tcgen05.mma kind::f16, M = 128, N = TN, K = 16), and four warps that write a
// finished tile out while the next one is accumulated (two accumulators in tensor memory; warp w reads
// lanes 32 (w % 4) ..).  A layer's product of 16384 cells is K = 1024 - 1920: 1 - 2 us of loads and MMAs a
// tile against as long an epilogue, so the overlap is worth up to half.  Results leave through shared
// memory, 64 or 128 contiguous bytes of a row at a time: written straight from the accumulator layout
// (a thread per row) every store touched 32 half-used sectors.
// Every mbarrier wait is bounded.  A wait that gives up stops its role (the others run out in turn),
// records EF_ERR_TIMEOUT in the status word, the CTA's tiles from there on become NaN without a read of the
// accumulator, copies and MMAs still in flight are waited for (bounded), and the tensor memory is
// released in every case.
constexpr int TC_BM = 128, TC_BK = 64, TC_THREADS = 192;
constexpr int TC_SROW = 144;                     // staged row: 128 bytes, padded against bank conflicts
template <int TN>
__host__ __device__ constexpr int tc_stages() { return TN >= 256 ? 4 : TN >= 192 ? 5 : TN >= 128 ? 6 : 8; }
template <int TN>
__host__ __device__ constexpr size_t tc_smem()
{
    return (size_t)tc_stages<TN>() * (TC_BM + TN) * TC_BK * 2 + 4 * 32 * TC_SROW + 1024;
}

__device__ __forceinline__ uint64_t tc_sdesc(uint32_t addr)
{
    // K-major operand with 128-byte swizzle: start address, leading offset unused (1), stride 1024
    // bytes between 8-row groups, descriptor version 1, layout type 2 (128-byte swizzle)
    return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)2 << 61);
}

// instruction descriptor, kind::f16: FP32 accumulator, bf16 A and B, both K-major
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Bounded wait on one mbarrier phase: gives up after about one second of device time (or 2^26
// polls), far beyond any wait of a healthy pipeline (microseconds).
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity)
{
    uint64_t t0;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int it = 0; it < (1 << 26); ++it) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
        if ((it & 1023) == 1023) {
            uint64_t t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t - t0 > 1000000000ull) return false;
        }
    }
    return false;
}

template <int TN>
__global__ void __launch_bounds__(TC_THREADS, 1) gemm_tc_kernel(const __grid_constant__ CUtensorMap tA,
                                                                const __grid_constant__ CUtensorMap tB, const GemmArgs g)
{
    constexpr int A_BYTES = TC_BM * TC_BK * 2, B_BYTES = TN * TC_BK * 2, STAGE = A_BYTES + B_BYTES, ST = tc_stages<TN>();
    constexpr int TCOLS = TN <= 64 ? 64 : (TN <= 128 ? 128 : 256);     // tensor-memory columns of one accumulator
    extern __shared__ __align__(1024) unsigned char tc_raw[];
    unsigned char *tc_smem = (unsigned char *)(((uintptr_t)tc_raw + 1023) & ~(uintptr_t)1023);   // swizzle atoms
    __shared__ __align__(8) uint64_t full[ST], empty[ST], accf[2], acce[2], drain;
    __shared__ uint32_t tmem_base;
    __shared__ int s_issued, s_used, s_fail;     // K blocks loaded, K blocks multiplied, a wait gave up
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nk = g.K / TC_BK, ncol = g.N / TN, ntiles = (g.M / TC_BM) * ncol;
    const uint32_t sbase = smem_u32(tc_smem);

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base)),
                     "r"(2 * TCOLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
    }
    if (tid == 0) {
        auto init = [](uint64_t *b, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(b)), "r"(n)); };
        for (int i = 0; i < ST; ++i) {
            init(&full[i], 1);
            init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            init(&accf[i], 1);
            init(&acce[i], 4);
        }
        init(&drain, 1);
        s_issued = s_used = s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&tA));
        asm volatile("prefetch.tensormap [%0];\n" ::"l"(&tB));
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
    const uint32_t tmem = tmem_base;

    if (warp == 0) {
        if (lane == 0) {
            int it = 0;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x) {
                const int m0 = t / ncol * TC_BM, n0 = t % ncol * TN;
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const int st = it % ST;
                    if (it >= ST && !tc_wait(smem_u32(&empty[st]), (uint32_t)((it / ST - 1) & 1))) {
                        ok = false;
                        break;
                    }
                    const uint32_t a0 = sbase + st * STAGE, b0 = a0 + A_BYTES, bar = smem_u32(&full[st]);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(STAGE));
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
                                 ::"r"(a0), "l"(&tA), "r"(kb * TC_BK), "r"(m0), "r"(bar) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n"
                                 ::"r"(b0), "l"(&tB), "r"(kb * TC_BK), "r"(n0), "r"(bar) : "memory");
                }
            }
            s_issued = it;
            if (!ok) atomicExch(&s_fail, 1);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int it = 0, j = 0;                   // K blocks so far, tiles so far
            bool ok = true;
            for (int t = blockIdx.x; ok && t < ntiles; t += gridDim.x, ++j) {
                if (j >= 2 && !tc_wait(smem_u32(&acce[j & 1]), (uint32_t)((j / 2 - 1) & 1))) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
                const uint32_t acc_col = tmem + (uint32_t)(j & 1) * TCOLS;
                for (int kb = 0; kb < nk; ++kb, ++it) {
                    const int st = it % ST;
                    if (!tc_wait(smem_u32(&full[st]), (uint32_t)((it / ST) & 1))) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
                    const uint32_t a0 = sbase + st * STAGE, b0 = a0 + A_BYTES;
#pragma unroll
                    for (int k16 = 0; k16 < TC_BK / 16; ++k16) {
                        const uint64_t ad = tc_sdesc(a0 + k16 * 32), bd = tc_sdesc(b0 + k16 * 32);
                        const uint32_t acc = (kb > 0 || k16 > 0) ? 1u : 0u;
                        asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
                                     ::"r"(acc_col), "l"(ad), "l"(bd), "r"(tc_idesc(TC_BM, TN)), "r"(acc));
                    }
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                                 ::"r"(smem_u32(&empty[st])));
                }
                if (ok)
                    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                                 ::"r"(smem_u32(&accf[j & 1])));
            }
            s_used = it;
            if (!ok) {
                // the MMAs queued so far, before their stages and accumulators go away
                atomicExch(&s_fail, 1);
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(&drain)));
                tc_wait(smem_u32(&drain), 0);
            }
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
        }
    } else {
        const int sub = warp & 3;                // tensor-memory lanes 32 sub ..
        unsigned char *stg = tc_smem + ST * STAGE + sub * 32 * TC_SROW;
        const float nan = __int_as_float(0x7fc00000);
        bool ok = true;
        int j = 0;
        for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++j) {
            const int m0 = t / ncol * TC_BM + sub * 32, n0 = t % ncol * TN;
            if (ok && !__all_sync(0xffffffffu, tc_wait(smem_u32(&accf[j & 1]), (uint32_t)((j / 2) & 1)))) {
                ok = false;
                if (lane == 0) atomicExch(&s_fail, 1);
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
            const uint32_t acc = tmem + (uint32_t)(j & 1) * TCOLS + ((uint32_t)(sub * 32) << 16);
#pragma unroll 1
            for (int c0 = 0; c0 < TN; c0 += 32) {
                uint32_t r[32];
                if (ok) {                        // warp-uniform: after a give-up the accumulator is not read
                    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                                 : "r"(acc + c0));
                    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::);
                    if (c0 + 32 == TN) {         // the accumulator is read: the MMA thread may start on it again
                        asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
                        __syncwarp();
                        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&acce[j & 1])) : "memory");
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(nan);
                }
                const int col = n0 + c0;
                float v[32];
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                    const float4 b = g.bias ? __ldg(reinterpret_cast<const float4 *>(g.bias + col + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    v[i] = __uint_as_float(r[i]) + b.x;
                    v[i + 1] = __uint_as_float(r[i + 1]) + b.y;
                    v[i + 2] = __uint_as_float(r[i + 2]) + b.z;
                    v[i + 3] = __uint_as_float(r[i + 3]) + b.w;
                }
                if (g.Cf) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float4 *>(stg + lane * TC_SROW + i * 16) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int rr = i * 4 + (lane >> 3), pc = lane & 7;
                        *reinterpret_cast<float4 *>(g.Cf + (size_t)(m0 + rr) * g.ldcf + col + pc * 4) =
                            *reinterpret_cast<const float4 *>(stg + rr * TC_SROW + pc * 16);
                    }
                }
                if (!g.Cb && !g.CbT) continue;
                if (g.relu && ok) {              // (fmaxf would turn a given-up tile's NaN into 0)
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] = fmaxf(v[i], 0.f);
                }
                bf16 hi[32], lo[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    hi[i] = __float2bfloat16(v[i]);
                    lo[i] = __float2bfloat16(v[i] - __bfloat162float(hi[i]));
                }
                if (g.Cb) {
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        *reinterpret_cast<uint4 *>(stg + lane * TC_SROW + i * 16) = *reinterpret_cast<const uint4 *>(hi + 8 * i);
                        *reinterpret_cast<uint4 *>(stg + lane * TC_SROW + 64 + i * 16) = *reinterpret_cast<const uint4 *>(lo + 8 * i);
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {            // 64 bytes of the hi half and 64 of the lo half of a row
                        const int rr = i * 4 + (lane >> 3), pc = lane & 7, half = pc >> 2;
                        if (half == 0 || g.lo_off)
                            *reinterpret_cast<uint4 *>(g.Cb + (size_t)(m0 + rr) * g.ldcb + half * g.lo_off + col + (pc & 3) * 8) =
                                *reinterpret_cast<const uint4 *>(stg + rr * TC_SROW + pc * 16);
                    }
                }
                if (g.CbT) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        g.CbT[(size_t)(col + i) * g.ldcbt + m0 + lane] = hi[i];
                        if (g.lo_off) g.CbT[(size_t)(g.lo_off + col + i) * g.ldcbt + m0 + lane] = lo[i];
                    }
                }
            }
        }
    }
    __syncthreads();
    if (s_fail) {
        if (tid == 0) {
            if (g.status) atomicCAS(g.status, 0, 5);     // EF_ERR_TIMEOUT
            for (int it = s_used; it < s_issued; ++it) tc_wait(smem_u32(&full[it % ST]), (uint32_t)((it / ST) & 1));
        }
        __syncthreads();
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(2 * TCOLS));
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against the driver)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder()
{
    static std::once_flag once;
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    });
    return fn;
}

// rows x K bf16 operand with row stride ld elements, boxes of 64 K-elements x box_rows rows
bool tile_map(CUtensorMap *m, const bf16 *base, int rows, int K, int ld, int box_rows)
{
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (!enc || (uintptr_t)base % 16) return false;
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<bf16 *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int device_sms()
{
    static std::atomic<int> sms{0};
    int n = sms.load(std::memory_order_relaxed);
    if (n == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
        sms.store(n, std::memory_order_relaxed);
    }
    return n;
}

template <int TN>
cudaError_t gemm_tc(const GemmArgs &g, bool *used, cudaStream_t s)
{
    constexpr size_t smem = tc_smem<TN>();
    *used = false;
    CUtensorMap tA, tB;
    if (!tile_map(&tA, g.A, g.M, g.K, g.lda, TC_BM) || !tile_map(&tB, g.B, g.N, g.K, g.ldb, TN)) return cudaSuccess;
    static unsigned long long set_on = 0;    // devices on which the attribute has been raised
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(__atomic_load_n(&set_on, __ATOMIC_ACQUIRE) & bit)) {
        e = cudaFuncSetAttribute(gemm_tc_kernel<TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        __atomic_fetch_or(&set_on, bit, __ATOMIC_ACQ_REL);
    }
    const int64_t tiles = (int64_t)(g.M / TC_BM) * (g.N / TN);
    gemm_tc_kernel<TN><<<(int)std::min<int64_t>(tiles, device_sms()), TC_THREADS, smem, s>>>(tA, tB, g);
    *used = true;
    return cudaGetLastError();
}

// The tcgen05 kernel's tile width, 0 where the product is not its (small products keep the 64 x 64
// mma.sync kernel, whose many CTAs fill the device).  The width with the shortest run of the busiest
// SM: rounds of tiles, each as long as its columns and about 32 more (a narrow tile reads its rows of A
// from shared memory for fewer columns).
int tc_tile(const GemmArgs &g)
{
    const bool aligned = g.lda % 8 == 0 && g.ldb % 8 == 0 && (!g.Cf || g.ldcf % 4 == 0) && (!g.Cb || g.ldcb % 8 == 0) &&
                         g.lo_off % 8 == 0 && ((uintptr_t)g.bias | (uintptr_t)g.Cf | (uintptr_t)g.Cb) % 16 == 0;
    if (g.M % TC_BM || g.K % TC_BK || !aligned) return 0;
    const int64_t sms = device_sms(), mt = g.M / TC_BM;
    if (g.N % 64 || mt * (g.N / 64) < sms) return 0;
    int best = 0;
    int64_t cost = 0;
    for (int tn : {256, 192, 128, 64}) {
        if (g.N % tn) continue;
        const int64_t c = (mt * (g.N / tn) + sms - 1) / sms * (tn + 32);
        if (!best || c < cost) {
            best = tn;
            cost = c;
        }
    }
    return best;
}

// tcgen05 for the shapes it tiles (M multiple of 128, K of 64, N of 64, 16-byte aligned rows) with at
// least one tile per SM, the mma.sync kernel for the rest (and wherever a tensor map cannot be made)
cudaError_t gemm(const GemmArgs &g, cudaStream_t s)
{
    bool used = false;
    cudaError_t e = cudaSuccess;
    switch (tc_tile(g)) {
    case 256: e = gemm_tc<256>(g, &used, s); break;
    case 192: e = gemm_tc<192>(g, &used, s); break;
    case 128: e = gemm_tc<128>(g, &used, s); break;
    case 64: e = gemm_tc<64>(g, &used, s); break;
    default: break;
    }
    return e != cudaSuccess || used ? e : gemm_sync<EPI_FWD>(g, s);
}

// Transposed copies are made from 64 x 64 tiles in shared memory: the strided 2-byte stores of a
// thread-per-element pass touch a 32-byte sector each.
constexpr int TT = 64, TTL = TT + 2;             // tile, row stride (bf16)

// rows [c0, c0 + 64) of the transposed tile: 64 batch entries, 16 bytes a thread
__device__ __forceinline__ void store_tile_t(const bf16 (*t)[TTL], bf16 *out, int64_t ld, int64_t r0, int c0)
{
    for (int i = threadIdx.x; i < TT * (TT / 2); i += blockDim.x) {
        const int c = i / (TT / 2), r = (i % (TT / 2)) * 2;
        *reinterpret_cast<__nv_bfloat162 *>(out + (size_t)(c0 + c) * ld + r0 + r) = *reinterpret_cast<const __nv_bfloat162 *>(&t[c][r]);
    }
}

// X (fp32 [B][ldx], first nin used) -> split bf16 [B][2 ninp] (hi | lo) and its transpose
// [2 ninp][B]; pad zeroed.  One 64 x 64 tile per CTA (ninp and B are multiples of 64).
template <bool TR>
__global__ void __launch_bounds__(256) pack_input_kernel(const float *X, int ldx, int nin, int ninp, int64_t B, bf16 *Xb, bf16 *XbT)
{
    __shared__ bf16 th[TR ? TT : 1][TTL], tl[TR ? TT : 1][TTL];
    const int64_t b0 = (int64_t)blockIdx.x * TT;
    const int j0 = blockIdx.y * TT;
    for (int i = threadIdx.x; i < TT * TT / 2; i += blockDim.x) {
        const int r = i / (TT / 2), c = (i % (TT / 2)) * 2, j = j0 + c;
        const int64_t b = b0 + r;
        const float v0 = j < nin ? X[b * ldx + j] : 0.f, v1 = j + 1 < nin ? X[b * ldx + j + 1] : 0.f;
        const bf16 h0 = __float2bfloat16(v0), h1 = __float2bfloat16(v1);
        const bf16 l0 = __float2bfloat16(v0 - __bfloat162float(h0)), l1 = __float2bfloat16(v1 - __bfloat162float(h1));
        *reinterpret_cast<__nv_bfloat162 *>(Xb + b * 2 * ninp + j) = __halves2bfloat162(h0, h1);
        *reinterpret_cast<__nv_bfloat162 *>(Xb + b * 2 * ninp + ninp + j) = __halves2bfloat162(l0, l1);
        if (TR) {
            th[c][r] = h0;
            th[c + 1][r] = h1;
            tl[c][r] = l0;
            tl[c + 1][r] = l1;
        }
    }
    if (TR) {
        __syncthreads();
        store_tile_t(th, XbT, B, b0, j0);
        store_tile_t(tl, XbT, B, b0, ninp + j0);
    }
}

// g[o][k] = dW2[o][k] + dW2[o][in + k]: the weight gradient of the tied hi / lo halves
__global__ void fold_split_kernel(const float *dW2, int out, int in, float *g)
{
    const int64_t n = (int64_t)out * in;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i / in), k = (int)(i % in);
        g[i] = dW2[(size_t)o * 2 * in + k] + dW2[(size_t)o * 2 * in + in + k];
    }
}

// MSE loss over the first nout outputs (optionally weighted): loss = sum w_j (y - t)^2 / (B n_w),
// dY = 2 w_j (y - t) / (B n_w) in bf16 [B][noutp] and [noutp][B] (pad columns zero).  One 64 x 64 tile
// per CTA.
__global__ void __launch_bounds__(256) mse_kernel(const float *Y, int ldy_pred, const float *T, int ldt, const float *wmask, const float *roww,
                           int nout, int noutp, int64_t B, float inv_count, bf16 *dY, bf16 *dYT, float *loss)
{
    __shared__ bf16 th[TT][TTL];
    const int64_t b0 = (int64_t)blockIdx.x * TT;
    const int j0 = blockIdx.y * TT;
    float acc = 0.f;
    for (int i = threadIdx.x; i < TT * TT / 2; i += blockDim.x) {
        const int r = i / (TT / 2), c = (i % (TT / 2)) * 2;
        const int64_t b = b0 + r;
        bf16 h[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int j = j0 + c + e;
            float g = 0.f;
            if (j < nout) {
                const float w = (wmask ? wmask[j] : 1.f) * (roww ? roww[b] : 1.f);
                const float d = Y[b * ldy_pred + j] - T[b * ldt + j];
                acc += w * d * d;
                g = 2.f * w * d * inv_count;
            }
            h[e] = __float2bfloat16(g);
            th[c + e][r] = h[e];
        }
        *reinterpret_cast<__nv_bfloat162 *>(dY + b * noutp + j0 + c) = __halves2bfloat162(h[0], h[1]);
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ float red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    store_tile_t(th, dYT, B, b0, j0);
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        atomicAdd(loss, t * inv_count);
    }
}

// dPre = dA * (pre > 0), as bf16 [B][n] and [n][B]
__global__ void relu_back_kernel(const float *dA, const float *pre, int64_t B, int n, bf16 *dP, bf16 *dPT)
{
    const int64_t total = B * n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = i / n;
        const int j = (int)(i % n);
        const float g = pre[i] > 0.f ? dA[i] : 0.f;
        const bf16 h = __float2bfloat16(g);
        dP[i] = h;
        dPT[(size_t)j * B + b] = h;
    }
}

// db[j] = sum_b dYT[j][b]
__global__ void rowsum_kernel(const bf16 *dYT, int64_t B, int n, float *db)
{
    const int j = blockIdx.x;
    if (j >= n) return;
    float acc = 0.f;
    for (int64_t b = threadIdx.x; b < B; b += blockDim.x) acc += __bfloat162float(dYT[(size_t)j * B + b]);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    __shared__ float red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        db[j] = t;
    }
}

// Adam on a parameter block (fp32 master p), then the bf16 copies W[out][in] and W^T[in][out].
__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int64_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2, int out, int in, bf16 *Wb, bf16 *WbT)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        if (Wb) {
            const int o = (int)(i / in), k = (int)(i % in);
            const bf16 h = __float2bfloat16(pi);
            Wb[(size_t)o * 2 * in + k] = h;
            Wb[(size_t)o * 2 * in + in + k] = h;
            WbT[(size_t)k * out + o] = h;
        }
    }
}

__global__ void refresh_bf16_kernel(const float *p, int out, int in, bf16 *Wb, bf16 *WbT)
{
    const int64_t n = (int64_t)out * in;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(i / in), k = (int)(i % in);
        const bf16 h = __float2bfloat16(p[i]);
        Wb[(size_t)o * 2 * in + k] = h;
        Wb[(size_t)o * 2 * in + in + k] = h;
        WbT[(size_t)k * out + o] = h;
    }
}

int grid_for(int64_t n) { return (int)std::min<int64_t>((n + 255) / 256, 152 * 16); }

int pad64(int x) { return (x + 63) / 64 * 64; }

}  // namespace

// ------------------------------------------------------------------ MLP object --------------

struct ef_mlp_s {
    int nin, nh, nl, nout;          // nl = number of weight layers (>= 2)
    int ninp, noutp;                // padded to 64
    int64_t max_batch;
    std::vector<int> din, dout;     // padded fan-in / fan-out per layer
    std::vector<int64_t> woff, boff;
    int64_t nparams = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;     // fp32 master, grad, Adam
    std::vector<bf16 *> Wb, WbT;    // per layer [out][in], [in][out]
    // activations for max_batch
    bf16 *Xb = nullptr, *XbT = nullptr;
    std::vector<float *> pre;       // [B][out_l]
    std::vector<bf16 *> act, actT;  // [B][out_l], [out_l][B] (hidden layers)
    float *dA = nullptr;            // [B][max out] fp32
    float *dW2 = nullptr;           // [max out][2 max in] fp32: gradient of the split halves
    bf16 *dY[2] = {}, *dYT[2] = {}; // gradient at a layer's output and its transpose, layers in turn
    int64_t step = 0;
    int device = 0;
    int *status = nullptr;          // device status word (EF_ERR_TIMEOUT from a GEMM's bounded waits)
    int h_status = 0;
};

namespace {

ef_status mlp_fail(ef_status s, const std::string &m)
{
    ef::set_last_error(m.c_str());
    return s;
}

ef_status cuda_err(cudaError_t e, const char *what)
{
    std::string m = std::string(what) + ": " + cudaGetErrorString(e);
    ef::set_last_error(m.c_str());
    return e == cudaErrorMemoryAllocation ? EF_ERR_OOM : EF_ERR_CUDA;
}

void mlp_free(ef_mlp_s *n)
{
    if (!n) return;
    cudaFree(n->p);
    cudaFree(n->g);
    cudaFree(n->m);
    cudaFree(n->v);
    for (auto q : n->Wb) cudaFree(q);
    for (auto q : n->WbT) cudaFree(q);
    cudaFree(n->Xb);
    cudaFree(n->XbT);
    for (auto q : n->pre) cudaFree(q);
    for (auto q : n->act) cudaFree(q);
    for (auto q : n->actT) cudaFree(q);
    cudaFree(n->dA);
    cudaFree(n->dW2);
    for (int i = 0; i < 2; ++i) {
        cudaFree(n->dY[i]);
        cudaFree(n->dYT[i]);
    }
    cudaFree(n->status);
    delete n;
}

// forward pass for batch B (multiple of 64) from the packed input Xb
ef_status mlp_forward_packed(ef_mlp_s *n, const bf16 *Xb, int64_t B, float *Yout, int ldy, bool keep_T, cudaStream_t s)
{
    for (int l = 0; l < n->nl; ++l) {
        GemmArgs g{};
        g.A = l == 0 ? Xb : n->act[l - 1];
        g.lda = 2 * n->din[l];
        g.B = n->Wb[l];
        g.ldb = 2 * n->din[l];
        g.M = (int)B;
        g.N = n->dout[l];
        g.K = 2 * n->din[l];
        g.bias = n->p + n->boff[l];
        const bool last = l + 1 == n->nl;
        g.relu = last ? 0 : 1;
        g.Cf = last ? Yout : keep_T ? n->pre[l] : nullptr;     // hidden pre-activations: for the backward pass
        g.ldcf = last ? ldy : n->dout[l];
        g.Cb = last ? nullptr : n->act[l];
        g.ldcb = 2 * n->dout[l];
        g.CbT = (last || !keep_T) ? nullptr : n->actT[l];
        g.ldcbt = (int)B;
        g.lo_off = n->dout[l];
        g.status = n->status;
        cudaError_t e = gemm(g, s);
        if (e != cudaSuccess) return cuda_err(e, "mlp gemm");
    }
    return EF_OK;
}

}  // namespace

namespace ef {

ef_status mlp_forward_same_input(ef_mlp_t n, ef_mlp_t first, float *Y, int ldy, int64_t B, cudaStream_t s)
{
    if (n->ninp != first->ninp || B > n->max_batch || B > first->max_batch) return mlp_fail(EF_ERR_INVALID_ARG, "networks of one input");
    return mlp_forward_packed(n, first->Xb, B, Y, ldy, false, s);
}

}  // namespace ef

extern "C" {

ef_status ef_mlp_create(int nin, int nhidden, int nlayers, int nout, int64_t max_batch, uint64_t seed, ef_mlp_t *out)
{
    if (!out) return mlp_fail(EF_ERR_INVALID_ARG, "null output handle");
    *out = nullptr;
    if (nin < 1 || nhidden < 1 || nout < 1 || nlayers < 2 || max_batch < 64 || max_batch % 64)
        return mlp_fail(EF_ERR_INVALID_ARG, "need nin, nhidden, nout >= 1, nlayers >= 2, max_batch a positive multiple of 64");
    ef_mlp_s *n = new ef_mlp_s();
    n->nin = nin;
    n->nh = nhidden;
    n->nl = nlayers;
    n->nout = nout;
    n->ninp = pad64(nin);
    n->noutp = pad64(nout);
    n->max_batch = max_batch;
    cudaGetDevice(&n->device);
    const int nhp = pad64(nhidden);
    for (int l = 0; l < nlayers; ++l) {
        n->din.push_back(l == 0 ? n->ninp : nhp);
        n->dout.push_back(l + 1 == nlayers ? n->noutp : nhp);
    }
    for (int l = 0; l < nlayers; ++l) {
        n->woff.push_back(n->nparams);
        n->nparams += (int64_t)n->dout[l] * n->din[l];
        n->boff.push_back(n->nparams);
        n->nparams += n->dout[l];
    }
    // He-normal initialisation of the real (unpadded) weights, zero biases and padding
    std::vector<float> h((size_t)n->nparams, 0.f);
    std::mt19937_64 rng(seed);
    for (int l = 0; l < nlayers; ++l) {
        const int fin = l == 0 ? nin : nhidden, fout = l + 1 == nlayers ? nout : nhidden;
        std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / fin) * (l + 1 == nlayers ? 0.5 : 1.0));
        for (int o = 0; o < fout; ++o)
            for (int k = 0; k < fin; ++k) h[(size_t)(n->woff[l] + (int64_t)o * n->din[l] + k)] = (float)nd(rng);
    }
    cudaError_t e = cudaSuccess;
    auto alloc = [&](void **ptr, size_t bytes) {
        if (e == cudaSuccess) e = cudaMalloc(ptr, bytes);
        if (e == cudaSuccess) e = cudaMemset(*ptr, 0, bytes);
    };
    alloc((void **)&n->p, n->nparams * 4);
    alloc((void **)&n->g, n->nparams * 4);
    alloc((void **)&n->m, n->nparams * 4);
    alloc((void **)&n->v, n->nparams * 4);
    if (e == cudaSuccess) e = cudaMemcpy(n->p, h.data(), h.size() * 4, cudaMemcpyHostToDevice);
    n->Wb.assign(nlayers, nullptr);
    n->WbT.assign(nlayers, nullptr);
    n->pre.assign(nlayers, nullptr);
    n->act.assign(nlayers, nullptr);
    n->actT.assign(nlayers, nullptr);
    int maxd = 0;
    for (int l = 0; l < nlayers; ++l) {
        alloc((void **)&n->Wb[l], (size_t)n->dout[l] * 2 * n->din[l] * 2);
        alloc((void **)&n->WbT[l], (size_t)n->dout[l] * n->din[l] * 2);
        alloc((void **)&n->pre[l], (size_t)max_batch * n->dout[l] * 4);
        alloc((void **)&n->act[l], (size_t)max_batch * 2 * n->dout[l] * 2);
        alloc((void **)&n->actT[l], (size_t)max_batch * 2 * n->dout[l] * 2);
        maxd = std::max(maxd, std::max(n->dout[l], n->din[l]));
    }
    alloc((void **)&n->Xb, (size_t)max_batch * 2 * n->ninp * 2);
    alloc((void **)&n->XbT, (size_t)max_batch * 2 * n->ninp * 2);
    alloc((void **)&n->dW2, (size_t)maxd * 2 * maxd * 4);
    alloc((void **)&n->dA, (size_t)max_batch * maxd * 4);
    for (int i = 0; i < 2; ++i) {
        alloc((void **)&n->dY[i], (size_t)max_batch * maxd * 2);
        alloc((void **)&n->dYT[i], (size_t)max_batch * maxd * 2);
    }
    alloc((void **)&n->status, sizeof(int));
    if (e != cudaSuccess) {
        mlp_free(n);
        return cuda_err(e, "mlp allocation");
    }
    for (int l = 0; l < nlayers; ++l) {
        refresh_bf16_kernel<<<grid_for((int64_t)n->dout[l] * n->din[l]), 256>>>(n->p + n->woff[l], n->dout[l], n->din[l],
                                                                                n->Wb[l], n->WbT[l]);
    }
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        mlp_free(n);
        return cuda_err(e, "mlp init");
    }
    *out = n;
    return EF_OK;
}

ef_status ef_mlp_destroy(ef_mlp_t n)
{
    if (!n) return mlp_fail(EF_ERR_INVALID_ARG, "null mlp");
    mlp_free(n);
    return EF_OK;
}

ef_status ef_mlp_status(ef_mlp_t n, int sync, int reset)
{
    if (!n) return mlp_fail(EF_ERR_INVALID_ARG, "null mlp");
    if (sync) {
        cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return cuda_err(e, "device synchronize");
        e = cudaMemcpy(&n->h_status, n->status, sizeof(int), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return cuda_err(e, "status read");
        if (reset) {
            e = cudaMemset(n->status, 0, sizeof(int));
            if (e != cudaSuccess) return cuda_err(e, "status reset");
        }
    }
    const int st = n->h_status;
    if (reset) n->h_status = 0;
    return (ef_status)st;
}

ef_status ef_mlp_info(ef_mlp_t n, int64_t info[8])
{
    if (!n || !info) return mlp_fail(EF_ERR_INVALID_ARG, "null mlp or info");
    info[0] = n->nin;
    info[1] = n->nh;
    info[2] = n->nl;
    info[3] = n->nout;
    info[4] = n->nparams;
    info[5] = n->ninp;
    info[6] = n->noutp;
    info[7] = n->max_batch;
    return EF_OK;
}

ef_status ef_mlp_params(ef_mlp_t n, float *host, int set)
{
    if (!n || !host) return mlp_fail(EF_ERR_INVALID_ARG, "null mlp or buffer");
    cudaError_t e = set ? cudaMemcpy(n->p, host, n->nparams * 4, cudaMemcpyHostToDevice)
                        : cudaMemcpy(host, n->p, n->nparams * 4, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return cuda_err(e, "mlp params");
    if (set) {
        for (int l = 0; l < n->nl; ++l)
            refresh_bf16_kernel<<<grid_for((int64_t)n->dout[l] * n->din[l]), 256>>>(n->p + n->woff[l], n->dout[l],
                                                                                    n->din[l], n->Wb[l], n->WbT[l]);
        e = cudaDeviceSynchronize();
        if (e != cudaSuccess) return cuda_err(e, "mlp params");
    }
    return EF_OK;
}

ef_status ef_mlp_forward(ef_mlp_t n, const float *X, int ldx, float *Y, int ldy, int64_t B, ef_stream_t stream)
{
    if (!n || !X || !Y) return mlp_fail(EF_ERR_INVALID_ARG, "null mlp, X or Y");
    if (B < 0 || B % 64 || B > n->max_batch) return mlp_fail(EF_ERR_INVALID_ARG, "batch must be a multiple of 64 <= max_batch");
    if (ldx < n->nin || ldy < n->noutp || ldy % 2 || (uintptr_t)Y % 8)
        return mlp_fail(EF_ERR_INVALID_ARG, "ldx >= nin, ldy >= padded nout (even), Y 8-byte aligned");
    if (B == 0) return EF_OK;
    cudaStream_t s = (cudaStream_t)stream;
    pack_input_kernel<false><<<dim3((unsigned)(B / TT), n->ninp / TT), 256, 0, s>>>(X, ldx, n->nin, n->ninp, B, n->Xb, nullptr);
    return mlp_forward_packed(n, n->Xb, B, Y, ldy, false, s);
}

// loss and gradients (into the MLP's gradient buffer); optionally the Adam update
static ef_status mlp_grad_impl(ef_mlp_s *n, const float *X, int ldx, const float *T, int ldt, const float *wmask,
                               const float *roww, int64_t B, float *loss_dev, cudaStream_t s)
{
    pack_input_kernel<true><<<dim3((unsigned)(B / TT), n->ninp / TT), 256, 0, s>>>(X, ldx, n->nin, n->ninp, B, n->Xb, n->XbT);
    // forward (last layer's fp32 output into dA as scratch)
    ef_status st = mlp_forward_packed(n, n->Xb, B, n->dA, n->noutp, true, s);
    if (st != EF_OK) return st;
    cudaError_t e = cudaMemsetAsync(loss_dev, 0, sizeof(float), s);
    if (e != cudaSuccess) return cuda_err(e, "loss reset");
    mse_kernel<<<dim3((unsigned)(B / TT), n->noutp / TT), 256, 0, s>>>(n->dA, n->noutp, T, ldt, wmask, roww, n->nout, n->noutp, B,
                                                                        1.f / ((float)B * (float)n->nout), n->dY[0], n->dYT[0],
                                                                        loss_dev);
    int cur = 0;
    // backward
    for (int l = n->nl - 1; l >= 0; --l) {
        const int out = n->dout[l], in = n->din[l];
        // dW_l = dPre_l^T A_{l-1}:  M = out, N = in, K = B; A = dPreT [out][B], B = A_{l-1}^T [in][B]
        // (hi and lo halves: 2 in rows), folded to the gradient of the tied halves
        GemmArgs g{};
        g.A = n->dYT[cur];
        g.lda = (int)B;
        g.B = l == 0 ? n->XbT : n->actT[l - 1];
        g.ldb = (int)B;
        g.M = out;
        g.N = 2 * in;
        g.K = (int)B;
        g.status = n->status;
        g.Cf = n->dW2;
        g.ldcf = 2 * in;
        if (tc_tile(g)) {
            e = gemm(g, s);
            if (e != cudaSuccess) return cuda_err(e, "mlp grad gemm");
            fold_split_kernel<<<grid_for((int64_t)out * in), 256, 0, s>>>(n->dW2, out, in, n->g + n->woff[l]);
            rowsum_kernel<<<out, 256, 0, s>>>(n->dYT[cur], B, out, n->g + n->boff[l]);
        } else {
            g.Cf = n->g + n->woff[l];
            g.ldcf = in;
            g.db = n->g + n->boff[l];
            e = gemm_sync<EPI_DW>(g, s);
            if (e != cudaSuccess) return cuda_err(e, "mlp grad gemm");
        }
        if (l == 0) break;
        // dPre_{l-1} = (dPre_l W_l) masked by pre_{l-1} > 0:  M = B, N = in, K = out; A = dPre [B][out],
        // B = W^T [in][out].  The next layer's buffers: other CTAs still read this one's as operand.
        GemmArgs h{};
        h.A = n->dY[cur];
        h.lda = out;
        h.B = n->WbT[l];
        h.ldb = out;
        h.M = (int)B;
        h.N = in;
        h.K = out;
        h.Cf = n->dA;
        h.ldcf = in;
        h.status = n->status;
        if (tc_tile(h)) {
            e = gemm(h, s);
            if (e != cudaSuccess) return cuda_err(e, "mlp backprop gemm");
            relu_back_kernel<<<grid_for(B * in), 256, 0, s>>>(n->dA, n->pre[l - 1], B, in, n->dY[cur ^ 1], n->dYT[cur ^ 1]);
        } else {
            h.Cf = nullptr;
            h.pre = n->pre[l - 1];
            h.ldpre = in;
            h.Cb = n->dY[cur ^ 1];
            h.ldcb = in;
            h.CbT = n->dYT[cur ^ 1];
            h.ldcbt = (int)B;
            e = gemm_sync<EPI_DA>(h, s);
            if (e != cudaSuccess) return cuda_err(e, "mlp backprop gemm");
        }
        cur ^= 1;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_err(e, "mlp backward");
    return EF_OK;
}

ef_status ef_mlp_grad(ef_mlp_t n, const float *X, int ldx, const float *T, int ldt, const float *wmask,
                      const float *rowweight, int64_t B, float *loss_dev, float *grad_dev, ef_stream_t stream)
{
    if (!n || !X || !T || !loss_dev) return mlp_fail(EF_ERR_INVALID_ARG, "null argument");
    if (B <= 0 || B % 64 || B > n->max_batch) return mlp_fail(EF_ERR_INVALID_ARG, "batch must be a multiple of 64 <= max_batch");
    if (ldx < n->nin || ldt < n->nout) return mlp_fail(EF_ERR_INVALID_ARG, "ldx >= nin, ldt >= nout");
    cudaStream_t s = (cudaStream_t)stream;
    ef_status st = mlp_grad_impl(n, X, ldx, T, ldt, wmask, rowweight, B, loss_dev, s);
    if (st != EF_OK) return st;
    if (grad_dev) {
        cudaError_t e = cudaMemcpyAsync(grad_dev, n->g, n->nparams * 4, cudaMemcpyDeviceToDevice, s);
        if (e != cudaSuccess) return cuda_err(e, "grad copy");
    }
    return EF_OK;
}

ef_status ef_mlp_train_step(ef_mlp_t n, const float *X, int ldx, const float *T, int ldt, const float *wmask,
                            const float *rowweight, int64_t B, float lr, float *loss_dev, ef_stream_t stream)
{
    ef_status st = ef_mlp_grad(n, X, ldx, T, ldt, wmask, rowweight, B, loss_dev, nullptr, stream);
    if (st != EF_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;
    n->step += 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - std::pow(b1, (float)n->step), c2 = 1.f - std::pow(b2, (float)n->step);
    for (int l = 0; l < n->nl; ++l) {
        const int64_t nw = (int64_t)n->dout[l] * n->din[l];
        adam_kernel<<<grid_for(nw), 256, 0, s>>>(n->p + n->woff[l], n->g + n->woff[l], n->m + n->woff[l],
                                                 n->v + n->woff[l], nw, lr, b1, b2, eps, c1, c2, n->dout[l], n->din[l],
                                                 n->Wb[l], n->WbT[l]);
        adam_kernel<<<grid_for(n->dout[l]), 256, 0, s>>>(n->p + n->boff[l], n->g + n->boff[l], n->m + n->boff[l],
                                                         n->v + n->boff[l], n->dout[l], lr, b1, b2, eps, c1, c2, 0, 1,
                                                         nullptr, nullptr);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_err(e, "adam");
    return EF_OK;
}

}  // extern "C"
