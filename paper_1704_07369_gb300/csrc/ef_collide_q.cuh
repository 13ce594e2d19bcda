// ef_collide_q.cuh -- the FP64 collision kernel: four lanes per line transform (one thread-block
// cluster per cell).
//
// Same operations and memory plan as collide_kernel (forward spectrum in the cluster's L2-resident
// workspace, spectral slabs in shared memory, S / G accumulators in shared or global memory, the op
// lists of ef_internal.h), laid out for an FP64 pipe that takes one warp instruction per sub-partition
// every 64 cycles (2 FP64 lanes a cycle and SM):
//   * that pipe is the bound, so everything else (shuffles, table loads, bank conflicts) hides behind
//     it as long as every sub-partition has a warp with FP64 work.  A line is transformed by four
//     lanes, N / 4 values each: the transform of N = 64 takes 64 registers in place of 256 (which
//     spilled), a CTA runs up to 16 warps, and the few lines of a small cell still reach all four
//     sub-partitions;
//   * the modes with a component -N/2 vanish in every multiplier (sigma_N(-N/2) = 0, Sec. 4.1), so the
//     column k_x = -N/2 is neither stored nor transformed: N/2 columns and N^(d-1)/2 pencils fill the
//     warps evenly where N/2 + 1 left a nearly empty last round.
// Lane s of a team holds the line's values 4 m + s, transforms them locally (length N/4), multiplies by
// exp(+-2 pi i s k / N) and finishes with a radix-4 butterfly across the team (two shuffle exchanges);
// it then holds the outputs k + (N/4) t(s), k < N/4, t the bit reversal of s: a contiguous block.
//
// Measured against one thread per line with N/2 + 1 columns (both split alike, with the first finishing kernel): Q of 24
// cells of N = 64 13.3 -> 10.4 ms (of which the FP64 pipe needs 5.8 ms on all SMs, 7.9 on the 112 that the
// 7 resident clusters of 16 reach), two Euler steps of one cell of N = 32 1.11 -> 0.925 ms, 100 steps of one 2D
// cell of N = 16 4.7 -> 2.87 ms, two SSP-RK3 steps of four 2D cells of N = 64 1.17 -> 0.87 ms.
#pragma once

#include "ef_collide_impl.cuh"

namespace ef {

constexpr int kQuadThreads = 512;

// row stride of a slab plane (complex values): odd, N/2 stored
template <int N>
__host__ __device__ constexpr int quad_row() { return N / 2 + 1; }

template <int D, int N>
__host__ __device__ constexpr size_t quad_smem(int planes, int sg_global, int paired)
{
    constexpr int N1 = (D == 3) ? N : 1;
    const size_t is = (size_t)(paired ? 2 : 1) * planes * N1 * quad_row<N>() * sizeof(C2<double>);
    const size_t sg = sg_global ? 0 : (size_t)(paired ? 1 : 2) * planes * N1 * N * sizeof(double);
    // diagnostics, cell index and flag, plane addresses, team twiddles
    return is + sg + (32 + 1) * kDiag * sizeof(double) + 16 + (N + N % 4) * sizeof(uint32_t) + N * sizeof(C2<double>);
}

__device__ __forceinline__ double flip_sign(double x, bool neg)
{
    return __hiloint2double(__double2hiint(x) ^ (neg ? (int)0x80000000 : 0), __double2loint(x));
}

// output block of lane s
__device__ __forceinline__ int quad_block(int s) { return ((s & 1) << 1) | (s >> 1); }

// length-N transform of a team's line (see above); tw[s * N/4 + k] = exp(-2 pi i s k / N)
template <int N, int SIGN>
__device__ __forceinline__ void quad_fft(C2<double> (&v)[N / 4], const C2<double> *tw, int s)
{
    constexpr int M = N / 4;
    fft<M, SIGN, N>(v);
#pragma unroll
    for (int k = 1; k < M; ++k) {
        C2<double> w = tw[s * M + k];
        if (SIGN > 0) w.y = -w.y;
        v[k] = cmul(v[k], w);
    }
    const bool hi = s & 2, odd = s & 1, last = s == 3;
#pragma unroll
    for (int k = 0; k < M; ++k) {
        // t0 + t2 | t1 + t3 | t0 - t2 | t1 - t3 in lanes 0 .. 3
        double x = __shfl_xor_sync(0xffffffffu, v[k].x, 2) + flip_sign(v[k].x, hi);
        double y = __shfl_xor_sync(0xffffffffu, v[k].y, 2) + flip_sign(v[k].y, hi);
        // lane 3: SIGN i (t1 - t3)
        const double xr = last ? flip_sign(y, SIGN > 0) : x, yr = last ? flip_sign(x, SIGN < 0) : y;
        v[k].x = __shfl_xor_sync(0xffffffffu, xr, 1) + flip_sign(xr, odd);
        v[k].y = __shfl_xor_sync(0xffffffffu, yr, 1) + flip_sign(yr, odd);
    }
}

// two Hermitian half rows (k < N/2; zero at k = N/2) -> this lane's part of IFFT(R0) + i IFFT(R1)
template <int N>
__device__ __forceinline__ void quad_rows(const C2<double> *R0, const C2<double> *R1, const C2<double> *tw, int s,
                                          C2<double> (&z)[N / 4])
{
#pragma unroll
    for (int m = 0; m < N / 4; ++m) {
        const int k = 4 * m + s;
        const bool up = k > N / 2;
        const int kk = up ? N - k : k;
        const C2<double> a = R0[kk], b = R1[kk];       // kk = N/2 reads the row's pad, not used
        z[m].x = a.x + flip_sign(b.y, !up);
        z[m].y = b.x + flip_sign(a.y, up);
        if (k == 0) z[m] = C2<double>{a.x, b.x};
        if (k == N / 2) z[m] = C2<double>{0.0, 0.0};
    }
    quad_fft<N, 1>(z, tw, s);
}

template <int M>
__device__ __forceinline__ void quad_load(const double *src, double (&x)[M])
{
    if constexpr (M % 2 == 0) {
#pragma unroll
        for (int i = 0; i < M; i += 2) {
            const double2 v = *reinterpret_cast<const double2 *>(src + i);
            x[i] = v.x;
            x[i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i) x[i] = src[i];
    }
}
template <int M>
__device__ __forceinline__ void quad_store(double *dst, const double (&x)[M])
{
    if constexpr (M % 2 == 0) {
#pragma unroll
        for (int i = 0; i < M; i += 2) *reinterpret_cast<double2 *>(dst + i) = make_double2(x[i], x[i + 1]);
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i) dst[i] = x[i];
    }
}

// emit_row for a lane's block of M values starting at x0
template <int D, int N>
__device__ __forceinline__ bool quad_emit(const CollideArgs &a, const double (&fr)[N / 4], double *O, double (&q)[N / 4],
                                          int64_t grow, int x0, bool live, Diag &dg)
{
    constexpr int N1 = (D == 3) ? N : 1, M = N / 4;
    const int jz = (int)(grow / N1) - N / 2;
    const int jy = (D == 3) ? (int)(grow % N1) - N / 2 : 0;
    double s_m = 0, s_mx = 0, s_e2 = 0, s_eta = 0, s_prod = 0;
    double mn_f = fr[0], mn_out = 3.0e38;
    bool bad = false, neg = false;
#pragma unroll
    for (int n = 0; n < M; ++n) {
        const double f = fr[n], qv = q[n];
        double outv = qv;
        if (a.out_mode == OUT_EULER) {
            outv = f + a.dt * qv;
            if (outv < 0.0) neg = true;
        }
        q[n] = outv;
        if (!isfinite(outv)) bad = true;
        if (a.diag) {
            const double jx = (double)(x0 + n - N / 2);
            s_m += f;
            s_mx += f * jx;
            s_e2 += f * jx * jx;
            if (f > 0.0) {
                const double lf = log(f);
                s_eta += f * lf;
                s_prod += qv * lf;
            }
            mn_f = f < mn_f ? f : mn_f;
            mn_out = outv < mn_out ? outv : mn_out;
        }
    }
    if (!live) return false;
    quad_store<M>(O, q);
    if (bad) record_status(a.status, 7);     // EF_ERR_NOT_FINITE
    if (a.diag) dg.template add_row<D, double>(s_m, s_mx, s_e2, s_eta, s_prod, jz, jy, mn_f, mn_out);
    return neg;
}

template <int D, int N>
__global__ void __launch_bounds__(kQuadThreads, 1) collide_kernel_q(const CollideArgs a)
{
    using T = double;
    constexpr int H = N / 2 + 1, NH = N / 2;        // multiplier table columns, stored columns
    constexpr int N1 = (D == 3) ? N : 1;
    constexpr int NP = N1 * NH;                     // pencils
    constexpr int RS = quad_row<N>(), NPP = N1 * RS;
    constexpr int NPT = N1 * H;
    constexpr int M = N / 4;
    constexpr int64_t CELL = (int64_t)N * N1 * N;

    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    const int P = a.planes;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const int s = tid & 3, team = tid >> 2, nteam = nt >> 2;
    const int xb = M * quad_block(s);               // first output index of this lane
    Sync bar{cl, C};
    const int rows = P * N1, npairs = rows / 2;
    const int nbuf = a.paired ? 2 : 1;

    extern __shared__ __align__(16) unsigned char smem_raw[];
    C2<T> *Is0 = reinterpret_cast<C2<T> *>(smem_raw);
    C2<T> *Is1 = Is0 + (size_t)P * NPP;             // paired mode only
    C2<T> *tw = Is0 + (size_t)nbuf * P * NPP;       // [4][N/4]
    T *acc = reinterpret_cast<T *>(tw + N);
    T *Sb = nullptr, *Gb;
    if (a.sg_global) {
        T *base = reinterpret_cast<T *>(a.sg_ws) + (int64_t)blockIdx.x * 2 * rows * N;
        Sb = base;
        Gb = base + (int64_t)rows * N;
    } else {
        if (!a.paired) {
            Sb = acc;
            acc += (size_t)rows * N;
        }
        Gb = acc;
        acc += (size_t)rows * N;
    }
    double *part = acc;                                             // [32 warps + 1][kDiag]
    long long *s_cell = reinterpret_cast<long long *>(part + (32 + 1) * kDiag);
    int *s_nubig = reinterpret_cast<int *>(s_cell + 1);
    uint32_t *zt = reinterpret_cast<uint32_t *>(s_cell + 2);        // [N] cluster address of each plane
    const uint32_t slab1 = (uint32_t)((size_t)P * NPP * sizeof(C2<T>));
    {
        const uint32_t base0 = smem_u32addr(Is0);
        for (int z = tid; z < N; z += nt) zt[z] = cluster_map(base0 + (uint32_t)((z % P) * NPP * sizeof(C2<T>)), z / P);
        for (int j = tid; j < N; j += nt) {
            const int e = (j / M) * (j % M);        // < N
            tw[j] = tw_value<N, T>(e);
        }
    }
    __syncthreads();

    const int64_t nclusters = gridDim.x / C;
    const int64_t cid = blockIdx.x / C;
    const int NPC = a.npc;
    C2<T> *Fh = reinterpret_cast<C2<T> *>(a.fh_ws) + cid * (int64_t)N * NP;
    const T scale = T(1) / T(CELL);
    const T *Mbase = reinterpret_cast<const T *>(a.mult);
    auto rounds = [&](int n) { return (n + nteam - 1) / nteam; };

    const int64_t ncells = a.dev_ncells ? (int64_t)*a.dev_ncells : a.ncells;
    const int S = a.nsplit;                         // parts per cell, each with its share of the ops
    const int64_t nwork = ncells * S;
    int64_t w = cid - nclusters;
    for (;;) {
        if (a.counter) {            // dynamic: the cluster takes the next unclaimed item
            if (rank == 0 && tid == 0) *s_cell = (long long)atomicAdd(a.counter, 1ULL);
            bar.full();
            w = *cl.map_shared_rank(s_cell, 0);
        } else {
            w += nclusters;
        }
        if (w >= nwork) break;
        const int64_t c = S > 1 ? w / S : w;
        const int prt = S > 1 ? (int)(w - c * S) : 0;
        int o0, o1;
        split_range(a, prt, o0, o1);
        T *pnu = nullptr, *pg = nullptr;            // split: nu of the cell, this part's gain
        if (S > 1) {
            pnu = reinterpret_cast<T *>(a.part) + (c * (S + 1) + S) * CELL;
            pg = reinterpret_cast<T *>(a.part) + (c * (S + 1) + prt) * CELL;
            if (rank == 0 && tid == 0 && (a.paired ? o0 == 0 : o1 == a.nops)) fin_flags(a)[c] = 0;
        }
        const int64_t coff = a.cell_off ? a.cell_off[c] : c * CELL;
        const int64_t cglob = a.cell_id ? a.cell_id[c] : c;
        const T *F = reinterpret_cast<const T *>(a.F) + coff;
        T *Out = reinterpret_cast<T *>(a.Q) + coff;
        if (tid == 0) *s_nubig = 0;

        // ---------------- F1: two real rows a team as one complex line; the transform goes to the two
        // rows' storage (N + 2 values) and is split there into the half spectra
        for (int it = 0, nr = rounds(npairs); it < nr; ++it) {
            const int q = it * nteam + team;
            const bool has = q < npairs;
            const int r0 = has ? q : 0, r1 = r0 + npairs;
            const T *s0 = F + ((int64_t)rank * rows + r0) * N, *s1 = F + ((int64_t)rank * rows + r1) * N;
            C2<T> v[M];
#pragma unroll
            for (int m = 0; m < M; ++m) v[m] = C2<T>{s0[4 * m + s], s1[4 * m + s]};
            quad_fft<N, -1>(v, tw, s);
            C2<T> *d0 = Is0 + (r0 / N1) * NPP + (r0 % N1) * RS, *d1 = Is0 + (r1 / N1) * NPP + (r1 % N1) * RS;
            if (has) {
#pragma unroll
                for (int k = 0; k < M; ++k) (xb + k < RS ? d0 : d1 - RS)[xb + k] = v[k];
            }
            __syncwarp();
            constexpr int MK = (NH + 3) / 4;
            C2<T> X0[MK], X1[MK];
#pragma unroll
            for (int j = 0; j < MK; ++j) {
                const int k = 4 * j + s;
                if (k < NH) {
                    const int kc = k == 0 ? 0 : N - k;
                    const C2<T> p = (k < RS ? d0 : d1 - RS)[k], g = (kc < RS ? d0 : d1 - RS)[kc];
                    X0[j] = C2<T>{0.5 * (p.x + g.x), 0.5 * (p.y - g.y)};
                    X1[j] = C2<T>{0.5 * (p.y + g.y), -0.5 * (p.x - g.x)};
                }
            }
            __syncwarp();
#pragma unroll
            for (int j = 0; j < MK; ++j) {
                const int k = 4 * j + s;
                if (has && k < NH) {
                    d0[k] = X0[j];
                    d1[k] = X1[j];
                }
            }
            __syncwarp();
        }
        auto columns = [&](C2<T> *slab0, C2<T> *slab1p, int ncol, auto sign) {
            constexpr int SG = decltype(sign)::value;
            for (int it = 0, nr = rounds(ncol); it < nr; ++it) {
                const int q = it * nteam + team;
                const bool has = q < ncol;
                const int qc = has ? q : 0;
                const int b = qc >= P * NH, rem = qc - b * P * NH;
                C2<T> *col = (b ? slab1p : slab0) + (size_t)(rem / NH) * NPP + rem % NH;
                C2<T> v[M];
#pragma unroll
                for (int m = 0; m < M; ++m) v[m] = col[(4 * m + s) * RS];
                quad_fft<N, SG>(v, tw, s);
                __syncwarp();
                if (has) {
#pragma unroll
                    for (int k = 0; k < M; ++k) col[(xb + k) * RS] = v[k];
                }
            }
        };
        if constexpr (D == 3) {
            __syncthreads();
            columns(Is0, Is0, P * NH, IntC<-1>{});
        }
        bar.full();

        // ---------------- F2: own pencils, gathered, axis 0 forward, to the cluster's workspace
        for (int it = 0, nr = rounds(NPC); it < nr; ++it) {
            const int ql = it * nteam + team;
            const bool has = ql < NPC && rank * NPC + ql < NP;
            const int p = has ? rank * NPC + ql : 0;
            const uint32_t off = (uint32_t)(((p / NH) * RS + p % NH) * sizeof(C2<T>));
            C2<T> v[M];
#pragma unroll
            for (int m = 0; m < M; ++m) ld_cluster(zt[4 * m + s] + off, v[m]);
            quad_fft<N, -1>(v, tw, s);
            if (has) {
#pragma unroll
                for (int k = 0; k < M; ++k) Fh[(size_t)(xb + k) * NP + p] = cscale(v[k], scale);
            }
        }
        bar.full();

        Diag dg;
        dg.reset();
        bool have_g = false;                        // single mode, split: G already set in this part
        unsigned found = 0;                         // single-slab Euler step: what this thread's rows show

        for (int o = o0; o < o1; ++o) {
            const Op op = a.ops[o];
            const bool pair = op.kind >= OP_PAIR;
            // ---------------- A: multiply, axis 0 inverse, scatter to the owners' slabs
            const int nitems = (pair ? 2 : 1) * NPC;
            bool held = o > o0;
            for (int it = 0, nr = rounds(nitems); it < nr; ++it) {
                const int q = it * nteam + team;
                const int b = q >= NPC && pair;
                const int p0 = rank * NPC + (q - b * NPC);
                const bool has = q < nitems && p0 < NP;
                const int p = has ? p0 : 0;
                const int ky = p / NH, kx = p % NH;
                const T *Mu = Mbase + (size_t)(b ? op.dir2 : op.dir) * N * NPT + ky * H + kx;
                C2<T> v[M];
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    const int z = 4 * m + s;
                    v[m] = cscale(Fh[(size_t)z * NP + p], __ldg(Mu + (size_t)z * NPT));
                }
                quad_fft<N, 1>(v, tw, s);
                // only the scatter waits for the other CTAs' reads of the previous op
                if (held) {
                    __syncwarp();
                    bar.war_wait();
                    held = false;
                }
                const uint32_t off = (b ? slab1 : 0u) + (uint32_t)((ky * RS + kx) * sizeof(C2<T>));
                if (has) {
#pragma unroll
                    for (int k = 0; k < M; ++k) st_cluster(zt[xb + k] + off, v[k]);
                }
            }
            if (held) bar.war_wait();
            bar.full();

            // ---------------- B: axis 1 inverse
            if constexpr (D == 3) {
                columns(Is0, Is1, (pair ? 2 : 1) * P * NH, IntC<1>{});
                __syncthreads();
            }
            if (pair) {
                const bool last = op.kind == OP_PAIR_LAST && S == 1;
                const bool fresh = S > 1 && !have_g;
                const bool big = *s_nubig != 0;
                for (int it = 0, nr = rounds(rows); it < nr; ++it) {
                    const int q = it * nteam + team;
                    const bool has = q < rows;
                    const int r = has ? q : 0;
                    const int ro = (r / N1) * NPP + (r % N1) * RS;
                    C2<T> z[M];
                    quad_rows<N>(Is0 + ro, Is1 + ro, tw, s, z);
                    T *Gr = Gb + r + (size_t)xb * rows;
                    if (!last) {
                        if (has) {
#pragma unroll
                            for (int n = 0; n < M; ++n) Gr[n * rows] = (fresh ? T(0) : Gr[n * rows]) + z[n].x * z[n].y;
                        }
                    } else {
                        const int64_t grow = (int64_t)rank * rows + r;
                        T qv[M], fr[M];
#pragma unroll
                        for (int n = 0; n < M; ++n) qv[n] = Gr[n * rows] + z[n].x * z[n].y;
                        quad_load<M>(F + grow * N + xb, fr);
                        if (quad_emit<D, N>(a, fr, Out + grow * N + xb, qv, grow, xb, has, dg) && big) record_status(a.status, 6);
                    }
                }
                have_g = true;
            } else {
                for (int it = 0, nr = rounds(npairs); it < nr; ++it) {
                    const int q = it * nteam + team;
                    const bool has = q < npairs;
                    const int r0 = has ? q : 0, r1 = r0 + npairs;
                    C2<T> z[M];                     // (row r0, row r1) at x = xb + n
                    quad_rows<N>(Is0 + (r0 / N1) * NPP + (r0 % N1) * RS, Is0 + (r1 / N1) * NPP + (r1 % N1) * RS, tw, s, z);
                    T *S0 = Sb + r0 + (size_t)xb * rows, *S1 = Sb + r1 + (size_t)xb * rows;
                    T *G0 = Gb + r0 + (size_t)xb * rows, *G1 = Gb + r1 + (size_t)xb * rows;
                    const T wt = T(op.w);
                    if (op.kind <= OP_S_ADD) {
                        if (has) {
#pragma unroll
                            for (int n = 0; n < M; ++n) {
                                const bool set = op.kind == OP_S_SET;
                                S0[n * rows] = (set ? T(0) : S0[n * rows]) + wt * z[n].x;
                                S1[n * rows] = (set ? T(0) : S1[n * rows]) + wt * z[n].y;
                            }
                        }
                    } else if (op.kind <= OP_G_ADD) {
                        const bool set = op.kind == OP_G_SET || (S > 1 && !have_g);
                        if (has) {
#pragma unroll
                            for (int n = 0; n < M; ++n) {
                                G0[n * rows] = (set ? T(0) : G0[n * rows]) + z[n].x * S0[n * rows];
                                G1[n * rows] = (set ? T(0) : G1[n * rows]) + z[n].y * S1[n * rows];
                            }
                        }
                    } else {
                        // the loss: split, nu to the workspace; paired, G = -F nu; single (last), Q = G - F nu
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            const int64_t grow = (int64_t)rank * rows + (half ? r1 : r0);
                            T *Gr = half ? G1 : G0;
                            T nu[M], fr[M], qv[M];
#pragma unroll
                            for (int n = 0; n < M; ++n) nu[n] = half ? z[n].y : z[n].x;
                            if (S > 1) {
                                bool over = false;
#pragma unroll
                                for (int n = 0; n < M; ++n)
                                    if (a.dt * nu[n] > 1.0) over = true;
                                if (has) quad_store<M>(pnu + grow * N + xb, nu);
                                if (has && over && a.out_mode == OUT_EULER) fin_flags(a)[c] = 1;
                                continue;
                            }
                            quad_load<M>(F + grow * N + xb, fr);
                            T mx = nu[0];
                            bool big = false;
#pragma unroll
                            for (int n = 0; n < M; ++n) {
                                mx = nu[n] > mx ? nu[n] : mx;
                                if (a.dt * nu[n] > 1.0) big = true;
                            }
                            if (has) dg.max_nu = fmax(dg.max_nu, mx);
                            if (op.kind == OP_NU_INIT) {
                                if (has) {
#pragma unroll
                                    for (int n = 0; n < M; ++n) Gr[n * rows] = -fr[n] * nu[n];
                                    if (big && a.out_mode == OUT_EULER) flag_cluster(s_nubig, C, 0, 1u);
                                }
                            } else {
#pragma unroll
                                for (int n = 0; n < M; ++n) qv[n] = Gr[n * rows] - fr[n] * nu[n];
                                if (has && big) found |= 2;
                                if (quad_emit<D, N>(a, fr, Out + grow * N + xb, qv, grow, xb, has, dg)) found |= 1;
                            }
                        }
                    }
                }
                if (op.kind == OP_G_SET || op.kind == OP_G_ADD) have_g = true;
            }
            bar.war_arrive();
            if (o + 1 == o1) bar.war_wait();
        }

        if (S > 1) {
            // this part's gain (a part with only the loss leaves zeros)
            __syncthreads();
            for (int it = 0, nr = rounds(rows); it < nr; ++it) {
                const int r = it * nteam + team;
                if (r < rows) {
                    T g[M];
#pragma unroll
                    for (int n = 0; n < M; ++n) g[n] = have_g ? Gb[r + (size_t)(xb + n) * rows] : T(0);
                    quad_store<M>(pg + ((int64_t)rank * rows + r) * N + xb, g);
                }
            }
            __syncthreads();                        // G is rewritten by the next item
            continue;
        }

        if (!a.paired && a.out_mode == OUT_EULER) meet_positivity(a, found, cl, bar, rank, tid, s_nubig);
        // ---------------- per-cell FP64 reduction of the diagnostics
        if (a.diag) diag_reduce_f64<D>(a, dg, part, lane, tid, nt, rank, C, bar, cl, cglob);
    }
    bar.war();   // no CTA leaves while a peer may still read its shared memory
}

}  // namespace ef
