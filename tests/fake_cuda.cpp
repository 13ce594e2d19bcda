// A CUDA runtime on the host for the plan code (ef_plan.cpp) alone: device memory is host memory,
// streams and events are numbers, kernel launches are recorded instead of run.  Compiled together with
// ef_plan.cpp by tests/test_host_plan.py.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "ef.h"
#include "ef_launch.h"

// What happened, in order: launches (of a collide or finishing kernel), event records and waits.
struct FakeRec {
    int64_t kind;        // 0 collide, 1 finish, 2 event record, 3 event wait, 4 other kernel
    int64_t stream, event;
    int64_t N, ncells, cells_off, nsplit, cluster, threads, occ, sg_global, clusters;
    int64_t fh, sg, part, fin, paired, prefetch;
};

namespace {

std::vector<FakeRec> g_log;
std::map<void *, size_t> g_mem;
size_t g_used = 0, g_peak = 0, g_limit = (size_t)1 << 40;
double g_clock = 0.0;
cudaError_t g_error = cudaSuccess;
std::map<cudaStream_t, unsigned long long> g_capture;            // capturing streams
std::map<unsigned long long, std::vector<cudaUserObject_t>> g_graphs;
intptr_t g_next = 0x1000;
int g_smem_max = 227 * 1024;

struct Obj {
    void *p;
    cudaHostFn_t fn;
};
std::map<cudaEvent_t, double> g_event;

void rec(int64_t kind, cudaStream_t s, cudaEvent_t e)
{
    FakeRec r{};
    r.kind = kind;
    r.stream = (int64_t)(intptr_t)s;
    r.event = (int64_t)(intptr_t)e;
    g_log.push_back(r);
}

cudaError_t launch(int64_t kind, int N, const ef::CollideArgs &a, int grid, int tpb, int occ, cudaStream_t s)
{
    FakeRec r{};
    r.kind = kind;
    r.stream = (int64_t)(intptr_t)s;
    r.N = N;
    r.ncells = a.ncells;
    r.cells_off = a.cell_off != nullptr;
    r.nsplit = a.nsplit;
    r.cluster = a.cluster;
    r.threads = tpb;
    r.occ = occ;
    r.sg_global = a.sg_global;
    r.clusters = grid;
    r.fh = (int64_t)(intptr_t)a.fh_ws;
    r.sg = (int64_t)(intptr_t)a.sg_ws;
    r.part = (int64_t)(intptr_t)a.part;
    r.fin = (int64_t)(intptr_t)a.fin;
    r.paired = a.paired;
    r.prefetch = a.prefetch;
    g_log.push_back(r);
    g_clock += kind == 0 ? 1.0 / a.nsplit + 0.001 * a.cluster : 0.01;      // split launches tune as the faster ones
    return cudaSuccess;
}

// resident clusters as a GB300 would have them: 152 SMs, 228 KB each, 64K registers (128 a thread, 32 for the
// smallest cells; the register kernels one CTA per SM), at most 32 CTAs
int resident(int N, size_t smem, int cluster, int tpb, bool one_per_sm)
{
    const int regs = N <= 8 ? 32 : 128;
    int per_sm = one_per_sm ? 1 : std::min<int>(32, std::min<int>((int)(228 * 1024 / (smem + 1024)), 65536 / (regs * tpb)));
    return per_sm * 152 / cluster;
}

size_t smem_bytes(int el, int d, int N, int planes, int sg, int paired)
{
    const size_t rows = (size_t)planes * (d == 3 ? N : 1);
    return (paired ? 2 : 1) * rows * (N / 2 + 1) * 2 * el + (sg ? 0 : (paired ? 1 : 2) * rows * N * el) + 4096;
}
size_t rg_smem(int N, int planes) { return (size_t)2 * planes * N * (N / 2 + 2) * 8 + (size_t)N * planes * N / 2 * 8 + 4096; }

}  // namespace

extern "C" {

int64_t fake_log(FakeRec *out, int64_t n)
{
    const int64_t m = std::min<int64_t>(n, (int64_t)g_log.size());
    std::copy(g_log.begin(), g_log.begin() + m, out);
    return (int64_t)g_log.size();
}
void fake_clear(void) { g_log.clear(); }
void fake_limit(size_t bytes) { g_limit = bytes; }
size_t fake_used(void) { return g_used; }
size_t fake_peak(void)
{
    const size_t p = g_peak;
    g_peak = g_used;
    return p;
}
void fake_begin_capture(void *s, unsigned long long id)
{
    g_capture[(cudaStream_t)s] = id;
    g_graphs[id];
}
void fake_end_capture(void *s) { g_capture.erase((cudaStream_t)s); }
void fake_destroy_graph(unsigned long long id)
{
    for (cudaUserObject_t o : g_graphs[id]) {
        Obj *q = reinterpret_cast<Obj *>(o);
        q->fn(q->p);
        delete q;
    }
    g_graphs.erase(id);
}

cudaError_t cudaMalloc(void **p, size_t n)
{
    if (g_used + n > g_limit) return g_error = cudaErrorMemoryAllocation;
    *p = std::aligned_alloc(256, (n + 255) / 256 * 256 + 256);
    g_mem[*p] = n;
    g_used += n;
    g_peak = std::max(g_peak, g_used);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    if (!p) return cudaSuccess;
    if (!g_mem.count(p)) return cudaErrorInvalidValue;
    g_used -= g_mem[p];
    g_mem.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
// large workspaces are not touched: nothing reads them
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    std::memset(d, v, std::min<size_t>(n, 1 << 20));
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d)
{
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : g_smem_max;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    std::memset(p, 0, sizeof *p);
    std::strcpy(p->name, "fake");
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void)
{
    const cudaError_t e = g_error;
    g_error = cudaSuccess;
    return e;
}
cudaError_t cudaPeekAtLastError(void) { return g_error; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    *e = (cudaEvent_t)(g_next += 16);
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    g_event[e] = g_clock;
    rec(2, s, e);
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b)
{
    *ms = (float)(g_event[b] - g_event[a]);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    *s = (cudaStream_t)(g_next += 16);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    rec(3, s, e);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus *st)
{
    *st = g_capture.count(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus *st, unsigned long long *id, cudaGraph_t *g,
                                     const cudaGraphNode_t **, const cudaGraphEdgeData **, size_t *)
{
    cudaStreamIsCapturing(s, st);
    if (*st == cudaStreamCaptureStatusActive) {
        *id = g_capture[s];
        *g = (cudaGraph_t)(intptr_t)g_capture[s];
    }
    return cudaSuccess;
}
cudaError_t cudaUserObjectCreate(cudaUserObject_t *o, void *p, cudaHostFn_t fn, unsigned, unsigned)
{
    *o = reinterpret_cast<cudaUserObject_t>(new Obj{p, fn});
    return cudaSuccess;
}
cudaError_t cudaUserObjectRelease(cudaUserObject_t o, unsigned)
{
    Obj *q = reinterpret_cast<Obj *>(o);
    q->fn(q->p);
    delete q;
    return cudaSuccess;
}
cudaError_t cudaGraphRetainUserObject(cudaGraph_t g, cudaUserObject_t o, unsigned, unsigned)
{
    g_graphs[(unsigned long long)(intptr_t)g].push_back(o);
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    *g = (cudaGraph_t)(g_next += 16);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long)
{
    *x = (cudaGraphExec_t)(g_next += 16);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }

}  // extern "C"

namespace ef {

#define EF_FAKE_VARIANT(SUF, EL, D)                                                                                      \
    bool collide_supported_##SUF(int N) { return N == 8 || N == 12 || N == 16 || N == 24 || N == 32 || N == 40 || N == 48 || N == 64; } \
    int collide_maxthreads_##SUF(int N, int occ)                                                                          \
    {                                                                                                                     \
        if (EL == 8) return occ == 1 ? 512 : 0;                                                                           \
        if (D == 3 && occ >= 3) return N >= 16 && (occ == 3 || occ == 4) ? 288 : 0;                                       \
        return occ == 1 ? 256 : 0;                                                                                        \
    }                                                                                                                     \
    size_t collide_smem_##SUF(int N, int planes, int sg, int paired, int occ)                                             \
    {                                                                                                                     \
        return occ >= 3 ? rg_smem(N, planes) : smem_bytes(EL, D, N, planes, sg, paired);                                  \
    }                                                                                                                     \
    cudaError_t collide_setup_##SUF(int N, size_t smem, int cluster, int tpb, int occ, int *mc)                           \
    {                                                                                                                     \
        *mc = resident(N, smem, cluster, tpb, occ >= 3);                                                                    \
        return cudaSuccess;                                                                                               \
    }                                                                                                                     \
    cudaError_t collide_launch_##SUF(int N, const CollideArgs &a, int grid, int tpb, size_t, int occ, cudaStream_t s)     \
    {                                                                                                                     \
        return launch(0, N, a, grid, tpb, occ, s);                                                                        \
    }
EF_FAKE_VARIANT(f32_2d, 4, 2)
EF_FAKE_VARIANT(f32_3d, 4, 3)
EF_FAKE_VARIANT(f64_2d, 8, 2)
EF_FAKE_VARIANT(f64_3d, 8, 3)

int rg_rows_per_thread(int v) { return v == 2 ? 2 : 1; }
int rg_team(int) { return 1; }
cudaError_t rg_split_setup_f32(int N, int, size_t smem, int cluster, int tpb, int *mc)
{
    *mc = resident(N, smem, cluster, tpb, true);
    return cudaSuccess;
}
cudaError_t rg_split_launch_f32(int N, int v, const CollideArgs &a, int grid, int tpb, size_t, cudaStream_t s)
{
    return launch(0, N, a, grid, tpb, v + 2, s);
}
cudaError_t split_finish_setup(int, int) { return cudaSuccess; }
int split_finish_ctas(int, int d, int N, int64_t n, int sms)
{
    return (int)std::max<int64_t>(1, std::min<int64_t>((d == 3 ? N * N : N) / 4, 4 * sms / std::max<int64_t>(n, 1)));
}
cudaError_t split_finish_launch(int, int, int N, const CollideArgs &a, cudaStream_t s) { return launch(1, N, a, 0, 0, 0, s); }

bool features_fits_f32(int, int, int) { return true; }
bool features_fits_f64(int, int, int) { return true; }
cudaError_t features_launch_f32(int, int, const FeatArgs &, cudaStream_t s) { rec(4, s, nullptr); return cudaSuccess; }
cudaError_t features_launch_f64(int, int, const FeatArgs &, cudaStream_t s) { rec(4, s, nullptr); return cudaSuccess; }
cudaError_t transport_launch(int, int, int, const void *, void *, int64_t, double, cudaStream_t s) { rec(4, s, nullptr); return cudaSuccess; }
cudaError_t axpby_launch(int, void *, const void *, const void *, double, double, int64_t, cudaStream_t s) { rec(4, s, nullptr); return cudaSuccess; }
cudaError_t moments_launch(int, int, const void *, const void *, const int64_t *, const int64_t *, int64_t, int, double, double *,
                           cudaStream_t s) { rec(4, s, nullptr); return cudaSuccess; }

}  // namespace ef
