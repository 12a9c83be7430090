// A CUDA runtime without a GPU, for the library's host code: "device" memory is
// host memory, kernels do nothing, and a queued host-to-device copy is carried
// out only when its stream is waited for (which CUDA allows for pageable and
// pinned memory alike).  Freeing host memory that such a copy has still to read
// is counted, and an event or a launch on a stream of another device than its
// own is an error, as in CUDA.  Solver states read back are marked converged, so
// that solves end.  Two devices.
//
// Linked with the library's objects; runs the case named on the command line on
// the mesh in two files (float64 [n_nodes, 3], int32 [n, 3]).
#include <cuda_runtime_api.h>
#include <malloc.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "../include/bemfmm.h"

namespace {
struct Pending {
    void *dst;
    const char *src;
    size_t n;
    cudaStream_t s;
};
constexpr int kMax = 65536;
Pending g_pending[kMax];
int g_n = 0;
std::atomic<int> g_freed{0};
std::mutex g_mu;
thread_local int t_dev = 0;
thread_local cudaError_t t_err = cudaSuccess;
struct Obj {
    int dev;
};
struct Pinned {
    char *p;
    size_t n;
} g_pinned[64];
int g_npinned = 0;
size_t g_state = 0;

int dev_of(cudaStream_t s) { return s ? reinterpret_cast<Obj *>(s)->dev : t_dev; }
void flush(cudaStream_t s, bool all)
{
    std::lock_guard<std::mutex> lk(g_mu);
    int m = 0;
    for (int i = 0; i < g_n; ++i) {
        if (all || g_pending[i].s == s) std::memcpy(g_pending[i].dst, g_pending[i].src, g_pending[i].n);
        else g_pending[m++] = g_pending[i];
    }
    g_n = m;
}
void check_free(void *p)
{
    if (!p || g_n == 0) return;
    const char *a = (const char *)p, *b = a + malloc_usable_size(p);
    std::lock_guard<std::mutex> lk(g_mu);
    int m = 0;
    for (int i = 0; i < g_n; ++i) {
        if (g_pending[i].src >= a && g_pending[i].src < b) ++g_freed;   // the copy is dropped
        else g_pending[m++] = g_pending[i];
    }
    g_n = m;
}
cudaError_t fail(cudaError_t e) { return t_err = e; }
}  // namespace

void operator delete(void *p) noexcept
{
    check_free(p);
    std::free(p);
}
void operator delete(void *p, size_t) noexcept { operator delete(p); }

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = std::calloc(1, n ? n : 1)) ? cudaSuccess : fail(cudaErrorMemoryAllocation); }
cudaError_t cudaFree(void *p)
{
    flush(nullptr, true);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned int)
{
    *p = std::calloc(1, n);
    g_pinned[g_npinned++ % 64] = Pinned{(char *)*p, n};
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p)
{
    check_free(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *dst, const void *src, size_t n, cudaMemcpyKind kind, cudaStream_t s)
{
    if (kind == cudaMemcpyHostToDevice) {
        std::lock_guard<std::mutex> lk(g_mu);
        if (g_n == kMax) return fail(cudaErrorUnknown);
        g_pending[g_n++] = Pending{dst, (const char *)src, n, s};
        return cudaSuccess;
    }
    flush(s, kind == cudaMemcpyDeviceToDevice);
    std::memcpy(dst, src, n);
    if (kind == cudaMemcpyDeviceToHost)
        for (int i = 0; i < g_npinned && i < 64; ++i)
            if ((char *)dst >= g_pinned[i].p && (char *)dst < g_pinned[i].p + g_pinned[i].n && n >= 64) {
                if (!g_state) g_state = n;              // the first solve has one right-hand side
                for (char *q = (char *)dst; q < (char *)dst + n; q += g_state) ((int *)q)[1] = ((int *)q)[2] = 1;
            }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *dst, const void *src, size_t n, cudaMemcpyKind)
{
    flush(nullptr, true);
    std::memcpy(dst, src, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t s)
{
    flush(s, false);
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d)
{
    t_dev = d;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = t_dev;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b)
{
    *a = *b = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned int)
{
    *s = reinterpret_cast<cudaStream_t>(new Obj{t_dev});
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned int f, int) { return cudaStreamCreateWithFlags(s, f); }
cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    flush(s, false);
    delete reinterpret_cast<Obj *>(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    flush(s, false);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned int) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned int)
{
    *e = reinterpret_cast<cudaEvent_t>(new Obj{t_dev});
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e)
{
    delete reinterpret_cast<Obj *>(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    return reinterpret_cast<Obj *>(e)->dev == dev_of(s) ? cudaSuccess : fail(cudaErrorInvalidResourceHandle);
}
cudaError_t cudaEventSynchronize(cudaEvent_t)
{
    flush(nullptr, true);
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.f;
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = t_err;
    t_err = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorInvalidResourceHandle ? "invalid resource handle" : "error"; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return fail(cudaErrorUnknown); }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned int, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    return fail(cudaErrorUnknown);
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *,
                                          size_t, cudaStreamCaptureMode)
{
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned int)
{
    *g = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *, cudaGraph_t, unsigned int, unsigned int)
{
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t *, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *, size_t,
                             cudaGraphNodeParams *p)
{
    static cudaGraph_t body = nullptr;
    p->conditional.phGraph_out = &body;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    *e = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

void **__cudaRegisterFatBinary(void *)
{
    static void *h;
    return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
static thread_local cudaStream_t t_launch;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *s)
{
    t_launch = (cudaStream_t)s;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *s)
{
    *(cudaStream_t *)s = t_launch;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t s)
{
    return dev_of(s) == t_dev ? cudaSuccess : fail(cudaErrorInvalidResourceHandle);
}
}  // extern "C"

template <typename T>
static std::vector<T> read_all(const char *path)
{
    std::vector<T> v;
    FILE *f = std::fopen(path, "rb");
    if (!f) return v;
    std::fseek(f, 0, SEEK_END);
    v.resize((size_t)std::ftell(f) / sizeof(T));
    std::fseek(f, 0, SEEK_SET);
    if (std::fread(v.data(), sizeof(T), v.size(), f) != v.size()) v.clear();
    std::fclose(f);
    return v;
}

int main(int argc, char **argv)
{
    if (argc < 4) return 2;
    const std::string what = argv[1];
    const std::vector<double> nodes = read_all<double>(argv[2]);
    const std::vector<int32_t> tris = read_all<int32_t>(argv[3]);
    const int64_t n = (int64_t)tris.size() / 3, nn = (int64_t)nodes.size() / 3;
    std::vector<int32_t> bc(n), region(n);
    for (int64_t i = 0; i < n; ++i) {
        bc[i] = (int32_t)(i % 3);
        region[i] = (int32_t)(i % 2);
    }
    std::vector<float> x(8 * n), y(8 * n), q(8 * n), f(8 * 4096);
    double adm[4] = {1e-3, 0, 2e-3, 1e-4};
    std::vector<double> pts(3 * 1000);
    for (size_t i = 0; i < pts.size(); ++i) pts[i] = 0.3 + 0.0001 * (double)((i * 37) % 1000);
    bem_params p;
    bem_params_default(&p);
    bem_source src[4] = {};
    for (int r = 0; r < 4; ++r) {
        src[r].kind = 0;
        src[r].vec[r % 3] = 1.0;
        src[r].amp[0] = 1.0;
    }
    int bad = 0;
    auto ok = [&](const char *name, int code) {
        if (code < 0) {
            std::printf("%s: %d %s\n", name, code, bem_last_error());
            ++bad;
        }
    };
    for (int mode = 0; mode < 2; ++mode) {
        p.mode = mode ? BEM_MODE_DIRECT : BEM_MODE_FMM;
        p.field_mode = 2;
        void *m = nullptr;
        cudaSetDevice(what == "devices" ? 1 : 0);
        ok("create", bem_mesh_create(nodes.data(), nn, tris.data(), n, bc.data(), nullptr, region.data(), &p, &m));
        if (!m) return 1;
        if (what == "devices") {
            // the caller's current device is another one, the stream its default
            // one or one of the mesh's device
            cudaStream_t own;
            cudaStreamCreateWithFlags(&own, 0);
            cudaSetDevice(0);
            ok("matvec", bem_matvec(m, 1000.0, nullptr, adm, 2, x.data(), y.data(), 1, own));
            cudaSetDevice(0);
            ok("matvec", bem_matvec(m, 1000.0, nullptr, adm, 2, x.data(), y.data(), 1, nullptr));
            cudaSetDevice(0);
            ok("solve", bem_solve(m, 1000.0, nullptr, adm, 2, src, 1, 1e-5, 50, x.data(), y.data(), nullptr, nullptr));
            bem_mesh_destroy(m);
            continue;
        }
        bem_solve_info info[4];
        double loss, grad[4];
        ok("solve", bem_solve(m, 900.0, nullptr, adm, 2, src, 1, 1e-5, 50, x.data(), y.data(), info, nullptr));
        ok("matvec", bem_matvec(m, 1000.0, nullptr, adm, 2, x.data(), y.data(), 4, nullptr));
        adm[0] *= 2;
        ok("matvec", bem_matvec(m, 1000.0, nullptr, adm, 2, x.data(), y.data(), 1, nullptr));
        ok("transpose", bem_matvec_transpose(m, 1000.0, nullptr, adm, 2, x.data(), y.data(), nullptr));
        ok("solve_multi", bem_solve_multi(m, 1100.0, nullptr, adm, 2, src, 4, 1e-5, 50, x.data(), q.data(), info, nullptr));
        ok("evaluate", bem_evaluate(m, 1100.0, nullptr, src, 2, x.data(), y.data(), pts.data(), 1000, f.data(), nullptr));
        ok("velocity", bem_evaluate_velocity(m, 1100.0, nullptr, src, 1, x.data(), y.data(), pts.data(), 1000, f.data(), nullptr));
        ok("gradient", bem_admittance_gradient(m, 1200.0, nullptr, adm, 2, src, 1, pts.data(), 50, 1e-5, 50, x.data(),
                                               y.data(), &loss, grad, info, nullptr));
        const double freqs[3] = {500.0, 2000.0, 4000.0};
        ok("sweep", bem_solve_sweep(m, freqs, 3, nullptr, adm, 2, src, 1, 1e-5, 50, x.data(), y.data(), nullptr, 0, nullptr,
                                    info, nullptr));
        bem_mesh_destroy(m);
    }
    std::printf("errors %d, freed in flight %d\n", bad, g_freed.load());
    return bad || g_freed.load() ? 1 : 0;
}
