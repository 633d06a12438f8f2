// What a kernel launch that fails leaves behind in the host state of a context
// (csrc/dust_api.cu): the library's own objects linked with a CUDA runtime of
// host functions, whose kernels do nothing and one of whose launches returns an
// error.  Whatever launch failed, the next step clears the deposit and the
// counts before it adds to them, and sorts by counts of its own.
// Prints "ok" or the first failure and exits non-zero.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "dust.h"

namespace {

int g_fail_at = 0;      // the launch (from 1, since the last arm()) that fails; 0: none
int g_launches = 0;     // launches since the last arm()
bool g_only_capture = false, g_capturing = false;
cudaError_t g_last = cudaSuccess;

struct Event {
    size_t bytes;       // of a clear; 0: a launch
};
std::vector<Event> g_log;

void arm(int fail_at, bool only_capture)
{
    g_fail_at = fail_at;
    g_only_capture = only_capture;
    g_launches = 0;
    g_log.clear();
}

void launch()
{
    if (g_only_capture && !g_capturing) return;
    ++g_launches;
    g_log.push_back({0});
    if (g_launches == g_fail_at) g_last = cudaErrorLaunchFailure;
}

void *handle() { return std::malloc(16); }

}  // namespace

extern "C" {
// the parts of the runtime that launches are compiled to
int __cudaGetKernel(void **kernel, const void *fn) { *kernel = const_cast<void *>(fn); return 0; }
unsigned __cudaPushCallConfiguration() { return 0; }
int __cudaPopCallConfiguration() { return 0; }
int __cudaLaunchKernel() { launch(); return 0; }
void **__cudaRegisterFatBinary(void *) { return static_cast<void **>(handle()); }
void __cudaRegisterFatBinaryEnd() {}
void __cudaUnregisterFatBinary() {}
void __cudaRegisterFunction() {}
void __cudaRegisterVar() {}

cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "injected"; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 1; return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::calloc(1, n + 64); return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::calloc(1, n + 64); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaHostRegister(void *, size_t, unsigned) { return cudaSuccess; }
cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t)
{
    if (!g_capturing) std::memset(p, v, n);
    g_log.push_back({n});
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { std::memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    if (!g_capturing) std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)handle(); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { g_capturing = true; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    g_capturing = false;
    *g = (cudaGraph_t)handle();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)handle(); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = (cudaEvent_t)handle(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long)
{
    *e = (cudaGraphExec_t)handle();
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { std::free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidSymbol; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { launch(); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *)
{
    return cudaErrorNotSupported;  // no tensor maps
}
}

namespace {

constexpr int kSide = 8, kGrains = 64;
constexpr size_t kDepositBytes = (size_t)kSide * kSide * kSide * 32;
constexpr size_t kCountBytes = ((size_t)kSide * kSide * kSide + 2) * 4;
constexpr double kDt = 1e-3;

int check(int rc, const char *what)
{
    if (rc != DUST_OK) { std::printf("%s returned %d\n", what, rc); std::exit(1); }
    return rc;
}

dust_ctx *context(int predictor, int sort_interval)
{
    static double e[kSide + 1];
    for (int i = 0; i <= kSide; ++i) e[i] = i;
    dust_geometry geo{};
    geo.kind = DUST_CARTESIAN;
    dust_grid grid{};
    for (int d = 0; d < 3; ++d) { grid.n[d] = kSide; grid.edges[d] = e; grid.bc[d] = DUST_BC_PERIODIC; }
    dust_species sp{};
    sp.mass = 1.0;
    sp.tau_mode = DUST_TAU_CONST;
    sp.tau_value = 1.0;
    dust_options opt{};
    opt.precision = DUST_MIXED;
    opt.weight = DUST_WEIGHT_TSC;
    opt.gas_predictor = predictor;
    opt.sort_interval = sort_interval;
    dust_ctx *c = nullptr;
    check(dust_create(&c, &geo, &grid, &sp, 1, &opt), "dust_create");
    std::vector<double> one(kSide * kSide * kSide, 1.0), q(kGrains, 4.5), v(kGrains, 0.0);
    check(dust_set_gas(c, one.data(), one.data(), one.data(), one.data(), DUST_MEM_HOST), "dust_set_gas");
    check(dust_load_particles(c, kGrains, q.data(), q.data(), q.data(), v.data(), v.data(), v.data(), nullptr, nullptr,
                              DUST_MEM_HOST), "dust_load_particles");
    return c;
}

bool cleared(size_t bytes)
{
    for (const Event &e : g_log)
        if (e.bytes == bytes) return true;
    return false;
}

// A batch whose capture fails at its k-th launch, then a step that does not
// sort.  Returns false once k lies past the capture's launches.
bool capture_fails_at(int k, int predictor)
{
    dust_ctx *c = context(predictor, 2);
    check(dust_step(c, kDt), "dust_step");
    dust_batch *b = nullptr;
    check(dust_batch_create(&b, &c, 1, nullptr), "dust_batch_create");
    arm(k, true);
    const double dt = kDt;
    const int rc = dust_batch_step(b, &dt, 2);
    const bool reached = g_launches >= k;
    if (reached && rc == DUST_OK) { std::printf("launch %d of the capture failed unnoticed\n", k); std::exit(1); }
    arm(0, false);
    if (reached) {
        check(dust_step(c, kDt), "dust_step after the capture");
        if (!cleared(kDepositBytes)) { std::printf("launch %d failed: the deposit is not cleared\n", k); std::exit(1); }
        if (!cleared(kCountBytes)) { std::printf("launch %d failed: the counts are not cleared\n", k); std::exit(1); }
    }
    dust_batch_destroy(b);
    dust_destroy(c);
    return reached;
}

// A step whose k-th launch fails, then another: the keys that the first step
// predicted may have been turned into offsets by the failed step's scan, so
// the counts are formed anew (cleared before the first launch).
bool step_fails_at(int k, int predictor)
{
    dust_ctx *c = context(predictor, 1);
    check(dust_step(c, kDt), "dust_step");
    arm(k, false);
    const int rc = dust_step(c, kDt);
    const bool reached = g_launches >= k;
    const bool sorting = k <= 4;  // the scan (one launch), the scatter and the two segment sorts
    if (reached && rc == DUST_OK) { std::printf("launch %d of a step failed unnoticed\n", k); std::exit(1); }
    arm(0, false);
    if (reached && sorting) {
        check(dust_step(c, kDt), "dust_step after a failed one");
        if (g_log.empty() || g_log[0].bytes != kCountBytes) {
            std::printf("launch %d of a sort failed: the next sort uses its counts\n", k);
            std::exit(1);
        }
    }
    dust_destroy(c);
    return reached;
}

}  // namespace

int main()
{
    for (int predictor = 0; predictor < 2; ++predictor) {
        int captured = 0, stepped = 0;
        while (capture_fails_at(captured + 1, predictor)) ++captured;
        while (step_fails_at(stepped + 1, predictor)) ++stepped;
        if (captured < 10 || stepped < 5) { std::printf("only %d and %d launches\n", captured, stepped); return 1; }
    }
    std::printf("ok\n");
    return 0;
}
