// A CUDA runtime and the library's launchers for tests of csrc/stereo_api.cu on
// the CPU: every call succeeds and does nothing but write its line to a log, except
// the one launch that fake_fail_at() names and the capture queries while
// fake_fail_query() is on. As in the runtime, an error also stays until
// cudaGetLastError() takes it, and a launch without a status of its own asks that.
#include "internal.cuh"

#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

using namespace stereo;

namespace {
std::string g_log;
int g_launch = 0, g_fail = -1, g_nodes = 0;
bool g_fail_query = false;
cudaError_t g_last = cudaSuccess;
uintptr_t g_next = 0x1000;
bool g_capturing = false;

void say(const std::string &line) { g_log += line + "\n"; }
std::string hex(const void *p)
{
    char b[32];
    snprintf(b, sizeof b, "%zx", (size_t)p);
    return b;
}
template <class T> T handle() { return reinterpret_cast<T>(g_next += 0x10); }
cudaError_t launch(const char *name, cudaStream_t s, int *launches = nullptr)
{
    say(std::string("launch ") + name + " " + hex(s));
    ++g_nodes;
    if (launches) ++*launches;
    if (g_launch++ == g_fail) return g_last = cudaErrorLaunchFailure;
    return cudaSuccess;
}
}  // namespace

extern "C" {
STEREO_TEST_API void fake_reset()
{
    g_log.clear();
    g_launch = 0;
    g_fail = -1;
    g_fail_query = false;
    g_last = cudaSuccess;
}
STEREO_TEST_API void fake_fail_at(int launch) { g_fail = launch; }
STEREO_TEST_API void fake_fail_query(int on) { g_fail_query = on != 0; }
STEREO_TEST_API const char *fake_log() { return g_log.c_str(); }
}

// ---- launchers (internal.cuh)
namespace stereo {
cudaError_t costagg_setup() { return cudaSuccess; }
cudaError_t refine_setup() { return cudaSuccess; }
cudaError_t diff_setup() { return cudaSuccess; }
// one tile with 16-bit window sums, the others take anything
bool costagg_fits(const CostAggArgs &a, int tile) { return tile != 0 || (uint64_t)(2 * a.wx + 1) * a.P < 65536u; }
int costagg_pick(const CostAggArgs &a, int) { return costagg_fits(a, 0) ? 0 : 1; }
cudaError_t launch_grey(const uint8_t *, const uint8_t *, uint8_t *, uint8_t *, int, int, cudaStream_t s)
{
    launch("grey", s);
    return cudaGetLastError();
}
cudaError_t launch_grey_down(const GreyJob *jobs, int n, cudaStream_t s, int *launches)
{
    bool kind[2] = {false, false};
    for (int i = 0; i < n; ++i) kind[jobs[i].W % 4 == 0] = true;
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 2; ++k)
        if (kind[k] && e == cudaSuccess) e = launch("grey_down", s, launches);
    return e;
}
cudaError_t launch_support(const SupImage *, int, int, int, int, uint32_t *, cudaStream_t s)
{
    return launch("support", s);
}
cudaError_t launch_costagg(const CostAggArgs &, cudaStream_t s) { return launch("costagg", s); }
cudaError_t launch_costagg_batch(BatchArgs &b, int tile, int, cudaStream_t s)
{
    for (int j = 0; j < b.njobs; ++j)
        if (!costagg_fits(b.job[j], tile)) return cudaErrorInvalidValue;
    return launch("batch", s);
}
cudaError_t launch_refine(const RefineJob *, int, bool, int, int, cudaStream_t s) { return launch("refine", s); }
cudaError_t launch_unpack_planes(const uint32_t *, const uint32_t *, uint8_t *, uint8_t *, uint32_t *, int, int,
                                 cudaStream_t s)
{
    return launch("unpack", s);
}
size_t diff_workspace_bytes(int, int, int, int) { return 256; }
cudaError_t diff_run(const DiffArgs &, cudaStream_t s)
{
    for (int i = 0; i < 4; ++i) {
        const cudaError_t e = launch("diff", s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
}  // namespace stereo

// ---- the runtime calls of stereo_api.cu
extern "C" {
cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp *p, int)
{
    memset(p, 0, sizeof *p);
    strcpy(p->name, "fake");
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "a call failed"; }
cudaError_t cudaMalloc(void **p, size_t n) { return *p = malloc(n), cudaSuccess; }
cudaError_t cudaFree(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { return free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = handle<cudaStream_t>(), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    say("wait " + hex(s) + " " + hex(e));
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s)
{
    say("record " + hex(e) + " " + hex(s));
    return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *c)
{
    if (g_fail_query) return g_last = cudaErrorStreamCaptureImplicit;
    return *c = cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode)
{
    g_capturing = true;
    g_nodes = 0;
    return cudaSuccess;
}
// a graph is the number of its nodes
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g)
{
    g_capturing = false;
    *g = reinterpret_cast<cudaGraph_t>(new int(g_nodes));
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g)
{
    delete reinterpret_cast<int *>(g);
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long)
{
    say("instantiate");
    *x = reinterpret_cast<cudaGraphExec_t>(new int(*reinterpret_cast<int *>(g)));
    return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t x, cudaGraph_t g, cudaGraphExecUpdateResultInfo *)
{
    return *reinterpret_cast<int *>(x) == *reinterpret_cast<int *>(g) ? cudaSuccess : cudaErrorGraphExecUpdateFailure;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x)
{
    delete reinterpret_cast<int *>(x);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s)
{
    say("graph " + hex(s));
    return cudaSuccess;
}
}
