// A CUDA runtime on host memory and launch functions that only record their
// arguments: csrc/qs_api.cu compiled as C++ against them runs the C ABI's host
// logic on a machine without a GPU (test_api_host_cpu.py).
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <map>

#include "qs.h"
#include "qs_internal.h"

namespace {
cudaError_t g_last = cudaSuccess, g_next_launch = cudaSuccess;
std::map<const void*, int> g_kind;  // pointers with a kind of memory of their own (else device memory)
bool g_capturing = false, g_invalid = false;  // a failed launch invalidates the capture
int g_captures = 0, g_replays = 0, g_bulk = -1;

cudaError_t ret(cudaError_t e) {
    if (e != cudaSuccess) g_last = e;
    return e;
}
cudaError_t launch() {  // fails once after fake_fail_next_launch
    const cudaError_t e = g_next_launch;
    g_next_launch = cudaSuccess;
    g_invalid |= g_capturing && e != cudaSuccess;
    return ret(e);
}
cudaError_t rollout(const qsk::RolloutIO& io) {
    g_bulk = io.bulk;
    return launch();
}
}  // namespace

extern "C" {
void fake_set_kind(const void* p, int kind) { g_kind[p] = kind; }
void fake_fail_next_launch(int e) { g_next_launch = (cudaError_t)e; }
int fake_captures() { return g_captures; }
int fake_replays() { return g_replays; }
int fake_bulk() { return g_bulk; }  // of the last rollout launched or captured
int fake_pending_error() { return g_last; }

cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { *p = aligned_alloc(256, (n + 511) & ~size_t(255)); return cudaSuccess; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void** d, void* p, unsigned) { *d = p; return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    *a = cudaPointerAttributes{};
    a->type = g_kind.count(p) ? (cudaMemoryType)g_kind[p] : cudaMemoryTypeDevice;
    a->devicePointer = const_cast<void*>(p);
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return ret(cudaErrorInvalidValue); }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamGetFlags(cudaStream_t, unsigned* f) { *f = cudaStreamNonBlocking; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    g_capturing = true;
    g_invalid = false;
    ++g_captures;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    g_capturing = false;
    *g = g_invalid ? nullptr : (cudaGraph_t)(size_t)g_captures;
    return g_invalid ? ret(cudaErrorStreamCaptureInvalidated) : cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    *e = (cudaGraphExec_t)g;
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { ++g_replays; return cudaSuccess; }
}

namespace qsk {
typedef cudaError_t E;
typedef cudaStream_t S;
E launch_step(const Consts&, const Dev&, const ClassPlan&, const Tile*, const int*, const StepIO&, int, S) {
    return launch();
}
E launch_rollout(const Consts&, const Dev&, const Tile*, int, int, const int*, int*, const RolloutIO& io, int, int, int,
                 bool, S) {
    return rollout(io);
}
E launch_rollout_ws(const Consts&, const Dev&, const Tile*, int, int, const int*, const RolloutIO& io, int, int, S) {
    return rollout(io);
}
E launch_serve(const Consts&, const Dev&, const Tile*, int, int, const int*, const ServeIO&, int, S) { return launch(); }
E launch_diff(int, const Consts&, const Dev&, const Tile*, int, int, const int*, const float*, const float*, float*,
              const float*, float*, float*, void*, int, int, S) {
    return launch();
}
E launch_philox(const uint32_t*, uint32_t, uint32_t, int, uint32_t*, long long, S) { return launch(); }
E launch_reset(const Consts&, const Dev&, uint32_t, uint32_t, const uint8_t*, S) { return launch(); }
E launch_get_state(const Dev&, float*, float*, float*, int32_t*, uint32_t*, S) { return launch(); }
E launch_set_state(const Consts&, const Dev&, const float*, const float*, const float*, const int32_t*,
                   const uint32_t*, S) {
    return launch();
}
E launch_get_events(const Dev&, int, uint32_t*, int16_t*, S) { return launch(); }
E launch_scenario_io(const Dev&, float*, const float*, S) { return launch(); }
E launch_goals(const Consts&, const Dev&, float*, S) { return launch(); }
E launch_check_selftest(const Dev&, int, S) { return launch(); }
int serve_resident_ctas(const Consts&, int P) { return 152 * 6 / P; }
int rollout_ws_resident_ctas(const Consts&, int P) { return 152 * 6 / P; }
int rollout_grid(const Consts&, int, int, bool) { return 152; }
size_t diff_workspace_bytes(int, int, int, int) { return 256; }
}  // namespace qsk
