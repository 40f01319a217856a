// fake_cuda.cpp -- a CUDA runtime and kernel launchers without a GPU, linked with the
// library's host code (vr_api.o) to test what it does with device buffers.
//
// Device memory is host memory. The one thing modelled is which work the device may still
// have: fake_replay() stands for work that the library does not know of (a caller's graph
// holding a batch launch, replayed on a stream of the caller's) and that uses every buffer
// allocated at that moment. It lasts until something waits for the whole device:
// cudaDeviceSynchronize or cudaFree. Until then, a write into one of those buffers on behalf
// of a new object counts as a violation.
// fake_capture() stands for a capture by another thread that forbids this one nothing
// (cudaStreamCaptureModeThreadLocal): cudaFree works, but cudaDeviceSynchronize fails and
// invalidates the capture, as on the device.
#include <cuda_runtime_api.h>

#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <set>
#include <utility>
#include <vector>

#include "vr.h"

namespace {

std::map<char*, size_t> g_live;    // allocations by address
std::vector<std::pair<char*, size_t>> g_spare;  // freed into the memory pool, the oldest first
size_t g_capacity = ~(size_t)0;    // of the device
std::set<char*> g_replayed;        // those the unknown work uses
bool g_busy = false, g_fail_waits = false, g_capture = false, g_capture_valid = false;
int g_violations = 0, g_pool_allocs = 0;

void device_done() {
    g_busy = false;
    g_replayed.clear();
}

void written(const void* p) {
    if (!g_busy) return;
    char* c = static_cast<char*>(const_cast<void*>(p));
    auto it = g_live.upper_bound(c);
    if (it == g_live.begin()) return;
    --it;
    if (c < it->first + it->second && g_replayed.count(it->first)) ++g_violations;
}

size_t held() {
    size_t s = 0;
    for (auto& kv : g_live) s += kv.second;
    for (auto& e : g_spare) s += e.second;
    return s;
}

// The pool gives its oldest spare memory back until the device holds at most `keep` bytes.
void trim(size_t keep) {
    while (!g_spare.empty() && held() > keep) {
        free(g_spare.front().first);
        g_spare.erase(g_spare.begin());
    }
}

bool room(size_t n) {
    if (n > g_capacity) return false;
    trim(g_capacity - n);  // as the driver does for any allocation of the process
    return held() <= g_capacity - n;
}

cudaError_t wait() { return g_fail_waits ? cudaErrorStreamCaptureUnsupported : cudaSuccess; }

}  // namespace

extern "C" {

// ---- controls of the test
void fake_replay() {
    g_busy = true;
    g_replayed.clear();
    for (auto& kv : g_live) g_replayed.insert(kv.first);
}
void fake_fail_waits(int on) { g_fail_waits = on != 0; }
int fake_violations() { return g_violations; }
int fake_pool_allocs() { return g_pool_allocs; }
void fake_capture(int on) { g_capture = on != 0, g_capture_valid = true; }
int fake_capture_valid() { return g_capture_valid; }
long long fake_held_bytes() { return (long long)held(); }
void fake_capacity(long long n) { g_capacity = n < 0 ? ~(size_t)0 : (size_t)n; }

// ---- the runtime
cudaError_t cudaMalloc(void** p, size_t n) {
    if (!room(n)) return cudaErrorMemoryAllocation;
    *p = calloc(n ? n : 1, 1);
    g_live[static_cast<char*>(*p)] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    if (!p) return cudaSuccess;
    if (g_fail_waits) return cudaErrorStreamCaptureUnsupported;
    device_done();  // the real call waits for the device
    g_live.erase(static_cast<char*>(p));
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    *p = reinterpret_cast<cudaMemPool_t>(3);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) {
    trim(0);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t, cudaMemPoolAttr, void* v) {
    size_t used = 0;
    for (auto& kv : g_live) used += kv.second;
    *static_cast<unsigned long long*>(v) = used;
    return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) {
    trim(keep);
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
    ++g_pool_allocs;
    for (size_t i = g_spare.size(); i-- > 0;)
        if (g_spare[i].second == n) {
            *p = g_spare[i].first;
            g_live[g_spare[i].first] = n;
            g_spare.erase(g_spare.begin() + (long)i);
            return cudaSuccess;
        }
    return cudaMalloc(p, n);
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {  // waits for nothing
    char* c = static_cast<char*>(p);
    if (g_busy && g_replayed.count(c)) ++g_violations;
    g_spare.emplace_back(c, g_live[c]);
    g_live.erase(c);
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    if (g_capture) {
        g_capture_valid = false;
        return cudaErrorStreamCaptureUnsupported;
    }
    const cudaError_t e = wait();
    if (e == cudaSuccess) device_done();
    return e;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return wait(); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    written(d);
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
    written(d);
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = reinterpret_cast<cudaEvent_t>(1);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) {
    *t = 1.0f;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    *e = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(2);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}

}  // extern "C"

// ---- the launchers of the library's other translation units
namespace vr {

struct VolConst;
struct RenderLaunch;
struct BackwardLaunch;
struct BatchLaunch;
struct SkipStore;

unsigned long long current_cuda_context() { return 7; }
int minmax_blocks(long long) { return 4; }
cudaError_t launch_minmax_partials(const void*, vr_dtype, long long, float*, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_minmax_final(const float*, int, float* out2, cudaStream_t) {
    written(out2);
    out2[0] = 0.0f, out2[1] = 1.0f;
    return cudaSuccess;
}
cudaError_t launch_normalize(const void*, vr_dtype, long long, const float*, VolConst*, float* norm, cudaStream_t) {
    written(norm);
    return cudaSuccess;
}
cudaError_t launch_make_bricks(const float*, const int*, const int*, float* bricks, cudaStream_t) {
    written(bricks);
    return cudaSuccess;
}
cudaError_t launch_brick_minmax(const float*, const int*, const int*, int, uint16_t* grid, cudaStream_t) {
    written(grid);
    return cudaSuccess;
}
cudaError_t launch_make_derived(const float*, const int*, const int*, int, const float*, float* d, cudaStream_t) {
    written(d);
    return cudaSuccess;
}
cudaError_t launch_gmax(const float*, const int*, const float*, VolConst*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_classify(const uint16_t*, long long, const float*, int, int, uint8_t*, int*, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_cell_minmax(const float*, const int*, uint32_t* cellq, cudaStream_t) {
    written(cellq);
    return cudaSuccess;
}
cudaError_t launch_skip_field(const uint32_t*, const int*, const uint16_t*, long long, const float*, int, int, int*,
                              uint8_t*, const SkipStore&, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_frangi(const float*, const int*, const float*, int, float*, float*, float*, float* V, cudaStream_t) {
    written(V);
    return cudaSuccess;
}
cudaError_t launch_histogram(const float*, long long, unsigned long long*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_tissue_peaks(const unsigned long long*, int, int, int*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_median3(const float*, float* out, const int*, cudaStream_t) {
    written(out);
    return cudaSuccess;
}
cudaError_t launch_gauss3d(const float*, float* out, float*, const int*, float, cudaStream_t) {
    written(out);
    return cudaSuccess;
}
cudaError_t launch_render_gather(const RenderLaunch&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_render_backward(const BackwardLaunch&, bool, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_sum_copies(const float*, int, int, int, float*, const double*, float*, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_fma_peak(float*, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_wait_probe(unsigned*, long long, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_check_probe(unsigned*, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_channels_to_voxels(const float*, const int*, const float*, float*, cudaStream_t) {
    return cudaSuccess;
}
enum class BatchKind { kMixed, kFew, kMany };
cudaError_t launch_render_batch(const BatchLaunch&, int, int, BatchKind, int, cudaStream_t) { return cudaSuccess; }
BatchKind batch_kind(int, bool, bool) { return BatchKind::kFew; }
cudaError_t batch_ctas_per_sm(int, BatchKind, int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t launch_render_staged(const RenderLaunch&, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_render_staged_derived(const RenderLaunch&, int, int, cudaStream_t) { return cudaSuccess; }
cudaError_t staged_derived_config(int, int, int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t staged_config(int, bool, int* n) {
    *n = 1;
    return cudaSuccess;
}

}  // namespace vr
