// A CUDA runtime that runs nothing, for host tests of the library's runtime: it
// is linked with the host object in place of libcudart and of the kernels'
// launch functions.  "Device" memory is host memory.  Every launch, event record
// and event wait is kept with its stream, so that a test can ask which launches
// a stream has waited for; a launch or an event record can be made to fail, and
// a capture is replayed by its graph's launches.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

using Clock = std::map<cudaStream_t, long>;      // launches of each stream
struct Op {
    int kind;      // 0 launch, 1 record, 2 wait
    cudaStream_t st;
    cudaEvent_t ev;
    const char* name;
};
struct Graph {
    std::vector<Op> ops;
};

std::map<cudaStream_t, Clock> seen;              // launches ordered before a stream's next one
std::map<cudaEvent_t, Clock> recorded;
Clock host;                                      // launches that the host has waited for
std::map<cudaStream_t, int> priority;
std::vector<Op> log_;
cudaStream_t capture_origin = nullptr;
std::vector<Op> capture;
cudaError_t last = cudaSuccess;
int fail_launch = -1, fail_record = -1;          // countdowns, < 0: never
long next_handle = 0x10000;

cudaError_t err(cudaError_t e) { return last = e; }
void merge(Clock& into, const Clock& from) {
    for (const auto& kv : from) into[kv.first] = std::max(into[kv.first], kv.second);
}
void run(const Op& op) {
    if (op.kind == 0) {
        seen[op.st][op.st]++;
        log_.push_back(op);
    } else if (op.kind == 1) {
        recorded[op.ev] = seen[op.st];
    } else {
        merge(seen[op.st], recorded[op.ev]);
    }
}
cudaError_t submit(const Op& op) {
    if (capture_origin) capture.push_back(op);
    else run(op);
    return cudaSuccess;
}
cudaError_t launch(const char* name, cudaStream_t st) {
    if (fail_launch >= 0 && fail_launch-- == 0) return err(cudaErrorLaunchOutOfResources);
    submit({0, st, nullptr, name});
    return cudaGetLastError();
}
template <class H>
H handle() {
    return reinterpret_cast<H>(next_handle += 16);
}
CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}

}  // namespace

// Questions and orders of a test.
extern "C" {
void fake_reset() {
    log_.clear();
    last = cudaSuccess;
    fail_launch = fail_record = -1;
}
void fake_fail_launch(int n) { fail_launch = n; }
void fake_fail_record(int n) { fail_record = n; }
void fake_stream(void* st, int prio) { priority[(cudaStream_t)st] = prio; }
int fake_priority(void* st) { return priority.at((cudaStream_t)st); }
int fake_launches() { return (int)log_.size(); }
const char* fake_launch_name(int i) { return log_[i].name; }
void* fake_launch_stream(int i) { return log_[i].st; }
// Launches of other streams that neither st nor the host has waited for.
int fake_unordered(void* st) {
    int n = 0;
    for (const auto& kv : seen) {
        const long mine = std::max(seen[(cudaStream_t)st][kv.first], host[kv.first]);
        if (kv.first != (cudaStream_t)st) n += (int)std::max(0L, kv.second.at(kv.first) - mine);
    }
    return n;
}
}

// The runtime calls that the host object makes.
extern "C" {
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorNotReady ? "not ready" : "error"; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    std::memset(p, 0, sizeof *p);
    p->major = 10;
    p->minor = 3;
    p->multiProcessorCount = 152;
    return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
    *fn = reinterpret_cast<void*>(encode);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return *p = std::aligned_alloc(256, (n + 255) / 256 * 256), cudaSuccess; }
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void* d, int v, size_t n) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaDeviceSynchronize() {
    for (const auto& kv : seen) merge(host, kv.second);
    return cudaSuccess;
}

cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int p) {
    priority[*s = handle<cudaStream_t>()] = p;
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { return cudaStreamCreateWithPriority(s, f, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* p) { return *p = priority.at(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
    if (capture_origin) return err(cudaErrorStreamCaptureUnsupported);
    merge(host, seen[s]);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) { return submit({2, s, e, ""}); }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    *s = capture_origin ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
    capture_origin = s;
    capture.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    capture_origin = nullptr;
    *g = reinterpret_cast<cudaGraph_t>(new Graph{capture});
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
    *x = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
    for (const Op& op : reinterpret_cast<Graph*>(x)->ops) run(op);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete reinterpret_cast<Graph*>(g), cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return delete reinterpret_cast<Graph*>(x), cudaSuccess; }

cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = handle<cudaEvent_t>(), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) {
    if (fail_record >= 0 && fail_record-- == 0) return err(cudaErrorInvalidValue);
    return submit({1, s, e, ""});
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaEventRecordWithFlags(e, s, 0); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return merge(host, recorded[e]), cudaSuccess; }
// One millisecond between any two events whose work the host has waited for.
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
    for (const cudaEvent_t e : {a, b})
        for (const auto& kv : recorded[e])
            if (host[kv.first] < kv.second) return err(cudaErrorNotReady);
    *ms = 1.f;
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
int trimmoe_compact_noalloc() { return -1; }      // the one entry point outside the host object
}

// The kernels' launch functions.
namespace tmoe {
struct AttnParams;
struct CombineParams;
struct CompactParams;
struct DecideParams;
struct FeedbackParams;
struct GatherParams;
struct GemmLaunch;
struct LaLayer;
struct RouterParams;
using St = cudaStream_t;
cudaError_t launch_router(const CUtensorMap*, const CUtensorMap*, const CUtensorMap*, const RouterParams&, int, St s) { return launch("router", s); }
cudaError_t launch_decide(const DecideParams&, int, St s) { return launch("decide", s); }
cudaError_t launch_lookahead_shared(const DecideParams&, int, St s) { return launch("tables", s); }
cudaError_t launch_lookahead_all(const DecideParams&, const LaLayer*, int, int, int, int, int, St s) { return launch("tables", s); }
cudaError_t launch_compact(const CompactParams&, St s) { return launch("compact", s); }
cudaError_t launch_gather(const int32_t*, const int32_t*, const GatherParams&, int, int, St s) { return launch("gather", s); }
cudaError_t launch_compact_gather(const CompactParams&, const GatherParams&, int, St s) { return launch("compact", s); }
cudaError_t launch_grouped_gemm(const GemmLaunch&, int, St s) { return launch("gemm", s); }
cudaError_t launch_splitk_finish(const GemmLaunch&, int, St s) { return launch("finish", s); }
cudaError_t launch_combine(const CombineParams&, int, St s) { return launch("combine", s); }
cudaError_t launch_attn_norm(const AttnParams&, int, St s) { return launch("attn_norm", s); }
cudaError_t launch_attention(const AttnParams&, const CUtensorMap*, const CUtensorMap*, int, int, St s) { return launch("attention", s); }
cudaError_t launch_feedback(const FeedbackParams&, St s) { return launch("feedback", s); }
cudaError_t launch_watchdog_selftest(int*, unsigned long, St s) { return launch("watchdog", s); }
int router_lo_rows(int n, int) { return n; }
int router_pass_rows(int n) { return n; }
int router_ksplit(int, int, int, int) { return 1; }
size_t decide_smem_bytes(int, int, int, int) { return 0; }
size_t decide_la_scratch_floats(int, int, int, int) { return 1; }
bool compact_gather_fits(int T) { return T <= 1024; }
int grouped_gemm_ksplit(int, int, int) { return 2; }
}  // namespace tmoe
