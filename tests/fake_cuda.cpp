// fake_cuda.cpp -- the C ABI's host code (tlbm_api.cu) on a CUDA runtime made of
// host memory, so that what it does with streams, allocations and error codes can be
// seen without a GPU (test_host_faults.py).
//
// Streams are queues: what is put on one runs when that stream is waited for, and
// nothing orders two streams.  A host-to-device cudaMemcpy returns once the data is
// staged, its copy a queued operation of the default stream.  Freed memory is kept
// apart, so that an operation that still reads it is seen.  fake_fail(name, n) makes
// the n-th call of one function from then on return an error.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <map>
#include <new>
#include <set>
#include <string>
#include <vector>

#include "../paper_1511_02155_gb300/csrc/tlbm_internal.h"

namespace {

std::map<cudaStream_t, std::deque<std::function<void()>>> queues;
std::map<void*, size_t> live;
std::string text, failing;
int fail_in = 0, throws = 0, next_flag = 0, capturing = 0, build_fails = 0;
std::map<int, std::vector<int4>> items;  // by tile; fake_items

void note(const char* fmt, long long a = 0, long long b = 0, long long c = 0) {
    char buf[160];
    snprintf(buf, sizeof buf, fmt, a, b, c);
    text += buf;
    text += '\n';
}
bool fails(const char* name) { return failing == name && fail_in > 0 && --fail_in == 0; }
void drain(cudaStream_t s) {
    auto& q = queues[s];
    while (!q.empty()) {
        auto f = q.front();
        q.pop_front();
        f();
    }
}
void drain_all() {
    for (auto& q : queues) drain(q.first);
}
void maybe_throw() {
    if (throws) throw std::bad_alloc();
}
bool alive(const void* p) {
    for (auto& m : live)
        if ((const char*)p >= (char*)m.first && (const char*)p < (char*)m.first + m.second) return true;
    return false;
}

}  // namespace

extern "C" {

// ---- what the tests drive
void fake_reset() {
    drain_all();
    text.clear();
    failing.clear();
    fail_in = throws = next_flag = capturing = build_fails = 0;
    items.clear();
}
const char* fake_log() { return text.c_str(); }
void fake_fail(const char* name, int nth) {
    failing = name;
    fail_in = nth;
}
void fake_items(int tile, int n) {  // the work items of that tile
    items[tile].clear();
    for (int k = 0; k < n; ++k) items[tile].push_back(make_int4(tile, k, 0, 3));
}
void fake_flag(int v) { next_flag = v; }         // raised by the next steps
void fake_capturing(int on) { capturing = on; }  // every stream; 2: another than the engine's, the default one
void fake_build_fails(int n) { build_fails = n; }
void fake_throws(int on) { throws = on; }  // the kernel tables' host code
int fake_allocations() { return (int)live.size(); }

// ---- CUDA runtime
cudaError_t cudaMalloc(void** p, size_t n) {
    *p = nullptr;
    if (fails("cudaMalloc")) return cudaErrorMemoryAllocation;
    if (capturing) return cudaErrorStreamCaptureUnsupported;
    *p = malloc(n ? n : 1);
    memset(*p, 0xa5, n ? n : 1);
    live[*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    drain_all();
    if (p) live.erase(p);  // kept: late reads are reported, not undefined
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    if (fails("cudaMemcpyAsync")) return cudaErrorUnknown;
    if (k == cudaMemcpyHostToDevice) {
        std::vector<char> stage((const char*)s, (const char*)s + n);
        queues[st].push_back([d, stage] { memcpy(d, stage.data(), stage.size()); });
    } else {
        queues[st].push_back([d, s, n] { memcpy(d, s, n); });
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
    if (fails("cudaMemcpy")) return cudaErrorUnknown;
    const cudaError_t e = cudaMemcpyAsync(d, s, n, k, nullptr);
    if (k != cudaMemcpyHostToDevice) drain(nullptr);
    return e;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
    queues[st].push_back([d, v, n] { memset(d, v, n); });
    return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return cudaMemsetAsync(d, v, n, nullptr); }
cudaError_t cudaStreamSynchronize(cudaStream_t st) {
    if (fails("cudaStreamSynchronize")) return cudaErrorUnknown;
    if (capturing) return cudaErrorStreamCaptureUnsupported;
    drain(st);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
    if (capturing == 2) return cudaErrorStreamCaptureImplicit;
    *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
    drain_all();
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "ok" : "fake error"; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)1, cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)99, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }

}  // extern "C"

// ---- kernel tables that only say what they were given
namespace tlbm_host {
namespace {

cudaError_t step(DevState& d, int, cudaStream_t st, cudaEvent_t, cudaEvent_t) {
    maybe_throw();
    const int4* it = static_cast<const int4*>(d.items);
    const int n = d.nitems, raise = next_flag;
    int* const flag = d.flag;
    const uint8_t* const mask = d.solid;
    queues[st].push_back([=] {  // on the stream: what is in memory by then
        if (n > 0) note(alive(it) ? "step: %lld items of tile %lld" : "step: %lld items of tile %lld, freed", n, it[n - 1].x);
        else note("step: one grid");
        if (mask && mask[0] > 1) note("step: mask not there");
        *flag |= raise;
    });
    d.cur ^= 1;
    return cudaSuccess;
}
cudaError_t totals(DevState&, int, cudaStream_t) { return cudaSuccess; }
cudaError_t init(DevState&, const double*, const double*, const double*, const double*, cudaStream_t) { return cudaSuccess; }
cudaError_t fields(DevState&, double*, double*, double*, double*, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t mass(DevState&, double* out, cudaStream_t st) {
    queues[st].push_back([out] { out[0] = out[1] = out[2] = 1.0; });
    return cudaSuccess;
}
cudaError_t get_box(DevState&, int, int, int, int, int, int, double*, cudaStream_t) { return cudaSuccess; }
cudaError_t set_pops(DevState&, const double*, cudaStream_t) { return cudaSuccess; }
int launches(const DevState&, int) {
    maybe_throw();
    return 2;
}
int aux_per_node() { return 8; }
bool has_fused(const DevState&) { return true; }
int solid_items(const DevState& d, std::vector<int4>& out) {
    maybe_throw();
    out = items[d.tile];
    return (int)out.size();
}
cudaError_t batch_build(BatchState&, cudaStream_t) {
    maybe_throw();
    note("batch build");
    return build_fails > 0 && build_fails-- ? cudaErrorInvalidConfiguration : cudaSuccess;
}
cudaError_t batch_step(BatchState& b, cudaStream_t, cudaEvent_t, cudaEvent_t) {
    maybe_throw();
    note("batch step");
    for (int k = 0; k < b.count; ++k) b.sims[k]->cur ^= 1;
    return cudaSuccess;
}
cudaError_t batch_totals(BatchState&, cudaStream_t) { return cudaSuccess; }
cudaError_t adjoint(DevState& d, int, const AdjJob& J, cudaStream_t st) {
    maybe_throw();
    const int raise = next_flag;
    int* const flag = d.flag;
    double* const acc = J.acc;
    queues[st].push_back([=] {
        *flag |= raise;
        acc[0] = 1.0;
    });
    return cudaSuccess;
}
const Ops table = {&step,    &totals,       &init,      &fields,      &mass,        &get_box,    &set_pops,     &launches,
                   &aux_per_node, &has_fused, &solid_items, &batch_build, &batch_step, &batch_totals, &adjoint};

}  // namespace
const Ops* ops_fp64_q9() { return &table; }
const Ops* ops_fp64_q19() { return &table; }
const Ops* ops_fp32_q9() { return &table; }
const Ops* ops_fp32_q19() { return &table; }
const Ops* ops_fp16_q9() { return &table; }
const Ops* ops_fp16_q19() { return &table; }
const Ops* ops_bf16_q9() { return &table; }
const Ops* ops_bf16_q19() { return &table; }
}  // namespace tlbm_host
