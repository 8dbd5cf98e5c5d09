// The serving loop on a CUDA runtime made of host memory: copies are memcpy,
// events and streams complete at once, and calls fail on demand.  "Device"
// work is a plan that adds the step count to every element.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <atomic>
#include <map>
#include <mutex>
#include <string>

#include "runtime.h"

static std::atomic<int> fail_d2h{0}, fail_record{0};   // > 0: the next so many calls fail
static std::mutex mu;
static std::map<void*, size_t> pinned;
static size_t pinned_now = 0, pinned_most = (size_t)1 << 40;

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "injected"; }
const char* cudaGetErrorName(cudaError_t) { return "injected"; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free((void*)s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free((void*)e); return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) {
    return fail_record > 0 && fail_record-- > 0 ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { *p = malloc(n); return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    if (k == cudaMemcpyDeviceToHost && fail_d2h > 0 && fail_d2h-- > 0) return cudaErrorUnknown;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
    std::lock_guard<std::mutex> lk(mu);
    if (pinned_now + n > pinned_most) return cudaErrorMemoryAllocation;
    *p = malloc(n);
    pinned[*p] = n;
    pinned_now += n;
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::lock_guard<std::mutex> lk(mu);
    pinned_now -= pinned[p];
    pinned.erase(p);
    free(p);
    return cudaSuccess;
}

stencil_status stencil_plan_create(stencil_plan_t* out, int ndim, const int64_t* shape, int, stencil_kind,
                                   const double*, stencil_dtype, const stencil_options*) {
    *out = new stencil_plan_s;
    (*out)->points = 1;
    for (int d = 0; d < ndim; ++d) (*out)->points *= shape[d];
    return STENCIL_OK;
}
stencil_status stencil_plan_destroy(stencil_plan_t p) { delete p; return STENCIL_OK; }
stencil_status stencil_apply(stencil_plan_t p, const void* in, void* out, int64_t steps, stencil_stream_t) {
    for (int64_t i = 0; i < p->points; ++i) ((float*)out)[i] = ((const float*)in)[i] + (float)steps;
    return STENCIL_OK;
}
}
namespace stx {
static thread_local std::string err;
stencil_status fail(stencil_status st, const std::string& m) { err = m; return st; }
stencil_status cuda_fail(cudaError_t, const char* w) { err = w; return STENCIL_ECUDA; }
const std::string& last_error_string() { return err; }
stencil_status plan_error_status(const stencil_plan_s*, const char*) { return STENCIL_OK; }
cudaError_t fill_uniform(void*, bool, int64_t, uint64_t, int64_t, double, double, cudaStream_t) { return cudaErrorUnknown; }
}

// One request of side x side points that start at `value`, 10 steps; its status, and its result in `out`.
static int solve(stencil_server_t s, int side, float value, float* out) {
    static const double cg[9] = {};
    const int n = side * side;
    float* in = (float*)malloc(4 * n);
    for (int i = 0; i < n; ++i) in[i] = value;
    stencil_request rq = {};
    rq.ndim = 2;
    rq.radius = 1;
    rq.kind = STENCIL_BOX;
    rq.shape[0] = rq.shape[1] = side;
    rq.coeffs = cg;
    rq.h_in = in;
    rq.steps = 10;
    uint64_t id = 0;
    if (stencil_server_submit(s, &rq, &id) != STENCIL_OK) exit(2);
    const int st = stencil_server_wait(s, id, 20000);
    float* got = (float*)malloc(4 * n);
    const int rs = stencil_server_result(s, id, got, nullptr);
    *out = got[0];
    free(in);
    free(got);
    return st != STENCIL_OK ? st : rs;
}

int main(int argc, char** argv) {
    const std::string what = argv[1];
    stencil_server_t s = nullptr;
    if (stencil_server_create(&s, (int64_t)1 << 30, 4, 4, 2) != STENCIL_OK) return 2;
    float v = 0;
    // a first request leaves its result buffer, with its result, for the next
    if (solve(s, 64, 5.0f, &v) != STENCIL_OK || v != 15.0f) return 3;
    if (what == "copy") fail_d2h = 1;
    if (what == "record") fail_record = 1;
    if (what == "pinned") pinned_most = 140 << 10;   // the kept buffer has 64 KiB, the next result needs 128
    const int st = solve(s, what == "pinned" ? 130 : 64, 7.0f, &v);
    printf("%d", st);
    if (st == STENCIL_OK) printf(" %g", v);
    // the server goes on
    if (solve(s, 64, 9.0f, &v) != STENCIL_OK || v != 19.0f) return 4;
    stencil_server_destroy(s);
    if (pinned_now != 0) return 5;
    return 0;
}
