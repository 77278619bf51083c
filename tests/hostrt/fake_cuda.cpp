// A CUDA runtime on host memory and recording stand-ins for the kernels, so
// that the library's host code (plans, executions, batches, servers) runs
// without a GPU: which kernels it would launch in which shapes, and what it
// does when an allocation fails.  Device memory is host memory, streams run
// nothing, events are always complete.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <mutex>
#include <vector>

#include "dd_group.h"
#include "dd_internal.h"
#include "dd_kargs.h"

namespace {

struct Record {
    int kind;      // 0 direct launch, 1 grouped launch, 2 group table started, 3 host-to-device copy
    int dtype;     // bytes of a sample
    int dm_per_thread, dm_warps, time_warps, chan_per_stage, words;
    int beams;
    long long tiles, nsamp_out;
    int null_pointers;  // of a launch: descriptors or buffers that are NULL
    int captured;       // recorded between a capture's begin and end
};

std::mutex mu;
std::vector<Record> records;
int fail_malloc = 0;  // the n-th cudaMalloc from now fails
int table_ok = 1;     // tables turn out usable
int tables_done = 1;  // tables under way are complete when asked for
bool capturing = false;
int sms = 152;
long long allocations = 0;

void record(Record r) {
    std::lock_guard<std::mutex> lk(mu);
    r.captured = capturing;
    records.push_back(r);
}

cudaError_t direct(int elem, const dd::KArgs &a, unsigned grid, int dthr, int nw) {
    Record r{};
    r.dtype = elem;
    r.dm_per_thread = dthr;
    r.dm_warps = a.dm_warps;
    r.time_warps = a.time_warps;
    r.chan_per_stage = a.cstage;
    r.words = nw;
    r.tiles = a.total_tiles;
    r.beams = a.nbeams;
    r.nsamp_out = a.beams ? -1 : a.beam0.nsamp_out;
    r.null_pointers = !a.status || (a.beams ? !a.tile_counter : !a.beam0.in || !a.beam0.out) ||
                      (a.nbeams > 0 && !a.beams && !a.beam0.in);
    record(r);
    return grid > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

}  // namespace

extern "C" {

void fake_reset(void) {
    std::lock_guard<std::mutex> lk(mu);
    records.clear();
    fail_malloc = 0;
    table_ok = 1;
    tables_done = 1;
}
void fake_fail_malloc(int n) { fail_malloc = n; }
void fake_tables(int ok, int done) {
    table_ok = ok;
    tables_done = done;
}
void fake_capturing(int on) { capturing = on != 0; }
void fake_sms(int n) { sms = n; }
long long fake_allocations(void) { return allocations; }
int fake_records(Record *out, int max) {
    std::lock_guard<std::mutex> lk(mu);
    const int n = (int)records.size();
    if (out)
        std::memcpy(out, records.data(), sizeof(Record) * (size_t)(n < max ? n : max));
    return n;
}

cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = sms; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::mutex> lk(mu);
    if (fail_malloc > 0 && --fail_malloc == 0) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
    }
    *p = std::malloc(n ? n : 1);
    ++allocations;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::mutex> lk(mu);
    allocations -= p != nullptr;
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    if (n)
        std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void *, size_t, const void *, size_t, size_t, size_t,
                              cudaMemcpyKind k, cudaStream_t) {
    if (k == cudaMemcpyHostToDevice) {
        Record r{};
        r.kind = 3;
        record(r);
    }
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemset2DAsync(void *, size_t, int, size_t, size_t, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = reinterpret_cast<cudaStream_t>(std::malloc(1));
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned f, int) {
    return cudaStreamCreateWithFlags(s, f);
}
cudaError_t cudaDeviceGetStreamPriorityRange(int *l, int *g) { *l = 0; *g = -5; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    *st = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    capturing = true;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    capturing = false;
    *g = nullptr;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
    *e = reinterpret_cast<cudaGraphExec_t>(std::malloc(1));
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
    *e = reinterpret_cast<cudaEvent_t>(std::malloc(1));
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1; return cudaSuccess; }

}  // extern "C"

namespace dd {

cudaError_t launch_kernel_u8(const KArgs &a, unsigned g, int, int, cudaStream_t, int d, int w) {
    return direct(1, a, g, d, w);
}
cudaError_t launch_kernel_f16(const KArgs &a, unsigned g, int, int, cudaStream_t, int d, int w) {
    return direct(2, a, g, d, w);
}
cudaError_t launch_kernel_f32(const KArgs &a, unsigned g, int, int, cudaStream_t, int d, int w) {
    return direct(4, a, g, d, w);
}
cudaError_t launch_group(const GroupArgs &a, unsigned grid, cudaStream_t) {
    Record r{};
    r.kind = 1;
    r.dtype = 1;
    r.beams = a.nbeams;
    r.tiles = grid;
    r.null_pointers = !a.status || (a.beams ? 0 : !a.beam0.in || !a.beam0.entries);
    record(r);
    return grid > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}
bool start_group_table(GroupPrep a, int, GroupBuild *b) {
    Record r{};
    r.kind = 2;
    r.beams = a.G;
    record(r);
    void *p = nullptr;
    if (cudaMalloc(&p, sizeof(GroupEntry)) != cudaSuccess)
        return false;
    b->entries = static_cast<GroupEntry *>(p);
    return true;
}
TableState finish_group_table(GroupBuild *b, int, bool wait) {
    if (!wait && !tables_done)
        return TableState::kUnderWay;
    if (!table_ok)
        cudaFree(b->entries);
    *b = GroupBuild();
    return table_ok ? TableState::kComplete : TableState::kUnusable;
}
dd_status detect_begin(int, int, double *, double *, double *, cudaStream_t) { return DD_OK; }
dd_status detect_finalize_int(int, int64_t, int, double *, double *, double *, int64_t *,
                              cudaStream_t) {
    return DD_OK;
}

}  // namespace dd
