// A CUDA runtime on the host for the batch calls of api.cu: device memory is
// host memory, a graph's launches wait in a queue until an event they precede
// is waited for (or fake_run), and a launch counts, in each genotype's energy,
// how often it was searched.  Enough of it to see which work items a launch
// reads, without a GPU.
#include <stdlib.h>
#include <string.h>

#include <utility>
#include <vector>

#include "adgb_internal.cuh"

namespace {
struct Launch {
    const adgb::WorkItem *items;
    int n;
};
struct Event {
    size_t pos = 0;   // launches queued before it
};
std::vector<Launch> queue_, graph_;
size_t done_ = 0;
bool capturing_ = false;
std::vector<std::pair<char *, size_t>> live_, freed_;
int freed_reads_ = 0, fail_elapsed_ = -1;

bool is_freed(const void *p) {
    for (auto &f : freed_)
        if ((const char *)p >= f.first && (const char *)p < f.first + f.second) return true;
    return false;
}
void run(const Launch &l) {
    for (int i = 0; i < l.n; i++) {
        if (is_freed(l.items) || is_freed(l.items[i].energy)) {
            freed_reads_++;
            continue;
        }
        for (int k = 0; k < l.items[i].count; k++) l.items[i].energy[k] += 1.f;
    }
}
void run_to(size_t pos) {
    while (done_ < pos) run(queue_[done_++]);
}
cudaError_t launch(const adgb::WorkItem *items, int n) {
    if (capturing_) graph_.push_back({items, n});
    else run({items, n});
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_run() { run_to(queue_.size()); }
int fake_queued() { return (int)(queue_.size() - done_); }
int fake_freed_reads() { return freed_reads_; }
void fake_fail_elapsed(int nth) { fail_elapsed_ = nth; }   // the nth call from now fails

cudaError_t cudaMalloc(void **p, size_t n) {
    *p = calloc(1, n ? n : 1);
    live_.push_back({(char *)*p, n});
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {   // (memory is kept, to see later uses of it)
    run_to(queue_.size());
    for (size_t i = 0; i < live_.size(); i++)
        if (live_[i].first == p) {
            freed_.push_back(live_[i]);
            live_.erase(live_.begin() + i);
            break;
        }
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    if (n) memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }

cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = (cudaEvent_t) new Event();
    return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
    delete (Event *)e;
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
    ((Event *)e)->pos = queue_.size();
    return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
    return ((Event *)e)->pos <= done_ ? cudaSuccess : cudaErrorNotReady;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
    run_to(((Event *)e)->pos);
    return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t e, unsigned) { return cudaEventSynchronize(e); }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return fail_elapsed_ >= 0 && fail_elapsed_-- == 0 ? cudaErrorUnknown : cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
    *s = (cudaStream_t)malloc(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
    free(s);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    capturing_ = true;
    graph_.clear();
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    capturing_ = false;
    *g = (cudaGraph_t) new std::vector<Launch>(graph_);
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
    *st = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
    *x = (cudaGraphExec_t) new std::vector<Launch>(*(std::vector<Launch> *)g);
    return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
    delete (std::vector<Launch> *)g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
    delete (std::vector<Launch> *)x;
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
    for (const Launch &l : *(std::vector<Launch> *)x) queue_.push_back(l);
    return cudaSuccess;
}

cudaError_t cudaGetDeviceCount(int *n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorUnknown; }
cudaError_t cudaMallocAsync(void **, size_t, cudaStream_t) { return cudaErrorMemoryAllocation; }
cudaError_t cudaFreeAsync(void *, cudaStream_t) { return cudaSuccess; }
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
}

namespace adgb {
cudaError_t launch_eval_items(const WorkItem *items, int n, const LigDev *, const RecDev *, int *,
                              const EvalCfg &, int, int, cudaStream_t) { return launch(items, n); }
cudaError_t launch_eval_ring_items(const WorkItem *items, int n, const LigDev *, const RecDev *, int, int,
                                   int, int, cudaStream_t) { return launch(items, n); }
int items_grid(const EvalCfg &, int, int) { return 1; }
int items_layout_bytes(const EvalCfg &, int, int, int) { return 1024; }
int ring_layout_bytes(int, int, int) { return 1024; }
cudaError_t tc_gave_up_async(unsigned int n[TC_COUNTS], cudaStream_t) {
    for (int i = 0; i < TC_COUNTS; i++) n[i] = 0;
    return cudaSuccess;
}
cudaError_t launch_pack_grid(const float *, int, int, int, int, float *, cudaStream_t) { return cudaSuccess; }
// not reached by the batch calls
#define FAKE_NONE(...) __VA_ARGS__ { return cudaErrorNotSupported; }
FAKE_NONE(cudaError_t launch_dock(const RecDev &, const LigDev &, const EvalCfg &, const DockCfg &, float *,
                                  double *, long long *, DockScratch &, cudaStream_t))
FAKE_NONE(cudaError_t launch_eval(const RecDev &, const LigDev &, const EvalCfg &, int, const float *, float *,
                                  int, int, float, float, int, float *, float *, float *, cudaStream_t,
                                  const int *))
FAKE_NONE(cudaError_t launch_coords(const LigDev &, const float *, int, float *, cudaStream_t))
FAKE_NONE(cudaError_t launch_philox(const uint32_t *, int, uint32_t *, cudaStream_t))
FAKE_NONE(cudaError_t launch_l2_bench(int, const float *, long long, int, int, int, int, float *, cudaStream_t))
FAKE_NONE(cudaError_t launch_alu_bench(int, int, int, int, float *, cudaStream_t))
FAKE_NONE(cudaError_t launch_ga_converged(int, int, int, float, const float *, int *, cudaStream_t))
FAKE_NONE(cudaError_t launch_rescore_fp64(const RecDev &, const LigDev &, int, const float *, double *,
                                          cudaStream_t))
FAKE_NONE(cudaError_t launch_ga_generation(const DockCfg &, int, int, const float *, const float *, float *,
                                           int *, cudaStream_t))
FAKE_NONE(cudaError_t launch_pair_ablation(const RecDev &, const LigDev &, const EvalCfg &, float *, int, int,
                                           float *, cudaStream_t, int))
FAKE_NONE(cudaError_t launch_reduce4_bench(int, const float *, int, int, int, float *, cudaStream_t))
FAKE_NONE(cudaError_t launch_init_population(const RecDev &, int, uint64_t, int, int, float *, int *,
                                             cudaStream_t))
FAKE_NONE(cudaError_t launch_sw(const RecDev &, const LigDev &, const EvalCfg &, const SwCfg &, float *, int,
                                float *, int *, float *, cudaStream_t, const int *))
}  // namespace adgb
