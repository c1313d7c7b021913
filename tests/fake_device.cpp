// A CUDA runtime and kernel launchers that run nothing, linked with sg_host.cu for tests of
// what the host does: which launches with which parameters, what it reports, and what is
// left of its work when a call fails.  Memory is host memory, copies and memsets are done,
// launches are written to a log, and a stream is busy from its last launch or copy to the
// next wait for it.  The hooks at the end plant failures and results.
#include "sg_internal.cuh"

#include <cstdlib>
#include <cstring>
#include <set>
#include <vector>

namespace {

struct Entry {
    char what[16];
    double v[8];
};
std::vector<Entry> g_log;
std::set<void*> g_busy;
int g_alloc_fails_in = 0;               // > 0: that allocation from now fails
double g_sumsq = 1.0;                   // of every norm
unsigned g_lean_waits = 0, g_tail_waits = 0;
int g_loop_status = 0, g_loop_pending = 0;   // what the inner loop of a solve graph leaves
double g_confirm_sumsq = 0.0;           // the residual that its confirmation reads
struct Loop {
    void* graph;                        // the graph it is captured into
    sg::DeviceLoop* d;
};
std::vector<Loop> g_loops;
void* g_capturing = nullptr;

void log(const char* what, std::vector<double> v) {
    Entry e{};
    std::strncpy(e.what, what, sizeof(e.what) - 1);
    for (size_t i = 0; i < v.size() && i < 8; ++i) e.v[i] = v[i];
    g_log.push_back(e);
}
cudaError_t busy(cudaStream_t st) {
    if (!g_capturing) g_busy.insert(st);
    return cudaSuccess;
}
double cells(const sg::LevelGeom& g) { return double(g.nx) * g.ny * g.nz; }

}  // namespace

// ---- the runtime ----------------------------------------------------------------
extern "C" {
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

static cudaError_t allocate(void** p, size_t n) {
    if (g_alloc_fails_in > 0 && --g_alloc_fails_in == 0) return cudaErrorMemoryAllocation;
    *p = std::calloc(n ? n : 1, 1);
    return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
    if (!g_capturing) std::memmove(d, s, n);
    return busy(st);
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) {
    if (!g_capturing) std::memset(p, v, n);
    return busy(st);
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes*, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "planted"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidValue; }
cudaError_t cudaStreamCreate(cudaStream_t* st) { *st = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t st) { g_busy.erase(st); std::free(st); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { g_busy.erase(st); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)std::calloc(1, sizeof(void*)); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) { *(void**)e = st; return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { g_busy.erase(*(void**)e); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }

// graphs: the handle of the graph that a loop is captured into is also its executable's
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = (cudaGraph_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }        // (kept: the executable's identity)
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
    *e = (cudaGraphExec_t)g;
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
    *h = 0;
    return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* node, cudaGraph_t g, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                             size_t, cudaGraphNodeParams* p) {
    static cudaGraph_t body[1];
    body[0] = g;                        // (the loops of a body belong to its graph)
    p->conditional.phGraph_out = body;
    *node = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) { g_capturing = st; return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t g, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
    g_capturing = g;
    return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = (cudaGraph_t)g_capturing;
    g_capturing = nullptr;
    return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* s, unsigned long long*, cudaGraph_t* g,
                                     const cudaGraphNode_t** deps, const cudaGraphEdgeData**, size_t* n) {
    *s = cudaStreamCaptureStatusActive;
    if (g) *g = (cudaGraph_t)g_capturing;
    if (deps) *deps = nullptr;
    if (n) *n = 0;
    return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                                unsigned) {
    return cudaSuccess;
}
// A solve graph: one cycle whose outcome is planted, then the confirmation as the kernel takes it.
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
    for (Loop& l : g_loops) {
        if (l.graph != (void*)e || l.d->status != sg::kLoopRunning) continue;
        l.d->m += 1;
        l.d->rel = 0.5;
        l.d->status = g_loop_status;
        l.d->pending = g_loop_pending;
        sg::Reduced r = {g_confirm_sumsq, 1.0, 0.0, 0.0};
        sg::loop_confirm(*l.d, r);
    }
    return busy(st);
}
}  // extern "C"

// ---- the launchers --------------------------------------------------------------
namespace sg {

long long residual_blocks(const LevelGeom&) { return 1; }
long long residual_zero_blocks(const LevelGeom&) { return 1; }
long long restrict_blocks(const LevelGeom&) { return 1; }

template <typename T>
cudaError_t launch_stage(const LevelGeom& g, int order, bool first, const StageCoef& c, const T*, const T*, const T*,
                         const T*, const T*, T*, T*, cudaStream_t st) {
    log("stage", {cells(g), double(order), double(first), c.tau, c.mut1, c.mut_tau, c.gt, double(sizeof(T))});
    return busy(st);
}
template <typename T>
cudaError_t launch_gsrb(const LevelGeom& g, int, double, T*, const T*, cudaStream_t st) {
    log("gsrb", {cells(g)});
    return busy(st);
}
template <typename TI, typename TO>
cudaError_t launch_residual(const LevelGeom&, const TI*, const TI*, TO*, Partial*, int* nb, cudaStream_t st, TI*) {
    if (!g_capturing) log("residual", {});
    if (nb) *nb = 1;
    return busy(st);
}
template <typename TO>
cudaError_t launch_residual_zero(const LevelGeom&, const double*, TO*, Partial*, int* nb, cudaStream_t st, double*,
                                 int* nk) {
    if (nb) *nb = 1;
    if (nk) *nk = 1;
    return busy(st);
}
template <typename T>
cudaError_t launch_residual_restrict(const LevelGeom& g, const T*, const T*, T*, Partial*, int* nb, cudaStream_t st,
                                     int) {
    log("restrict", {cells(g)});
    if (nb) *nb = 1;
    return busy(st);
}
template <typename T>
cudaError_t launch_prolong_correct(const LevelGeom& g, const T*, T*, cudaStream_t st) {
    log("prolong", {cells(g)});
    return busy(st);
}
cudaError_t launch_finalize(const Partial*, int, Reduced* out, cudaStream_t st) {
    if (!g_capturing) *out = Reduced{g_sumsq, 1.0, 0.0, 0.0};
    return busy(st);
}
cudaError_t launch_residual_exact(const LevelGeom&, const double*, const double*, float*, double*, Partial*, unsigned*,
                                  int* nb, int* nk, cudaStream_t st) {
    if (!g_capturing) log("residual", {});
    if (nb) *nb = 1;
    if (nk) *nk = 2;
    return busy(st);
}
cudaError_t launch_update_residual(const LevelGeom& g, double*, const float*, double*, float*, Partial*, int* nb,
                                   cudaStream_t st) {
    log("update", {cells(g)});
    if (nb) *nb = 1;
    return busy(st);
}
template <typename T>
cudaError_t launch_subtract_mean(T*, long long, const Reduced*, cudaStream_t st) { return busy(st); }
cudaError_t launch_scale_copy(const double*, double*, double, long long, cudaStream_t st) { return busy(st); }
cudaError_t launch_link_copy(const double*, double*, double, bool, long long, cudaStream_t st) { return busy(st); }
cudaError_t launch_add_f32_to_f64(double*, const float*, long long, cudaStream_t st) { return busy(st); }
cudaError_t launch_sub_mean_f64(double*, long long, const Reduced*, cudaStream_t st) { return busy(st); }
cudaError_t launch_sum_partials_f64(const double*, long long, Partial*, int* nb, cudaStream_t st) {
    if (nb) *nb = 1;
    return busy(st);
}
cudaError_t launch_gravity(const LevelGeom&, const double*, double*, const double*, unsigned*, int* nk, cudaStream_t st) {
    if (nk) *nk = 1;
    return busy(st);
}
cudaError_t probe_fp64_rate(double*, double*) { return cudaSuccess; }

cudaError_t launch_loop_init(const DeviceLoop* d, cudaGraphConditionalHandle, cudaGraphConditionalHandle, bool,
                             cudaStream_t) {
    g_loops.push_back(Loop{g_capturing, const_cast<DeviceLoop*>(d)});
    return cudaSuccess;
}
cudaError_t launch_loop_step(DeviceLoop*, const Partial*, int, Reduced*, const int*, const int*,
                             cudaGraphConditionalHandle, cudaStream_t) {
    return cudaSuccess;
}
cudaError_t launch_loop_confirm(DeviceLoop*, const Partial*, int, Reduced*, cudaGraphConditionalHandle,
                                cudaGraphConditionalHandle, bool, cudaStream_t) {
    return cudaSuccess;
}

bool fused_supported(int order, int s) { return (order == 1 || order == 2) && s >= 2 && s <= kFusedMaxS; }
cudaError_t fused_configure() { return cudaSuccess; }
cudaError_t columns_configure() { return cudaSuccess; }
bool columns_configured() { return true; }
cudaError_t launch_superstep_fused(const LevelGeom& g, int order, int s, bool zero, const FusedCoef&, const float*,
                                   const float*, float*, cudaStream_t st, int tile_rows, bool tma) {
    log("superstep", {cells(g), double(order), double(s), double(zero), double(tile_rows), double(tma)});
    return busy(st);
}
unsigned lean_wait_failures() { return g_lean_waits; }

template <typename T>
bool coarse_fits(long long n) { return n <= 8192; }
template <typename T>
cudaError_t launch_coarse_solve(const CoarseParams& p, cudaStream_t st) {
    log("coarse", {cells(p.g)});
    return busy(st);
}
cudaError_t coarse_configure() { return cudaSuccess; }

cudaError_t tail_configure() { return cudaSuccess; }
unsigned tail_wait_failures() { return g_tail_waits; }
template <typename T>
bool tail_plan(TailParams<T>& p, bool, TailLaunch* t) {
    *t = TailLaunch{1, 32, 0};
    return (long long)p.lv[0].nx * p.lv[0].ny * p.lv[0].nz <= (sizeof(T) == 8 ? 16384 : 32768);
}
template <typename T>
cudaError_t launch_tail(const TailParams<T>& p, bool, const TailLaunch&, cudaStream_t st) {
    log("tail", {double(p.lv[0].nx) * p.lv[0].ny * p.lv[0].nz, double(p.nl), double(sizeof(T)), p.loop ? 1.0 : 0.0});
    return busy(st);
}

#define FOR_BOTH(F) F(float) F(double)
#define INSTANTIATE(T)                                                                                              \
    template cudaError_t launch_stage<T>(const LevelGeom&, int, bool, const StageCoef&, const T*, const T*, const T*, \
                                         const T*, const T*, T*, T*, cudaStream_t);                                  \
    template cudaError_t launch_gsrb<T>(const LevelGeom&, int, double, T*, const T*, cudaStream_t);                  \
    template cudaError_t launch_residual<T, T>(const LevelGeom&, const T*, const T*, T*, Partial*, int*, cudaStream_t, T*); \
    template cudaError_t launch_residual_zero<T>(const LevelGeom&, const double*, T*, Partial*, int*, cudaStream_t,  \
                                                 double*, int*);                                                     \
    template cudaError_t launch_residual_restrict<T>(const LevelGeom&, const T*, const T*, T*, Partial*, int*,       \
                                                     cudaStream_t, int);                                             \
    template cudaError_t launch_prolong_correct<T>(const LevelGeom&, const T*, T*, cudaStream_t);                    \
    template cudaError_t launch_subtract_mean<T>(T*, long long, const Reduced*, cudaStream_t);                       \
    template bool coarse_fits<T>(long long);                                                                         \
    template cudaError_t launch_coarse_solve<T>(const CoarseParams&, cudaStream_t);                                  \
    template bool tail_plan<T>(TailParams<T>&, bool, TailLaunch*);                                                   \
    template cudaError_t launch_tail<T>(const TailParams<T>&, bool, const TailLaunch&, cudaStream_t);
FOR_BOTH(INSTANTIATE)

}  // namespace sg

// ---- hooks ----------------------------------------------------------------------
extern "C" {
void fake_reset() {
    g_log.clear();
    g_busy.clear();
    g_alloc_fails_in = 0;
    g_sumsq = 1.0;
    g_lean_waits = g_tail_waits = 0;
    g_loop_status = sg::kLoopDone;
    g_loop_pending = 0;
    g_confirm_sumsq = 0.0;
}
void fake_fail_alloc(int nth) { g_alloc_fails_in = nth; }
void fake_norm(double sumsq) { g_sumsq = sumsq; }
void fake_waits(unsigned lean, unsigned tail) { g_lean_waits = lean; g_tail_waits = tail; }
void fake_loop(int status, int pending, double confirm_sumsq) {
    g_loop_status = status;
    g_loop_pending = pending;
    g_confirm_sumsq = confirm_sumsq;
}
int fake_busy() { return (int)g_busy.size(); }
int fake_log_size() { return (int)g_log.size(); }
void fake_log_entry(int i, char* what, double* v) {
    std::memcpy(what, g_log[i].what, sizeof(g_log[i].what));
    std::memcpy(v, g_log[i].v, sizeof(g_log[i].v));
}
}
