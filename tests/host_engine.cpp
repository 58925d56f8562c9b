// The plan, solve and engine host code on a fake CUDA runtime: device memory is host memory, kernels
// advance the slots' records or a clock by set amounts, and what was launched, captured and freed is
// kept.  One scenario per run, named by the first argument; 0 is returned where all it checks holds.
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <thread>

#include "engine.cuh"

namespace {

std::mutex mu;
std::map<void *, size_t> live;                 // device allocations
std::function<void()> on_stream;               // run once by the next stream creation
bool retire = true;                            // a graph replay ends every slot, or advances its sweeps
double sweeps_per_replay[kRtMaxDepth + 1];     // by depth, where it does not end them
double clock_us = 0.0, launch_us[kRtMaxDepth + 1];
int last_depth = 0;                            // of the last FP32 sweep launch, or imported slot
std::atomic<int> last_step{0}, instances{0};   // sweep launches of the last replay, graphs instantiated

struct Step {
    EngineDev e;
    int sweeps;
};
using Steps = std::vector<Step>;
thread_local Steps *capture = nullptr;

#define CHECK(x)                                                        \
    do {                                                                \
        if (!(x)) {                                                     \
            std::printf("line %d: %s does not hold\n", __LINE__, #x); \
            std::exit(1);                                               \
        }                                                               \
    } while (0)

cudaError_t get(void **p, size_t n) {
    std::lock_guard<std::mutex> lk(mu);
    *p = std::calloc(1, n ? n : 1);
    live[*p] = n;
    return cudaSuccess;
}

cudaError_t put(void *p) {
    std::lock_guard<std::mutex> lk(mu);
    if (p) {
        CHECK(live.erase(p) == 1);
        std::free(p);
    }
    return cudaSuccess;
}

cudaError_t copy2(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h) {
    for (size_t j = 0; j < h; ++j) std::memcpy((char *)d + j * dp, (const char *)s + j * sp, w);
    return cudaSuccess;
}

}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { return get(p, n); }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return get(p, n); }
cudaError_t cudaMallocHost(void **p, size_t n) { return get(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return get(p, n); }
cudaError_t cudaFree(void *p) { return put(p); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return put(p); }
cudaError_t cudaFreeHost(void *p) { return put(p); }
cudaError_t cudaMemset(void *p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
    return copy2(d, dp, s, sp, w, h);
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceGetStreamPriorityRange(int *a, int *b) { return *a = 0, *b = -5, cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) {
    std::function<void()> f;
    f.swap(on_stream);
    if (f) f();
    *s = (cudaStream_t)std::malloc(1);
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return *e = (cudaEvent_t) new double(0.0), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete (double *)e, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return *(double *)e = clock_us, cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t a, cudaEvent_t b) {
    return *ms = (float)(1e-3 * (*(double *)b - *(double *)a)), cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return capture = new Steps, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = (cudaGraph_t)capture;
    capture = nullptr;
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
    ++instances;
    return *x = (cudaGraphExec_t) new Steps(*(Steps *)g), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete (Steps *)g, cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return delete (Steps *)x, cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t *, size_t *n) { return *n = 0, cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType *) { return cudaErrorInvalidValue; }
cudaError_t cudaGraphKernelNodeGetParams(cudaGraphNode_t, cudaKernelNodeParams *) { return cudaErrorInvalidValue; }
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, const cudaKernelNodeParams *) {
    return cudaErrorInvalidValue;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
    std::this_thread::sleep_for(std::chrono::microseconds(200));  // the engine's autotuner reads the wall clock
    const Steps &steps = *(Steps *)x;
    last_step = 0;
    for (const Step &t : steps) last_step += t.sweeps;
    const EngineDev &e = steps[0].e;
    for (int q = 0; q < e.max_slots; ++q) {
        SlotDev &S = e.slots[q];
        if (S.phase == PHASE_FREE) continue;
        if (retire) S.phase = PHASE_RETIRED;
        S.sweeps += (long long)sweeps_per_replay[S.depth];
        e.status[q] = SlotStatus{S.phase, CJ_OK, S.sweeps, 1, 0.0, 0.0, 0.0};
    }
    return cudaSuccess;
}
}

// ---- what of the kernel files the scenarios reach (the rest stays unresolved)
Grid make_grid(int Nx, int Ny, int elem_bytes) {
    const int pad = 128 / elem_bytes;
    return Grid{Nx, Ny, pad, (pad + Nx + 2 + pad - 1) / pad * pad};
}
cudaError_t eng_launch_step(const EngineDev &e, int, int, unsigned, int, const EngineBranches &, int sweeps,
                            cudaStream_t) {
    return capture->push_back(Step{e, sweeps}), cudaSuccess;
}
cudaError_t eng_launch_import(const EngineDev &e, int slot, int, const double *, long long, const double *, long long,
                              cudaStream_t) {
    last_depth = e.slots[slot].depth;
    e.slots[slot].phase = PHASE_OUTER;
    return cudaSuccess;
}
cudaError_t launch_sweep32(const cj_plan *, const float *, const float *, float *, float, cudaStream_t) {
    return last_depth = 1, clock_us += launch_us[1], cudaSuccess;
}
cudaError_t launch_sweep32_rtile(const cj_plan *, const float *, const float *, float *, const float *, int k,
                                 cudaStream_t) {
    return last_depth = k, clock_us += launch_us[k], cudaSuccess;
}
cudaError_t launch_import32(const cj_plan *, const float *, long long, float *, cudaStream_t) { return cudaSuccess; }
cudaError_t launch_export32(const cj_plan *, const float *, float *, long long, cudaStream_t) { return cudaSuccess; }
int cluster_solve_size(const cj_plan *) { return 0; }
cudaError_t rtile_prepare(int) { return cudaSuccess; }
int rtile_depth(int, int, int, long long sweeps) { return sweeps < 12 ? (int)sweeps : 12; }
March plan_march(int, int Ny, int, bool) { return March{1, 1, Ny}; }
Sweep64Shape sweep64_shape(int, int Ny, int) { return Sweep64Shape{Ny, 1, 1}; }
cudaError_t eng_prepare() { return cudaSuccess; }
int eng_default_depth(int st) { return st == 17 ? 4 : 8; }
int eng_list(int st, int Nx, int Ny) { return 2 * stencil_slot(st) + ((long long)Nx * Ny > (1LL << 20) ? 1 : 0); }
int eng_list_of_kernel(const void *) { return -1; }
bool eng_is_tile_kernel(const void *) { return false; }
void eng_rt_items(int slot, int Nx, int Ny, int, int, std::vector<int4> &items) {
    for (int n = 0; n < (Nx / 112 + 1) * (Ny / 48 + 1); ++n) items.push_back(make_int4(slot, 1, 1, 1));
}

namespace {

constexpr int N = 100;
double f_[N * N], u_[N * N];

cj_problem problem(int depth = 0) {
    cj_problem p{};
    p.Nx = p.Ny = p.ld_f = p.ld_u = N;
    p.st = CJ_ST9;
    p.tol = 1e-6;
    p.temporal_depth = depth;
    p.f = f_;
    p.u = u_;
    return p;
}

// The engine's autotuner on problem()'s class, with these sweeps a replay at depths 1, 2, 4 and 8.
void tune_engine(double d1, double d2, double d4, double d8) {
    retire = false;
    sweeps_per_replay[1] = d1, sweeps_per_replay[2] = d2, sweeps_per_replay[4] = d4, sweeps_per_replay[8] = d8;
    CHECK(cj_autotune_engine(N, N, CJ_ST9, nullptr, nullptr, nullptr) == CJ_OK);
    retire = true;
}

// A batch takes its problem whatever another thread's autotuner records meanwhile, and leaves no memory.
void batch_while_tuned() {
    on_stream = [] { tune_engine(4000, 1000, 1000, 1000); };
    const cj_problem p = problem();
    cj_result r{};
    CHECK(cj_solve_batch(&p, 1, nullptr, &r) == CJ_OK);
    CHECK(r.status == CJ_OK);
    CHECK(!on_stream && live.empty());
}

// What the engine's autotuner records is what a batch of the class then runs, and no slower than what
// an untuned one runs: the default depth where that is faster than those the tuner reports.
void engine_tuned_depth() {
    const cj_problem p = problem();
    cj_result r{};
    const double cases[3][5] = {{2000, 1000, 1000, 9000, 8}, {4000, 1000, 1000, 1000, 1}, {1000, 4000, 1000, 1000, 2}};
    for (const double *c : cases) {
        tune_engine(c[0], c[1], c[2], c[3]);
        CHECK(cj_solve_batch(&p, 1, nullptr, &r) == CJ_OK);
        CHECK(last_depth == (int)c[4]);
    }
}

// cj_autotune_depth leaves a class at the plan's own depth where that is faster than the four it reports.
void plan_tuned_depth() {
    for (const double own : {4.0, 12.0}) {  // us of a launch of 12 sweeps; one of k of the four: 2 + k / 2
        for (int k = 1; k <= kRtMaxDepth; ++k) launch_us[k] = k == 12 ? own : 2.0 + 0.5 * k;
        int best = 0;
        double gupd[4];
        CHECK(cj_autotune_depth(N, N, CJ_ST9, 8, nullptr, &best, gupd) == CJ_OK);
        CHECK(best == 8 && gupd[3] > gupd[2] && gupd[2] > gupd[1] && gupd[1] > gupd[0]);
        cj_options o{};
        o.precision = CJ_FP32_INNER;
        o.inner_cycle = 64;
        cj_plan *p = nullptr;
        CHECK(cj_plan_create(N, N, CJ_ST9, CJ_BC_DIRICHLET0, 1e-6, &o, &p) == CJ_OK);
        static float r[N * N], e[N * N];
        CHECK(cj_sweeps_f32(p, r, N, e, N, 0, 24, nullptr) == CJ_OK);
        CHECK(last_depth == (own == 4.0 ? 12 : 8));
        cj_plan_destroy(p);
    }
}

void serve(cj_server *sv, int n) {
    static double f[1000 * 1000], u[1000 * 1000];
    uint64_t t = 0;
    CHECK(cj_submit(sv, n, n, CJ_ST9, 1e-6, f, &t) == CJ_OK);
    cj_status st = CJ_PENDING;
    while (st == CJ_PENDING) st = cj_poll(sv, t, u, nullptr);
    CHECK(st == CJ_OK);
}

// A request's steps are those of the requests beside it, whatever a lane ran before: 32 sweep launches
// for long inner cycles, 8 for the shortest.
void steps_follow_requests() {
    for (const bool large_first : {true, false}) {
        cj_server *sv = nullptr;
        CHECK(cj_server_create(1 << 30, 4, &sv) == CJ_OK);
        for (int k = 0; k < 4; ++k) {
            const bool large = (k % 2 == 0) == large_first;
            serve(sv, large ? 300 : 16);
            CHECK(last_step == (large ? 32 : 8));
        }
        cj_server_destroy(sv);
        CHECK(live.empty());
    }
}

// A fresh server's graph is not captured again for each larger request of its first ones.
void graph_kept_in_first_burst() {
    cj_server *sv = nullptr;
    CHECK(cj_server_create(1 << 30, 4, &sv) == CJ_OK);
    for (const int n : {200, 300, 600, 1000}) serve(sv, n);
    CHECK(instances == 1);
    cj_server_destroy(sv);
}

}  // namespace

int main(int argc, char **argv) {
    const std::map<std::string, void (*)()> scenarios{{"batch_while_tuned", batch_while_tuned},
                                                          {"engine_tuned_depth", engine_tuned_depth},
                                                          {"plan_tuned_depth", plan_tuned_depth},
                                                          {"steps_follow_requests", steps_follow_requests},
                                                          {"graph_kept_in_first_burst", graph_kept_in_first_burst}};
    const auto s = scenarios.find(argc > 1 ? argv[1] : "");
    if (s == scenarios.end()) return 2;
    s->second();
    return 0;
}
