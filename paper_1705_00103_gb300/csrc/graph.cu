// CUDA graphs of the FP64 sweeps for grids whose sweeps are shorter than a host-side launch.
//
// On grids of up to 2^22 nodes one FP64 sweep takes a few to a few tens of microseconds, about
// what the host needs to issue one kernel, so a cycle of M single-sweep launches is bound by the
// host, not the GPU.  A plan for such a grid captures, once, a graph of G sweeps (G = min(M, 128), a
// power of two, so an even chain that starts and ends in the buffer u0; sweep64.cu's kernels, with
// the overlap of one launch's end with the next one's start that they ask for), followed by one
// node that advances a device-side position in the weight table by G.  A cycle is then a reset
// of the position and M / G graph launches.  The sweeps read their weight w_n from a device copy
// of the plan's table at index position + k.
#include "cj_internal.h"

namespace {

constexpr long long kGraphMaxNodes = 1LL << 22;  // grids up to 2048 x 2048 use the graph
constexpr int kGraphChain = 128;                  // sweeps per graph launch (at most)

// Moves the table position on by one graph's worth of sweeps, modulo the cycle length.
__global__ void advance_pos_kernel(long long *pos, long long G, long long M) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *pos = (*pos + G) % M;
}

}  // namespace

bool sweep_graph_wanted(const cj_plan *p) {
    return p->M >= 2 && (long long)p->Nx * p->Ny <= kGraphMaxNodes;
}

cudaError_t make_sweep_graph(cj_plan *p) {
    const int G = (int)(p->M < kGraphChain ? p->M : kGraphChain);
    cudaError_t e = cudaMalloc((void **)&p->w_dev, sizeof(double) * (size_t)p->M);
    if (e == cudaSuccess) e = cudaMalloc((void **)&p->pos, sizeof(long long));
    if (e == cudaSuccess)
        e = cudaMemcpy(p->w_dev, p->w.data(), sizeof(double) * (size_t)p->M, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(p->pos, 0, sizeof(long long));
    if (e != cudaSuccess) return e;
    cudaStream_t cs = nullptr;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) return e;
    cudaGraph_t graph = nullptr;
    e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
    if (e == cudaSuccess) {
        for (int k = 0; k < G && e == cudaSuccess; ++k)
            e = launch_sweep64_tab(p, (k & 1) ? p->u1 : p->u0, (k & 1) ? p->u0 : p->u1, k, cs);
        if (e == cudaSuccess) {
            advance_pos_kernel<<<1, 32, 0, cs>>>(p->pos, G, p->M);
            e = cudaGetLastError();
        }
        const cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
        if (e == cudaSuccess) e = e2;
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&p->graph, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    cudaStreamDestroy(cs);
    if (e == cudaSuccess) p->graph_G = G;
    return e;
}

cudaError_t launch_sweep_cycle_graph(const cj_plan *p, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(p->pos, 0, sizeof(long long), s);
    for (long long r = 0; r < p->M / p->graph_G && e == cudaSuccess; ++r) e = cudaGraphLaunch(p->graph, s);
    return e;
}
