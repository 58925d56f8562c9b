// Device helpers shared by the kernel translation units: writing an interior node
// together with the odd-reflection ghost values that mirror it, and the block reduction
// of the residual statistics.
#pragma once

#include "cj_internal.h"

// Writes v at interior node (i, j) and, for a radius-2 stencil, the odd-reflection ghost
// values that mirror it (u[-1] = -u[1], u[N+2] = -u[N], corners +u).
template <int R, typename T>
__device__ __forceinline__ void store_node(T *out, const Grid &g, int i, int j, T v) {
    out[g.idx(i, j)] = v;
    if (R == 2) {
        const T nv = -v;
        if (i == 1) out[g.idx(-1, j)] = nv;
        if (i == g.Nx) out[g.idx(g.Nx + 2, j)] = nv;
        if (j == 1) {
            out[g.idx(i, -1)] = nv;
            if (i == 1) out[g.idx(-1, -1)] = v;
            if (i == g.Nx) out[g.idx(g.Nx + 2, -1)] = v;
        }
        if (j == g.Ny) {
            out[g.idx(i, g.Ny + 2)] = nv;
            if (i == 1) out[g.idx(-1, g.Ny + 2)] = v;
            if (i == g.Nx) out[g.idx(g.Nx + 2, g.Ny + 2)] = v;
        }
    }
}


// fmax(m, |r|) for m >= 0, a NaN r left out: on the bits, as the FP64 pipe's compare costs as much as
// an addition.
__device__ __forceinline__ double max_abs(double m, double r) {
    const long long b = __double_as_longlong(r) & 0x7fffffffffffffffLL;
    return b > __double_as_longlong(m) && b <= 0x7ff0000000000000LL ? __longlong_as_double(b) : m;
}

// Block reduction of (sum, max, sum) into partials[3 * block], m >= 0.  The two sums share each
// step's addition: lanes 0..15 have the first and lanes 16..31 the second (a row of 128 nodes
// would otherwise spend as many FP64 instructions here as on its residual).
__device__ __forceinline__ void block_reduce3(double a, double m, double c, double *partials) {
    __shared__ double sh[kBX / 32][3];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double other = __shfl_xor_sync(0xffffffffu, lane < 16 ? c : a, 16);
    double v = (lane < 16 ? a : c) + other;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max_abs(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        sh[wid][0] = v;
        sh[wid][1] = m;
    }
    if (lane == 16) sh[wid][2] = v;
    __syncthreads();
    if (threadIdx.x < 3) {
        const long long blk = (long long)blockIdx.y * gridDim.x + blockIdx.x;
        double r = sh[0][lane];
        if (threadIdx.x == 1) {
            for (int k = 1; k < kBX / 32; ++k) r = max_abs(r, sh[k][1]);
        } else {
            for (int k = 1; k < kBX / 32; ++k) r += sh[k][lane];
        }
        partials[3 * blk + lane] = r;
    }
}
