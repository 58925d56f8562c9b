// The register tiles (rtile_dev.cuh) over one whole grid: k = 2 .. 16 FP32 inner sweeps per launch.
//
// Measured on one GB300 (us per sweep, one sweep per launch or the per-warp row wavefront these
// tiles replaced -> tiles at their default depth): 9-point 333 x 250: 3.9 -> 0.44; 1023^2: 3.8 ->
// 0.94; 4096^2: 13.9 -> 9.2 (1834 Gupd/s); 8192^2: 45 -> 32.7 (2053 Gupd/s); 17-point 8192^2:
// 159 -> 68.8 (976 Gupd/s); 400^2: 4.0 -> 1.2.  On large grids the FMA pipe is busy 66 % of an SM's
// cycles (4096^2; 9.25 operations per node and sweep for 9 points, times the tile's overlap of 1.34); the
// rest is the loads and stores at the ends of a tile's life, which the other block of the SM hides
// only in part.  On small ones the launch and the tile's load and store (2.3 us together, with
// programmatic dependent launch) stand beside k sweeps of a quarter of a microsecond each.
#include <cmath>

#include "rtile_dev.cuh"

namespace {

struct RtWeights {
    float w[kRtMaxDepth];
};

template <int ST, int RPT, int NW, int PER_SM>
__global__ void __launch_bounds__(NW * 32, PER_SM)
    sweep_rtile_kernel(const float *e, const float *__restrict__ r, float *out, Grid g,
                       const __grid_constant__ RtWeights wt, int k, int nstrips, int cols, int rows) {
    extern __shared__ float4 sm[];
    const int strip = (int)blockIdx.x % nstrips, rb = (int)blockIdx.x / nstrips;
    const int oy0 = 1 + rb * rows, oy1 = min(oy0 + rows - 1, g.Ny);
    rt_run<ST, RPT, NW>(e, r, out, g, wt.w, k, 1 + strip * cols, oy0, oy1, sm);
}

// Tile shapes (rows per warp, warps): 128 staged columns by RPT * NW rows.  The tall ones run two
// blocks of 8 warps per SM within 128 registers a thread; the short ones give small grids enough
// blocks for the SMs.  Other shapes measured slower at every size: 16 warps (one block per SM: its
// loads stand alone), 6 rows (more exchange per row), 64-register shapes (they spill).
struct RtKernel {
    int rpt, nw;
    const void *fn;
    int smem;
};

template <int ST, int RPT, int NW, int PER_SM>
RtKernel rt_kernel() {
    return RtKernel{RPT, NW, (const void *)sweep_rtile_kernel<ST, RPT, NW, PER_SM>, RtShape<ST, RPT, NW>::smem_bytes};
}

struct RtKernels {
    RtKernel k[5];
    int n;
    double row_us;  // measured us per staged row and sweep of one SM
    double t0_us;   // and per launch
};

const RtKernels &rt_kernels(int st) {
    static const RtKernels k5{{rt_kernel<5, 16, 8, 2>(), rt_kernel<5, 14, 8, 2>(), rt_kernel<5, 12, 8, 2>(),
                               rt_kernel<5, 8, 8, 2>(), rt_kernel<5, 8, 4, 4>()}, 5, 0.0060, 2.3};
    static const RtKernels k9{{rt_kernel<9, 16, 8, 2>(), rt_kernel<9, 14, 8, 2>(), rt_kernel<9, 12, 8, 2>(),
                               rt_kernel<9, 8, 8, 2>(), rt_kernel<9, 8, 4, 4>()}, 5, 0.0068, 2.3};
    static const RtKernels k17{{rt_kernel<17, 14, 8, 2>(), rt_kernel<17, 8, 8, 2>(), rt_kernel<17, 4, 8, 2>()},
                               3, 0.0145, 2.8};
    return st == 5 ? k5 : st == 9 ? k9 : k17;
}

// Shared memory per block when there is at most one block per SM: more than half an SM's, so that
// the next launch's blocks, which start while this one drains, spread over the SMs as well.
constexpr int kRtAloneSmem = 116 * 1024;

int rt_sms() {
    static const int n = [] {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
        return sms;
    }();
    return n;
}

struct RtTiles {
    int nstrips, nrb, cols, rows;
};

RtTiles rt_tiles(const RtKernel &K, int R, int Nx, int Ny, int k) {
    RtTiles t{0, 0, 128 - 2 * rt_halo_cols(R, k), K.nw * K.rpt - 2 * R * k};
    if (t.rows < 4) return t;
    t.nstrips = (Nx + t.cols - 1) / t.cols;
    t.nrb = (Ny + t.rows - 1) / t.rows;
    t.rows = (Ny + t.nrb - 1) / t.nrb;  // the same rows for every block
    return t;
}

// The shape with the shortest modelled launch of k sweeps, and that time in us: a fixed part (launch,
// first load, last store), and for the SM with the most tiles the sweeps of its staged rows (row_us
// each) and their loads and stores at its share of the HBM rate (0.032 us a row; 0.012 from the L2, and
// in between where e, r and the output take 20 to 60 MB of its 129), which overlap in part, as the blocks
// of an SM drift apart: the root of the sum of squares.  Over 34 sizes from 150 to 8192 a side the depth
// and shape chosen are within 1.2 / 0.4 / 0.6 % of the fastest on average (5 / 9 / 17 points) and
// within 13 / 6 / 8 % at worst; with one step from L2 to HBM at 100 MB the worst was 38 % (17-point 3000
// x 2700: 14.4 us a sweep, now 10.4; 9-point 2048^2: 3.23, now 2.84).
// Modelled / measured us (9-point unless said): 400^2, 8 x 4 rows, k = 8: 4.1 / 4.3; 640^2, 8 x 8,
// k = 16: 9.3 / 9.6; 1500^2, 12 x 8, k = 8: 12.8 / 13.5; 4096^2, 14 x 8, k = 4: 46.5 / 47.5, k = 8:
// 78 / 73; 8192^2, 16 x 8, k = 8: 294 / 262; 17-point 8192^2, 14 x 8, k = 2: 174 / 169, k = 4: 315 / 275.
int rt_choose(int st, int Nx, int Ny, int k, double *us) {
    const RtKernels &S = rt_kernels(st);
    const int R = st == 17 ? 2 : 1, sms = rt_sms();
    const double hbm = std::fmin(std::fmax((12e-6 * Nx * Ny - 20.0) / 40.0, 0.0), 1.0);
    const double mem_us = 0.012 + 0.020 * hbm;
    int best = 0;
    *us = 1e300;
    for (int i = 0; i < S.n; ++i) {
        const RtTiles t = rt_tiles(S.k[i], R, Nx, Ny, k);
        if (t.nstrips == 0) continue;
        const long long tiles = (long long)t.nstrips * t.nrb;
        const double q = tiles <= 2 * sms ? (double)((tiles + sms - 1) / sms) : (double)tiles / sms + 0.2;
        const double rows = q * S.k[i].rpt * S.k[i].nw;
        const double T = S.t0_us + rows * std::sqrt(S.row_us * S.row_us * k * k + mem_us * mem_us);
        if (T < *us) {
            *us = T;
            best = i;
        }
    }
    return best;
}

}  // namespace

int rtile_depth(int st, int Nx, int Ny, long long sweeps) {
    const int step = st == 17 ? 2 : 4;
    int best = 1;
    double best_us = 1e300;
    for (int k = step; k <= 4 * step; k += step) {
        double us;
        rt_choose(st, Nx, Ny, k, &us);
        if (us / k < best_us) {
            best_us = us / k;
            best = k;
        }
    }
    return sweeps < best ? (int)(sweeps < 1 ? 1 : sweeps) : best;
}

cudaError_t rtile_prepare(int st) {
    const RtKernels &S = rt_kernels(st);
    for (int i = 0; i < S.n; ++i) {
        const int smem = S.k[i].smem > kRtAloneSmem ? S.k[i].smem : kRtAloneSmem;
        const cudaError_t e = cudaFuncSetAttribute(S.k[i].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_sweep32_rtile(const cj_plan *p, const float *e, const float *r, float *out, const float *w, int k,
                                 cudaStream_t s) {
    if (k < 1 || k > (p->st == 17 ? 8 : kRtMaxDepth)) return cudaErrorInvalidValue;
    double us;
    const RtKernel &K = rt_kernels(p->st).k[rt_choose(p->st, p->Nx, p->Ny, k, &us)];
    const RtTiles t = rt_tiles(K, p->st == 17 ? 2 : 1, p->Nx, p->Ny, k);
    const int tiles = t.nstrips * t.nrb;
    RtWeights wt{};
    for (int q = 0; q < k; ++q) wt.w[q] = w[q];
    Grid g = p->g32;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3((unsigned)(K.nw * 32));
    cfg.dynamicSmemBytes = tiles <= rt_sms() && K.smem < kRtAloneSmem ? kRtAloneSmem : K.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&e, (void *)&r, (void *)&out, (void *)&g, (void *)&wt,
                    (void *)&k, (void *)&t.nstrips, (void *)&t.cols, (void *)&t.rows};
    return cudaLaunchKernelExC(&cfg, K.fn, args);
}
