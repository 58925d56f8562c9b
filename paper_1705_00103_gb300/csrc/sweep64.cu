// The FP64 weighted sweep u' = u + w (L u - b) of Sec. 2.1 over one whole grid, in the evaluation
// order of the FP64 reference (kernels.cu's header), one launch per sweep.
//
// What bounds it: the FP64 pipe, which issues 2 operations per SM clock (a warp's instruction every
// 64 clocks per scheduler) against 64 integer and 128 FP32 ones.  A sweep takes 6 / 8 / 14 FP64
// operations a node (5 / 9 / 17 points), 3 / 4 / 8 of them additions that only feed L u's
// coefficients, so those additions are done on the integer pipe (add_int): both operands' mantissas
// in 64-bit words aligned with 10 guard bits, one integer addition, one rounding to nearest even.
// That is exact IEEE addition wherever the operands have the same sign and exponents within 10 of each other,
// away from the ends of the exponent range; a warp with a lane outside that in any addition of a row
// (at zero crossings, beside the boundary's zeros, on non-finite values) does the row's additions
// on the FP64 pipe.  Both ways give the same bits.  An addition takes about 27 integer
// instructions, 54 clocks of a scheduler against the 64 of the FP64 pipe, and the two pipes overlap.
// On smooth iterates 2 of 32 warps take the FP64 row (the boundary's); where every warp does, the
// sweep is as fast as with FP64 additions alone, and the integer work hides behind them.  Additions
// of opposite signs as well (a shift by the leading zeros) measured slower at every size: 45
// instructions.
//
// A thread walks `ty` rows of one column, the next row's loads one iteration ahead; threads
// number the columns of one chunk of rows after the other, so narrow grids leave no lane idle.
// Sweeps follow one another with programmatic dependent launch (cj_internal.h).
//
// Measured on one GB300 (us per sweep; one 128-column block per strip with FP64 additions -> this) on
// smooth iterates: 9-point 1001 x 701: 13.6 -> 8.5; 1024^2: 18.1 -> 11.5; 4096^2: 268 -> 134; 5-point
// 600 x 500: 5.2 -> 4.1; 1024^2: 13.2 -> 8.8; 4096^2: 216 -> 112; 17-point 129 x 200: 4.1 -> 3.0; 1000 x
// 1100: 33.2 -> 23.9; 4096^2: 475 -> 276.  An iterate with a sign change in every warp's row, or of
// zeros, gains little (noise or zeros, 4096^2: 9-point 268 -> 248, 5-point 216 -> 187, 17-point 475 -> 466);
// others lie between (16 9-point sweeps of 4096^2 that smooth a rough iterate, with import and export:
// 4.67 -> 4.07 ms).
#include "cj_internal.h"
#include "grid_dev.cuh"
#include "stencil_dev.cuh"

namespace {

constexpr int kS64Threads = 128;

// Exponent field outside [32, 2015].  An addition's result (or its operands) tested so vouches for
// what is within 10 exponents of it: both operands of the sum, the other operand of the next one and
// the two that this one came from (at most 21 below or 11 above) are normal.
__device__ __forceinline__ bool range_bad(double x) {
    return (((unsigned)__double2hiint(x) >> 20 & 0x7ffu) - 32u) > 1983u;
}

// x + y on the integer pipe; sets bad where the signs differ or the exponents are more than 10 apart
// (the caller checks the range of one value per chain of additions).
__device__ __forceinline__ double add_int(double x, double y, bool &bad) {
    const unsigned long long bx = (unsigned long long)__double_as_longlong(x);
    const unsigned long long by = (unsigned long long)__double_as_longlong(y);
    const int sx = (int)((unsigned)(bx >> 32) >> 20), sy = (int)((unsigned)(by >> 32) >> 20);  // sign and exponent
    const int dif = sx - sy;
    bad = bad || (unsigned)(dif + 10) > 20u;
    // 53-bit mantissas below 10 guard bits, the smaller operand's shifted right by the difference
    const int kx = min(dif + 10, 10), ky = min(10 - dif, 10);
    const unsigned long long mx = (bx & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    const unsigned long long my = (by & 0x000fffffffffffffULL) | 0x0010000000000000ULL;
    unsigned long long t = (mx << (kx & 63)) + (my << (ky & 63));  // in [2^62, 2^64)
    const unsigned c = (unsigned)(t >> 32) >> 31;                  // carried past the larger exponent
    const unsigned k = 10u + c;
    t += (unsigned long long)(c * 512u + 511u + (((unsigned)t >> k) & 1u));  // ties to even
    const unsigned long long m = t >> k;  // its leading one (or the carry of the rounding) adds to the exponent
    const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(max(sx, sy) + (int)c - 1) << 20);
    return __hiloint2double((int)hi, (int)(unsigned)m);
}

// Does any lane running here have bad set?
__device__ __forceinline__ bool any_lane(bool bad) { return __any_sync(__activemask(), bad); }

// Keeps a rare branch a branch: made predicated instructions, its FP64 operations would take their
// turns of the pipe on every row.
__device__ __forceinline__ void keep_branch() { __syncwarp(__activemask()); }

struct S64Args {
    const double *u, *b;
    double *out;
    Grid g;
    int ty, chunks;
    int mirror;  // rewrite the odd-reflection ghosts of the 17-point stencil (homogeneous boundary)
    double w, one;
    const double *wtab;  // if not null, the weight is wtab[*pos + k]
    const long long *pos;
    int k;
};

// Rows j0..j1 of column i.  (u is read past L1; through it, the sweep takes the same time.)
template <int ST>
__device__ __forceinline__ void march64(const S64Args &a, int i, int j0, int j1, double w) {
    using C = Co<double>;
    const long long P = a.g.pitch;
    const double one = a.one;
    const double *row = a.u + a.g.idx(i, j0 - (ST == 17 ? 2 : 1));
    const double *bp = a.b + a.g.idx(i, j0);
    double *op = a.out + a.g.idx(i, j0);
    auto add = [&](double x, double y) { return fma(x, one, y); };
    if constexpr (ST == 5) {
        double um = __ldcg(row);
        row += P;
        double uc = __ldcg(row);
        double nu = __ldcg(row + P), nl = __ldcg(row - 1), nr = __ldcg(row + 1), nb = __ldcs(bp);
#pragma unroll 2
        for (int j = j0; j <= j1; ++j) {
            const double up = nu, l = nl, r = nr, bk = nb;
            const long long step = j < j1 ? P : 0;  // the last row loads itself again
            row += step;
            bp += step;
            nu = __ldcg(row + P);
            nl = __ldcg(row - 1);
            nr = __ldcg(row + 1);
            nb = __ldcs(bp);
            const double f = fma(C::c5(), uc, -bk);
            bool bad = false;
            const double v1 = add_int(um, up, bad), p0 = add_int(l, r, bad);
            double s = add_int(p0, v1, bad);
            if (any_lane(bad || range_bad(p0))) {
                keep_branch();
                s = add(add(l, r), add(um, up));
            }
            *op = fma(w, add(s, f), uc);
            op += P;
            um = uc;
            uc = up;
        }
    } else if constexpr (ST == 9) {
        double um = __ldcg(row);
        double pm = add(__ldcg(row - 1), __ldcg(row + 1));
        row += P;
        double uc = __ldcg(row);
        double pc = add(__ldcg(row - 1), __ldcg(row + 1));
        row += P;
        bool rm = range_bad(pm), rc = range_bad(pc);
        double nu = __ldcg(row), nl = __ldcg(row - 1), nr = __ldcg(row + 1), nb = __ldcs(bp);
#pragma unroll 2
        for (int j = j0; j <= j1; ++j) {
            const double up = nu, l = nl, r = nr, bk = nb;
            const long long step = j < j1 ? P : 0;
            row += step;
            bp += step;
            nu = __ldcg(row);
            nl = __ldcg(row - 1);
            nr = __ldcg(row + 1);
            nb = __ldcs(bp);
            bool bad = rm || rc;
            const double v1 = add_int(um, up, bad);
            double pp = add_int(l, r, bad);
            double d = add_int(pm, pp, bad), s = add_int(pc, v1, bad);
            bool rp = range_bad(pp);
            if (any_lane(bad || rp)) {
                keep_branch();
                pp = add(l, r);
                s = add(pc, add(um, up));
                d = add(pm, pp);
                rp = range_bad(pp);
            }
            const double res = fma(C::ax9(), s, fma(C::dg9(), d, fma(C::cc9(), uc, -bk)));
            *op = fma(w, res, uc);
            op += P;
            um = uc;
            uc = up;
            pm = pc;
            pc = pp;
            rm = rc;
            rc = rp;
        }
    } else {
        // rows j-2 .. j+1 in registers on entry to each iteration
        double u_[4], p_[4], Q_[4];
        bool rp_[4], rq_[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            u_[k] = __ldcg(row);
            p_[k] = add(__ldcg(row - 1), __ldcg(row + 1));
            Q_[k] = add(__ldcg(row - 2), __ldcg(row + 2));
            rp_[k] = range_bad(p_[k]);
            rq_[k] = range_bad(Q_[k]);
            row += P;
        }
        double n0 = __ldcg(row), nl = __ldcg(row - 1), nr = __ldcg(row + 1), nl2 = __ldcg(row - 2),
               nr2 = __ldcg(row + 2), nb = __ldcs(bp);
#pragma unroll 1
        for (int j = j0; j <= j1; ++j) {
            const double u4 = n0, l = nl, r = nr, l2 = nl2, r2 = nr2, bk = nb;
            const long long step = j < j1 ? P : 0;
            row += step;
            bp += step;
            n0 = __ldcg(row);
            nl = __ldcg(row - 1);
            nr = __ldcg(row + 1);
            nl2 = __ldcg(row - 2);
            nr2 = __ldcg(row + 2);
            nb = __ldcs(bp);
            bool bad = rq_[0] || rp_[1] || rp_[2] || rq_[2];
            const double v1 = add_int(u_[1], u_[3], bad), v2 = add_int(u_[0], u4, bad);
            double p4 = add_int(l, r, bad), Q4 = add_int(l2, r2, bad);
            double d2 = add_int(Q_[0], Q4, bad), d1 = add_int(p_[1], p_[3], bad);
            double a1 = add_int(p_[2], v1, bad), a2 = add_int(Q_[2], v2, bad);
            bool rp = range_bad(p4), rq = range_bad(Q4);
            if (any_lane(bad || rp || rq)) {
                keep_branch();
                p4 = add(l, r);
                Q4 = add(l2, r2);
                a1 = add(p_[2], add(u_[1], u_[3]));
                a2 = add(Q_[2], add(u_[0], u4));
                d1 = add(p_[1], p_[3]);
                d2 = add(Q_[0], Q4);
                rp = range_bad(p4);
                rq = range_bad(Q4);
            }
            const double res =
                fma(C::a1(), a1, fma(C::a2(), a2, fma(C::d1(), d1, fma(C::d2(), d2, fma(C::cc17(), u_[2], -bk)))));
            const double v = fma(w, res, u_[2]);
            if (a.mirror)
                store_node<2, double>(a.out, a.g, i, j, v);
            else
                *op = v;
            op += P;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                u_[k] = u_[k + 1];
                p_[k] = p_[k + 1];
                Q_[k] = Q_[k + 1];
                rp_[k] = rp_[k + 1];
                rq_[k] = rq_[k + 1];
            }
            u_[3] = u4;
            p_[3] = p4;
            Q_[3] = Q4;
            rp_[3] = rp;
            rq_[3] = rq;
        }
    }
}

template <int ST>
__global__ void __launch_bounds__(kS64Threads) sweep64_kernel(const __grid_constant__ S64Args a) {
    const int t = (int)(blockIdx.x * kS64Threads + threadIdx.x);
    const int ch = t / a.g.Nx, i = t - ch * a.g.Nx + 1;
    const double w = a.wtab ? a.wtab[*a.pos + a.k] : a.w;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");  // the previous sweep's end
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    if (ch >= a.chunks) return;
    const int j0 = ch * a.ty + 1;
    march64<ST>(a, i, j0, min(j0 + a.ty - 1, a.g.Ny), w);
}

cudaError_t s64_launch(const cj_plan *p, S64Args &a, cudaStream_t s) {
    a.g = p->g64;
    a.ty = p->s64.ty;
    a.chunks = p->s64.chunks;
    a.one = 1.0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)p->s64.blocks);
    cfg.blockDim = dim3(kS64Threads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&a};
    const void *fn = p->st == 5   ? (const void *)sweep64_kernel<5>
                     : p->st == 9 ? (const void *)sweep64_kernel<9>
                                  : (const void *)sweep64_kernel<17>;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace

// Rows per thread.  Blocks of both kinds of row cost (FP64 rows at the boundary) and the sweep's tail
// even out over 32 blocks an SM (9-point 4096^2: 148 us a sweep with 16, 138 with 32), but a
// chunk's first rows (two or four rows of sums) should serve four rows (9-point 1024^2: 11.5 us at
// 4 rows, 11.65 at 3, 11.7 at 2) unless that leaves fewer than 16 blocks an SM; the 9- and 17-point
// marches go no lower than 2 rows (9-point 400 x 300: 3.1 us, at 1 row 3.7; 17-point 500 x 400: 7.4 and 8.2).
Sweep64Shape sweep64_shape(int Nx, int Ny, int st) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
    const long long nodes = (long long)Nx * Ny, threads = (long long)sms * kS64Threads;
    auto rows = [&](int per_sm) { return (nodes + threads * per_sm - 1) / (threads * per_sm); };
    long long ty = rows(16) < 4 ? rows(16) : 4;
    if (rows(32) > ty) ty = rows(32);
    if (st != 5 && ty < 2) ty = 2;
    if (ty > Ny) ty = Ny;
    Sweep64Shape s;
    s.ty = (int)ty;
    s.chunks = (int)((Ny + ty - 1) / ty);
    s.blocks = (int)(((long long)Nx * s.chunks + kS64Threads - 1) / kS64Threads);
    return s;
}

cudaError_t launch_sweep64(const cj_plan *p, const double *u, double *out, double w, cudaStream_t s) {
    S64Args a{};
    a.u = u;
    a.b = p->b;
    a.out = out;
    a.w = w;
    a.mirror = p->bc == CJ_BC_DIRICHLET0;
    return s64_launch(p, a, s);
}

cudaError_t launch_sweep64_err(const cj_plan *p, const double *e, const double *rhs, double *out, double w,
                               cudaStream_t s) {
    S64Args a{};
    a.u = e;
    a.b = rhs;
    a.out = out;
    a.w = w;
    a.mirror = 1;
    return s64_launch(p, a, s);
}

cudaError_t launch_sweep64_tab(const cj_plan *p, const double *u, double *out, int k, cudaStream_t s) {
    S64Args a{};
    a.u = u;
    a.b = p->b;
    a.out = out;
    a.wtab = p->w_dev;
    a.pos = p->pos;
    a.k = k;
    a.mirror = p->bc == CJ_BC_DIRICHLET0;
    return s64_launch(p, a, s);
}
