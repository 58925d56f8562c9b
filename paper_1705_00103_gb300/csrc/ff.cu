// FP64-accuracy weighted sweeps evaluated on the FP32 pipe, in float-float arithmetic.
//
// GB300 issues FP64 fused multiply-adds at ~1/74 of its FP32 rate, so the FP64 sweep (every one
// of its 8 operations per 9-point update an FP64 instruction) is bound by the FP64 pipe at ~0.22
// of the HBM bandwidth.  Here the iterate and b are held as unevaluated pairs of floats, hi + lo
// with |lo| <= ulp(hi)/2 (48 significant bits against FP64's 53), and the sweep
// u' = u + w (L u - b) of Sec. 2.1 is evaluated with the error-free transformations of Knuth
// (TwoSum: s + e = a + b exactly) and Dekker (TwoProduct, here in its fused-multiply-add form:
// p + e = a b exactly).  17 points: in the evaluation order of the FP64 sweep.  5 and 9 points: in
// the algebraically equal scaled form
//   u' = (1 - c w / D) u + (w / D) (S - D b),
// S the neighbour sum of D L u + c u with coefficients 1 and 4 (D = 1, c = 4 for 5 points; D = 6,
// c = 20 for 9 points, Eq. 1 times 6): S needs float-float adds and one exact scaling by 4, D b is
// formed once on import, and w / D and 1 - c w / D are rounded once per sweep on the host
// -- 69 and 91 FP32 operations per update against 80 and 116 for the three float-float
// multiply-adds of the FP64 sweep's form.  The pair occupies the same 8 bytes as a double,
// so the sweep moves the FP64 sweep's bytes with FP32 instructions only.  The result is not the
// FP64 sweep's bits: it agrees with it to a few units of 2^-47 of the terms it adds (in the scaled
// form, |c1 u| and |w / D| |S - D b|, each at most about 3.4 |w| max|u| + |w| max|b| for 9 points), well
// inside the per-sweep tolerance of 1e-12 x (max|u| + |w| (9 max|u| + max|b|)) the sweeps are held to.
//
// What bounds it: HBM (24 bytes a node) for 5 and 9 points, FP32 issue for 17 (about 190 operations
// a node).  A thread
// holds two adjacent columns as pairs (hi, hi) and (lo, lo), so that every operation is one packed
// instruction for both, and walks ty rows with the next row's loads one iteration ahead.  In memory
// a pair of columns is (hi, hi, lo, lo), 16 bytes: one load brings both operands of the packed
// instructions to their registers.  The import writes this form straight from the caller's arrays
// and the export reads it, so no conversion passes stand between them and the sweeps.  Values must
// lie in the float range (|d| < 3.4e38); below 2^-126 their low part is lost (relative error 2^-24
// of a value that small).  Homogeneous-Dirichlet plans only: their ghost ring is 0 or the
// reflection of the interior, which the sweeps rewrite.
//
// Measured on one GB300, 4095 x 4001 (one column a thread with scalar operations and conversion
// passes -> this): 9 points 83.7 -> 67.0 us a sweep (245 Gupd/s, 0.88 of the copy bandwidth), 5
// points 68.2 -> 64.0, 17 points 167 -> 121; import and export 1190 -> 177 us; 9-point 333 x 250:
// 5.7 -> 2.3 us a sweep.
#include "cj_internal.h"

namespace {

struct ff {
    float hi, lo;
};

// float-float of a double, rounded once per part
__host__ __device__ __forceinline__ ff ff_of(double d) {
    const float hi = (float)d;
    return ff{hi, (float)(d - (double)hi)};
}

// The same on the integer pipe (a conversion between the types occupies the FP64 pipe like an
// operation, and ff_of takes four): the mantissa rounded to 24 bits, ties to even, and the remainder,
// below 2^29, as an integer.  Zeros, and values whose parts leave the normal float range, go the other way.
__device__ __forceinline__ ff ff_of_bits(double d) {
    const unsigned hw = (unsigned)__double2hiint(d), lw = (unsigned)__double2loint(d);
    const int e = (int)(hw >> 20 & 0x7ffu) - 1023;
    if ((unsigned)(e + 73) > 199u)  // not 2^-73 <= |d| < 2^127
        return (hw << 1 | lw) == 0 ? ff{__uint_as_float(hw), 0.0f} : ff_of(d);
    const unsigned m = __funnelshift_l(lw, hw & 0xfffffu | 0x100000u, 3);  // leading 24 bits
    const unsigned rest = lw & 0x1fffffffu;
    const unsigned up = (rest + 0x0fffffffu + (m & 1u)) >> 29;
    const int rem = (int)rest - (int)(up << 29);
    const unsigned sign = hw & 0x80000000u;
    const float hi = __uint_as_float(sign | (((unsigned)(e + 126) << 23) + m + up));
    const float unit = __uint_as_float(sign | ((unsigned)(e + 75) << 23));  // 2^(e - 52), signed
    return ff{hi, (float)rem * unit};
}

// fl64 of a float, on the integer pipe where it is normal or 0
__device__ __forceinline__ double double_of(float x) {
    const unsigned b = __float_as_uint(x), e = b >> 23 & 0xffu;
    if (e - 1u > 253u) return (b << 1) == 0 ? __hiloint2double((int)b, 0) : (double)x;
    return __hiloint2double((int)((b & 0x80000000u) | ((b & 0x7fffffffu) >> 3) + (896u << 20)), (int)(b << 29));
}

// ---- two columns' values, packed: each half rounded like the scalar instruction

__device__ __forceinline__ float2 bc(float c) { return make_float2(c, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, bc(-1.0f), a); }

struct ff2 {
    float2 h, l;
};

__device__ __forceinline__ ff2 ff2_of(const float4 &q) { return ff2{make_float2(q.x, q.y), make_float2(q.z, q.w)}; }

// Dekker's FastTwoSum: s + e = a + b exactly when |a| >= |b| (or a = 0).
__device__ __forceinline__ ff2 fast_two_sum(float2 a, float2 b) {
    const float2 s = add2(a, b);
    return ff2{s, sub2(b, sub2(s, a))};
}

// a + b: Knuth's TwoSum of the high parts (6 operations, no condition on |a|, |b|), the low parts
// added to its error, renormalised; the error is a few units of 2^-47 of |a| + |b|.
__device__ __forceinline__ ff2 ff_add(const ff2 &a, const ff2 &b) {
    const float2 s = add2(a.h, b.h), bb = sub2(s, a.h);
    const float2 e = add2(sub2(a.h, sub2(s, bb)), sub2(b.h, bb));
    return fast_two_sum(s, add2(e, add2(a.l, b.l)));
}

// 4 a + b: the same with 4 a, which is exact, inside the operations that read a
__device__ __forceinline__ ff2 ff_add4(const ff2 &a, const ff2 &b) {
    const float2 four = bc(4.0f);
    const float2 s = fma2(a.h, four, b.h), bb = fma2(a.h, bc(-4.0f), s);
    const float2 e = add2(fma2(a.h, four, sub2(bb, s)), sub2(b.h, bb));
    return fast_two_sum(s, add2(e, fma2(a.l, four, b.l)));
}

// c a for a constant c: the exact product of the high parts by a fused multiply-add (TwoProduct),
// formed negated for it, the cross terms added to its error, renormalised.
__device__ __forceinline__ ff2 ff_mul(ff c, const ff2 &a) {
    const float2 np = __fmul2_rn(bc(-c.hi), a.h);
    float2 e = fma2(bc(c.hi), a.h, np);
    e = fma2(bc(c.hi), a.l, e);
    e = fma2(bc(c.lo), a.h, e);
    const float2 s = sub2(e, np);
    return ff2{s, sub2(e, add2(s, np))};
}

// c a + b
__device__ __forceinline__ ff2 ff_fma(ff c, const ff2 &a, const ff2 &b) { return ff_add(ff_mul(c, a), b); }

// ---- the packed grid: node k of the padded layout has its high part at float 4 (k / 2) + k % 2 and
// its low part two floats on; columns c, c + 1 with odd c share 16 bytes

__host__ __device__ __forceinline__ long long ff_pos(long long k) { return ((k >> 1) << 2) + (k & 1); }

__device__ __forceinline__ void ff_put(float *a, long long k, ff v) {
    a[ff_pos(k)] = v.hi;
    a[ff_pos(k) + 2] = v.lo;
}

// Writes v at interior node (i, j) and, for the 17-point stencil, the reflections that mirror it.
template <int R>
__device__ __forceinline__ void ff_store(float *a, const Grid &g, int i, int j, ff v) {
    ff_put(a, g.idx(i, j), v);
    if (R == 2) {
        const ff nv{-v.hi, -v.lo};
        const bool x0 = i == 1, x1 = i == g.Nx;
        if (x0) ff_put(a, g.idx(-1, j), nv);
        if (x1) ff_put(a, g.idx(g.Nx + 2, j), nv);
        if (j == 1) {
            ff_put(a, g.idx(i, -1), nv);
            if (x0) ff_put(a, g.idx(-1, -1), v);
            if (x1) ff_put(a, g.idx(g.Nx + 2, -1), v);
        }
        if (j == g.Ny) {
            ff_put(a, g.idx(i, g.Ny + 2), nv);
            if (x0) ff_put(a, g.idx(-1, g.Ny + 2), v);
            if (x1) ff_put(a, g.idx(g.Nx + 2, g.Ny + 2), v);
        }
    }
}

// The weights of one sweep.  17 points: w, for u' = u + w (L u - b) in the FP64 sweep's order.
// 5 and 9 points, in the scaled form D L u = sum of the neighbours with small integer
// coefficients - c u (D = 1, c = 4; D = 6, c = 20), with b stored as -D b:
//   u' = c1 u + wD (D L u + c u - D b),   wD = w / D,   c1 = 1 - c wD,
// so the neighbour sum needs no multiplication (its coefficients 1 and 4 are powers of two).
struct FFArgs {
    const float *u, *nb;
    float *out;
    Grid g;
    int ty, chunks;
    ff w, wD, c1;
};

constexpr int kFFThreads = 128;

// One row of a thread's pair of columns: the pair, and the pairs to its left and right.
struct FFRow {
    float4 l, c, r;
};

__device__ __forceinline__ FFRow ff_row(const float4 *p) { return FFRow{__ldca(p - 1), __ldca(p), __ldca(p + 1)}; }

// u(i-1) + u(i+1) and u(i-2) + u(i+2) of both columns
__device__ __forceinline__ ff2 ff_side1(const FFRow &q) {
    return ff_add(ff2{make_float2(q.l.y, q.c.x), make_float2(q.l.w, q.c.z)},
                  ff2{make_float2(q.c.y, q.r.x), make_float2(q.c.w, q.r.z)});
}
__device__ __forceinline__ ff2 ff_side2(const FFRow &q) { return ff_add(ff2_of(q.l), ff2_of(q.r)); }

// One weighted sweep out = u + w (L u - b): thread t has pair t mod np of chunk t / np, rows
// chunk ty + 1 onwards.  Its launches overlap the end of the one before (programmatic dependent launch,
// cj_internal.h).
template <int ST>
__global__ void __launch_bounds__(kFFThreads, ST == 17 ? 4 : 7) sweep_ff_kernel(const __grid_constant__ FFArgs a) {
    constexpr int R = ST == 17 ? 2 : 1;
    const Grid &g = a.g;
    const int np = (g.Nx + 1) / 2;
    const int t = (int)(blockIdx.x * kFFThreads + threadIdx.x);
    const int ch = t / np, i = 2 * (t - ch * np) + 1;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    if (ch >= a.chunks) return;
    const int j0 = ch * a.ty + 1, j1 = min(j0 + a.ty - 1, g.Ny);
    const long long P = g.pitch / 2;  // pairs per row
    const bool both = i < g.Nx;
    const float4 *row = reinterpret_cast<const float4 *>(a.u) + g.idx(i, j0 - R) / 2;
    const float4 *bp = reinterpret_cast<const float4 *>(a.nb) + g.idx(i, j0) / 2;
    float4 *op = reinterpret_cast<float4 *>(a.out) + g.idx(i, j0) / 2;
    auto store = [&](int j, const ff2 &v) {
        const bool edge = R == 2 && (i == 1 || i + 1 >= g.Nx || j == 1 || j == g.Ny);
        if (both && !edge) {
            *op = make_float4(v.h.x, v.h.y, v.l.x, v.l.y);
        } else {
            ff_store<R>(a.out, g, i, j, ff{v.h.x, v.l.x});
            if (both) ff_store<R>(a.out, g, i + 1, j, ff{v.h.y, v.l.y});
        }
        op += P;
    };
    if constexpr (ST != 17) {
        ff2 um = ff2_of(__ldca(row)), pm, pc;
        if (ST == 9) pm = ff_side1(ff_row(row));
        row += P;
        FFRow c = ff_row(row);  // 5 points: row j; 9 points: of row j only the pair is used in the loop
        ff2 uc = ff2_of(c.c);
        if (ST == 9) {
            pc = ff_side1(c);
            row += P;
        }
        // 5 points: row j's sides and row j + 1's pair; 9 points: row j + 1
        FFRow n = ST == 9 ? ff_row(row) : FFRow{c.l, __ldca(row + P), c.r};
        float4 nb = __ldcs(bp);
#pragma unroll 2
        for (int j = j0; j <= j1; ++j) {
            const FFRow q = n;
            const ff2 bk = ff2_of(nb), up = ff2_of(q.c);
            const long long step = j < j1 ? P : 0;  // the last row loads itself again
            row += step;
            bp += step;
            n = ff_row(row);
            if (ST == 5) n.c = __ldca(row + P);
            nb = __ldcs(bp);
            ff2 s;
            if (ST == 5) {
                const FFRow e{q.l, make_float4(uc.h.x, uc.h.y, uc.l.x, uc.l.y), q.r};
                s = ff_add(ff_side1(e), ff_add(um, up));
            } else {
                const ff2 pp = ff_side1(q);
                s = ff_add4(ff_add(pc, ff_add(um, up)), ff_add(pm, pp));
                pm = pc;
                pc = pp;
            }
            store(j, ff_add(ff_mul(a.c1, uc), ff_mul(a.wD, ff_add(s, bk))));
            um = uc;
            uc = up;
        }
    } else {
        // rows j-2 .. j+1 in registers on entry to each iteration: the pair and its side sums
        ff2 u_[4], p_[4], Q_[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const FFRow q = ff_row(row);
            u_[k] = ff2_of(q.c);
            p_[k] = ff_side1(q);
            Q_[k] = ff_side2(q);
            row += P;
        }
        FFRow n = ff_row(row);
        float4 nb = __ldcs(bp);
#pragma unroll 1
        for (int j = j0; j <= j1; ++j) {
            const FFRow q = n;
            const ff2 bk = ff2_of(nb), u4 = ff2_of(q.c);
            const long long step = j < j1 ? P : 0;
            row += step;
            bp += step;
            n = ff_row(row);
            nb = __ldcs(bp);
            const ff2 p4 = ff_side1(q), Q4 = ff_side2(q);
            const ff2 a1 = ff_add(p_[2], ff_add(u_[1], u_[3])), a2 = ff_add(Q_[2], ff_add(u_[0], u4));
            const ff2 d1 = ff_add(p_[1], p_[3]), d2 = ff_add(Q_[0], Q4);
            const ff2 r = ff_fma(
                ff_of(64.0 / 72.0), a1,
                ff_fma(ff_of(-4.0 / 72.0), a2,
                       ff_fma(ff_of(16.0 / 72.0), d1,
                              ff_fma(ff_of(-1.0 / 72.0), d2, ff_fma(ff_of(-300.0 / 72.0), u_[2], bk)))));
            store(j, ff_fma(a.w, r, u_[2]));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                u_[k] = u_[k + 1];
                p_[k] = p_[k + 1];
                Q_[k] = Q_[k + 1];
            }
            u_[3] = u4;
            p_[3] = p4;
            Q_[3] = Q4;
        }
    }
}

// Caller grids -> packed u and nb = -D h^2 f.
template <int R>
__global__ void __launch_bounds__(kBX) import_ff_kernel(const double *__restrict__ f, long long ldf,
                                                        const double *__restrict__ uin, long long ldu, float *nb,
                                                        float *u, Grid g, double h2, double D) {
    const int i = blockIdx.x * kBX + threadIdx.x + 1;
    if (i > g.Nx) return;
    for (int j = blockIdx.y + 1; j <= g.Ny; j += gridDim.y) {
        const double bk = h2 * f[(long long)(j - 1) * ldf + (i - 1)];
        ff_put(nb, g.idx(i, j), ff_of_bits(-(D * bk)));
        ff_store<R>(u, g, i, j, ff_of_bits(uin[(long long)(j - 1) * ldu + (i - 1)]));
    }
}

// Packed interior -> caller grid.
__global__ void __launch_bounds__(kBX) export_ff_kernel(const float *__restrict__ src, Grid g, double *u,
                                                        long long ldu) {
    const int i = blockIdx.x * kBX + threadIdx.x + 1;
    if (i > g.Nx) return;
    for (int j = blockIdx.y + 1; j <= g.Ny; j += gridDim.y) {
        const long long k = ff_pos(g.idx(i, j));
        u[(long long)(j - 1) * ldu + (i - 1)] = double_of(src[k]) + double_of(src[k + 2]);
    }
}

// Zeroes the 16-byte pairs of both solution buffers that hold a ghost column: before the sweeps and
// after them, as the pairs share their bytes differently in the two forms.  (The interior is
// written before it is read, in either form, and so are the reflections of the 17-point stencil.)
__global__ void __launch_bounds__(256) ghost_pairs_kernel(double *u0, double *u1, Grid g) {
    const int j = (int)(blockIdx.x * 256 + threadIdx.x) - 1;
    if (j > g.Ny + 2) return;
    double *row[2] = {u0 + g.idx(1, j), u1 + g.idx(1, j)};
    const int first = g.Nx & ~1;  // column offset of the first pair with a column past Nx
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        row[q][-2] = row[q][-1] = 0.0;
        row[q][first] = row[q][first + 1] = 0.0;
        if (first < g.Nx) row[q][first + 2] = row[q][first + 3] = 0.0;
    }
}

cudaError_t ghost_pairs(const cj_plan *p, cudaStream_t s) {
    ghost_pairs_kernel<<<(p->Ny + 4 + 255) / 256, 256, 0, s>>>(p->u0, p->u1, p->g64);
    return cudaGetLastError();
}

// D and c of the scaled form of the 5- and 9-point sweeps (1 for 17 points, which keeps the
// FP64 sweep's form).
double ff_scale(int st) { return st == 9 ? 6.0 : 1.0; }
double ff_centre(int st) { return st == 9 ? 20.0 : 4.0; }

cudaError_t launch_sweep_ff(const cj_plan *p, FFArgs &a, cudaStream_t s) {
    const Grid &g = p->g64;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
    const long long np = (g.Nx + 1) / 2, threads = (long long)sms * kFFThreads;
    // about 28 blocks an SM even out the sweep's end (at 10, a wave and a half, 9 points take 73.6 us on
    // 4095 x 4001 against 67); on small grids a chunk's first rows should serve 4 rows (9-point
    // 1024 x 1000: 5.85 us, at 2 rows 6.4) unless that leaves fewer than 7 blocks an SM
    auto rows = [&](int per_sm) { return (np * g.Ny + threads * per_sm - 1) / (threads * per_sm); };
    long long ty = rows(7) < 4 ? rows(7) : 4;
    if (rows(28) > ty) ty = rows(28);
    if (ty < 2) ty = 2;
    if (ty > g.Ny) ty = g.Ny;
    a.g = g;
    a.ty = (int)ty;
    a.chunks = (int)((g.Ny + ty - 1) / ty);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)((np * a.chunks + kFFThreads - 1) / kFFThreads));
    cfg.blockDim = dim3(kFFThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    void *args[] = {(void *)&a};
    const void *fn = p->st == 5   ? (const void *)sweep_ff_kernel<5>
                     : p->st == 9 ? (const void *)sweep_ff_kernel<9>
                                  : (const void *)sweep_ff_kernel<17>;
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace

bool ff_sweeps_supported(const cj_plan *p) {
    return p && p->precision == CJ_FP64 && p->pattern == 0 && p->bc == CJ_BC_DIRICHLET0 && p->u1;
}

cudaError_t launch_sweeps_ff(const cj_plan *p, const double *f, long long ldf, double *u, long long ldu,
                             long long first, long long count, cudaStream_t s) {
    float *buf[2] = {reinterpret_cast<float *>(p->u0), reinterpret_cast<float *>(p->u1)};
    float *nb = reinterpret_cast<float *>(p->b);
    const double D = ff_scale(p->st);
    const dim3 grid((p->Nx + kBX - 1) / kBX, p->Ny < 1024 ? p->Ny : 1024);
    cudaError_t e = ghost_pairs(p, s);
    if (e != cudaSuccess) return e;
    if (p->st == 17)
        import_ff_kernel<2><<<grid, kBX, 0, s>>>(f, ldf, u, ldu, nb, buf[0], p->g64, p->h2, D);
    else
        import_ff_kernel<1><<<grid, kBX, 0, s>>>(f, ldf, u, ldu, nb, buf[0], p->g64, p->h2, D);
    e = cudaGetLastError();
    int cur = 0;
    for (long long k = 0; k < count && e == cudaSuccess; ++k) {
        const double wk = p->w[(first + k) % p->M], wD = wk / D;
        FFArgs a{};
        a.u = buf[cur];
        a.nb = nb;
        a.out = buf[cur ^ 1];
        a.w = ff_of(wk);
        a.wD = ff_of(wD);
        a.c1 = ff_of(1.0 - ff_centre(p->st) * wD);
        e = launch_sweep_ff(p, a, s);
        cur ^= 1;
    }
    if (e == cudaSuccess) {
        export_ff_kernel<<<grid, kBX, 0, s>>>(buf[cur], p->g64, u, ldu);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = ghost_pairs(p, s);
    return e;
}
