// Register tiles: temporal blocking of the FP32 inner sweep with the iterate held in registers.
//
// A block of NW warps stages 128 columns x NW * RPT rows of the grid: warp q owns rows
// q * RPT .. q * RPT + RPT - 1, each lane four adjacent columns of them, in registers, and the
// right-hand side r sits in shared memory (each lane reads back only what it copied).  The block
// then runs k weighted sweeps e <- e + w_n (L e - r) in place, one block barrier per sweep: a warp
// publishes its first and last R rows (R the stencil's radius) in shared memory, reads its
// neighbours', and marches down its rows carrying each row's differences, so every difference is
// formed once (a row's old values are not needed once the row below it has its differences).
// Side columns come from the neighbouring lanes by shuffles.  Every sweep loses R columns and R
// rows of validity on each side of the staged tile, so the tile's inner part is stored after k
// sweeps: 128 - 2 ceil4(R k) columns (whole lanes) and NW * RPT - 2 R k rows.
//
// What bounds it: instruction issue.  A row of four 9-point nodes takes 37 FP32 operations, two
// shuffles and one shared-memory load (10.6 instructions per staged node and sweep with the
// exchange).  The alternative, one warp streaming down a strip with all k stages in registers,
// spends 17.7 instructions per update (ring addressing, row tests, window moves) at 8 warps per
// SM.  HBM traffic per update is (8 B in + 4 B out) / k times the tile's overlap.
//
// Boundaries: the tile is staged on the odd extension of the grid in both directions
// (fold_dev.cuh): nodes 0 and N + 1 are 0 and stay 0, and every operation of the sweep is an odd
// function of its inputs under round-to-nearest, so the reflected nodes stay the exact negatives
// of their mirrors and no node of the sweep needs a boundary test.  The operation order per node
// is resid_diff32's, so results equal one-sweep launches bit for bit.
#pragma once

#include "cj_internal.h"
#include "fold_dev.cuh"
#include "grid_dev.cuh"
#include "stencil_dev.cuh"

namespace {

__device__ __forceinline__ void rt_cp_async16(void *dst, const void *src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// The launches of one inner cycle follow one another with programmatic dependent launch (cj_internal.h):
// a block may start while the previous launch drains, stages r (which no sweep writes, nor the launch
// before a cycle's first), and waits here for that launch's end before it reads e or writes; only
// then may the launch after this one start.  (e is read past L1: a block reads each node once.)
__device__ __forceinline__ void rt_wait_previous() {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// Shared memory of one block, in float4: r of the staged rows, then the exchanged rows of two
// sweeps (each warp's first R and last R rows).
template <int ST, int RPT, int NW>
struct RtShape {
    static constexpr int R = ST == 17 ? 2 : 1;
    static constexpr int rows = NW * RPT;
    static constexpr int r_vecs = rows * 32;
    static constexpr int x_vecs = 2 * NW * 2 * R * 32;
    static constexpr int smem_bytes = (r_vecs + x_vecs) * 16;
    static_assert(RPT >= R, "a warp's neighbours read R of its rows");
    static_assert(RPT <= 32 && 8 * rows <= 8 * x_vecs, "the table of folded rows");
};

// Halo of k sweeps: rows R k, columns rounded up to whole lanes.
__host__ __device__ constexpr int rt_halo_cols(int R, int k) { return (R * k + 3) / 4 * 4; }

// Two adjacent columns' values: the packed FP32 instructions work on both (each half rounded like
// the scalar instruction), at one issue slot instead of two.
__device__ __forceinline__ float2 p2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 p2_sub(float2 a, float2 b) {
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);  // a - b: the product is exact
}
__device__ __forceinline__ float2 p2_of(float c) { return make_float2(c, c); }

// A lane's four columns of a row, as two pairs.
struct Row4 {
    float2 a, b;
};

__device__ __forceinline__ Row4 row4_of(const float4 &q) { return Row4{make_float2(q.x, q.y), make_float2(q.z, q.w)}; }
__device__ __forceinline__ float4 vec_of(const Row4 &r) { return make_float4(r.a.x, r.a.y, r.b.x, r.b.y); }
__device__ __forceinline__ Row4 row4_sub(const Row4 &x, const Row4 &y) {
    return Row4{p2_sub(x.a, y.a), p2_sub(x.b, y.b)};
}
__device__ __forceinline__ Row4 row4_add(const Row4 &x, const Row4 &y) {
    return Row4{p2_add(x.a, y.a), p2_add(x.b, y.b)};
}
// c x + y
__device__ __forceinline__ Row4 row4_fma(float c, const Row4 &x, const Row4 &y) {
    return Row4{p2_fma(p2_of(c), x.a, y.a), p2_fma(p2_of(c), x.b, y.b)};
}
__device__ __forceinline__ Row4 row4_neg(const Row4 &x) {
    return Row4{make_float2(-x.a.x, -x.a.y), make_float2(-x.b.x, -x.b.y)};
}

// Horizontal second difference at spacing 1 of a row's four nodes, from their outer neighbours.
__device__ __forceinline__ Row4 rt_x1(const Row4 &v, float l, float r) {
    const float d0 = v.a.x - l, d1 = v.a.y - v.a.x, d2 = v.b.x - v.a.y, d3 = v.b.y - v.b.x, d4 = r - v.b.y;
    return Row4{make_float2(d1 - d0, d2 - d1), make_float2(d3 - d2, d4 - d3)};
}

__device__ __forceinline__ Row4 rt_row_x1(const Row4 &v) {
    const float l = __shfl_up_sync(0xffffffffu, v.b.y, 1), r = __shfl_down_sync(0xffffffffu, v.a.x, 1);
    return rt_x1(v, l, r);
}

// Horizontal second differences at spacings 1 and 2.
__device__ __forceinline__ void rt_row_x12(const Row4 &v, Row4 &X1, Row4 &X2) {
    float2 l, r;  // columns c0 - 2, c0 - 1 and c0 + 4, c0 + 5
    l.x = __shfl_up_sync(0xffffffffu, v.b.x, 1);
    l.y = __shfl_up_sync(0xffffffffu, v.b.y, 1);
    r.x = __shfl_down_sync(0xffffffffu, v.a.x, 1);
    r.y = __shfl_down_sync(0xffffffffu, v.a.y, 1);
    X1 = rt_x1(v, l.y, r.x);
    const float2 d01 = p2_sub(v.a, l), d23 = p2_sub(v.b, v.a), d45 = p2_sub(r, v.b);
    X2.a = p2_sub(d23, d01);
    X2.b = p2_sub(d45, d23);
}

// One sweep of a warp's RPT rows in place.  above: the R rows above (nearest last), below: the R
// rows below (nearest first); rk: this lane's r of the warp's rows, 32 vectors per row.
template <int ST, int RPT>
__device__ __forceinline__ void rt_sweep(Row4 (&e)[RPT], const Row4 (&above)[ST == 17 ? 2 : 1],
                                         const Row4 (&below)[ST == 17 ? 2 : 1], const float4 *rk, float w) {
    if constexpr (ST != 17) {
        Row4 Xm, Xc;
        if (ST == 9) {
            Xm = rt_row_x1(above[0]);
            Xc = rt_row_x1(e[0]);
        }
        Row4 dS = row4_sub(e[0], above[0]);
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const Row4 n = j + 1 < RPT ? e[j + 1 < RPT ? j + 1 : 0] : below[0];
            const Row4 rv = row4_of(rk[j * 32]);
            const Row4 Xn = rt_row_x1(ST == 9 ? n : e[j]);
            const Row4 dN = row4_sub(n, e[j]);
            const Row4 Y1 = row4_sub(dN, dS);
            Row4 res;
            if (ST == 5) {
                res = row4_sub(row4_add(Xn, Y1), rv);
            } else {
                res = row4_fma(1.0f / 6.0f, row4_add(Xm, Xn), row4_fma(2.0f / 3.0f, Xc, row4_sub(Y1, rv)));
                Xm = Xc;
                Xc = Xn;
            }
            dS = dN;
            e[j] = row4_fma(w, res, e[j]);
        }
    } else {
        // X1 of rows j-1, j, j+1 and X2 of rows j-2 .. j+1 on entry to row j; d1: row j less row
        // j-1, d2a / d2b: rows j and j+1 less the rows two above them
        Row4 X1a, X1b, X1c, X2a, X2b, X2c, X2d, junk;
        rt_row_x12(above[0], junk, X2a);
        rt_row_x12(above[1], X1a, X2b);
        rt_row_x12(e[0], X1b, X2c);
        rt_row_x12(e[1], X1c, X2d);
        Row4 d1 = row4_sub(e[0], above[1]), d2a = row4_sub(e[0], above[0]), d2b = row4_sub(e[1], above[1]);
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
            const Row4 n1 = j + 1 < RPT ? e[j + 1 < RPT ? j + 1 : 0] : below[0];
            const Row4 n2 = j + 2 < RPT ? e[j + 2 < RPT ? j + 2 : 0] : below[j + 2 - RPT > 0 ? 1 : 0];
            const Row4 rv = row4_of(rk[j * 32]);
            Row4 X1n, X2n;
            rt_row_x12(n2, X1n, X2n);
            const Row4 u1 = row4_sub(n1, e[j]), u2 = row4_sub(n2, e[j]);
            const Row4 Y1 = row4_sub(u1, d1), Y2 = row4_sub(u2, d2a);
            const Row4 res = row4_fma(
                2.0f / 9.0f, row4_add(X1a, X1c),
                row4_fma(8.0f / 9.0f, X1b,
                         row4_fma(4.0f / 3.0f, Y1,
                                  row4_fma(-1.0f / 72.0f, row4_add(X2a, X2n),
                                           row4_fma(-1.0f / 18.0f, X2c,
                                                    row4_fma(-1.0f / 12.0f, Y2, row4_neg(rv)))))));
            e[j] = row4_fma(w, res, e[j]);
            d1 = u1;
            d2a = d2b;
            d2b = u2;
            X1a = X1b;
            X1b = X1c;
            X1c = X1n;
            X2a = X2b;
            X2b = X2c;
            X2c = X2d;
            X2d = X2n;
        }
    }
}

// One block's work: k sweeps with weights w[0 .. k-1] of the tile whose output nodes are columns
// ox .. ox + (127 - 2 halo columns) and rows oy0 .. oy1 (clipped to the grid by the caller in y,
// here in x); oy1 - oy0 + 1 <= NW * RPT - 2 R k, ox - 1 a multiple of 4.  All arguments are
// uniform over the block.
template <int ST, int RPT, int NW>
__device__ __forceinline__ void rt_run(const float *e, const float *__restrict__ r, float *out, const Grid &g,
                                       const float *__restrict__ w, int k, int ox, int oy0, int oy1, float4 *sm) {
    using S = RtShape<ST, RPT, NW>;
    constexpr int R = S::R;
    const int lane = (int)threadIdx.x & 31, wid = (int)threadIdx.x >> 5;
    const int H = R * k, HC = rt_halo_cols(R, k);
    const int Nx = g.Nx, Ny = g.Ny;
    const int xs = ox - HC, ys = oy0 - H;
    const int c0 = xs + 4 * lane, yw = ys + wid * RPT;  // this lane's first column, this warp's first row
    float4 *rs = sm + wid * RPT * 32 + lane;
    float4 *xb = sm + S::r_vecs;
    const float wl = lane < k ? w[lane] : 0.0f;

    Row4 v[RPT];
    if (xs >= 1 && xs + 127 <= Nx && ys >= 1 && ys + S::rows - 1 <= Ny) {  // inside the grid: vectors as they are
        const long long q0 = g.idx(c0, yw);
#pragma unroll
        for (int j = 0; j < RPT; ++j) rt_cp_async16(rs + j * 32, r + q0 + j * g.pitch);
        rt_wait_previous();
#pragma unroll
        for (int j = 0; j < RPT; ++j) v[j] = row4_of(__ldcg(reinterpret_cast<const float4 *>(e + q0 + j * g.pitch)));
    } else {
        // at the grid's border every node is read from the node it mirrors (node 1 in place of a
        // Dirichlet node, whose value is then 0).  The staged rows are folded once, by one thread
        // each, into the second sweep's exchange rows (not used before the first sweep's barrier),
        // and the row loops have no branches, so that all rows' loads overlap.
        int *fy = reinterpret_cast<int *>(xb + S::x_vecs / 2);
        float *sy = reinterpret_cast<float *>(fy + S::rows);
        if ((int)threadIdx.x < S::rows) fy[threadIdx.x] = fold(ys + (int)threadIdx.x, Ny, sy[threadIdx.x]);
        const bool whole = c0 >= 1 && c0 + 3 <= Nx;
        float sx[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        int fx[4] = {c0, c0, c0, c0};
        if (!whole) {
#pragma unroll
            for (int m = 0; m < 4; ++m) fx[m] = fold(c0 + m, Nx, sx[m]);
        }
        __syncthreads();
        fy += wid * RPT;
        sy += wid * RPT;
        auto fetch = [&](const float *a) {
            const float *col = a + g.idx(0, 0);
            if (whole) {
#pragma unroll
                for (int j = 0; j < RPT; ++j)
                    v[j] = row4_of(__ldcg(reinterpret_cast<const float4 *>(col + fy[j] * g.pitch + c0)));
            } else {
#pragma unroll
                for (int j = 0; j < RPT; ++j) {
                    const float *row = col + fy[j] * g.pitch;
                    v[j].a = make_float2(__ldcg(row + fx[0]), __ldcg(row + fx[1]));
                    v[j].b = make_float2(__ldcg(row + fx[2]), __ldcg(row + fx[3]));
                }
            }
            auto put = [](float s, float q) { return s == 0.0f ? 0.0f : s * q; };
#pragma unroll
            for (int j = 0; j < RPT; ++j) {
                const float s = sy[j];
                v[j].a = make_float2(put(sx[0] * s, v[j].a.x), put(sx[1] * s, v[j].a.y));
                v[j].b = make_float2(put(sx[2] * s, v[j].b.x), put(sx[3] * s, v[j].b.y));
            }
        };
        fetch(r);
#pragma unroll
        for (int j = 0; j < RPT; ++j) rs[j * 32] = vec_of(v[j]);
        rt_wait_previous();
        fetch(e);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");

    const int wa = wid > 0 ? wid - 1 : 0, wb = wid < NW - 1 ? wid + 1 : wid;  // the outer warps' outer rows are halo
#pragma unroll 1
    for (int s = 0; s < k; ++s) {
        // this sweep's rows of warp q: first R at x + (q 2R) 32, last R at x + (q 2R + R) 32
        float4 *x = xb + (s & 1) * (S::x_vecs / 2) + lane;
#pragma unroll
        for (int q = 0; q < R; ++q) {
            x[(wid * 2 * R + q) * 32] = vec_of(v[q]);
            x[(wid * 2 * R + R + q) * 32] = vec_of(v[RPT - R + q]);
        }
        __syncthreads();
        Row4 above[R], below[R];
#pragma unroll
        for (int q = 0; q < R; ++q) {
            above[q] = row4_of(x[(wa * 2 * R + R + q) * 32]);
            below[q] = row4_of(x[(wb * 2 * R + q) * 32]);
        }
        rt_sweep<ST, RPT>(v, above, below, rs, __shfl_sync(0xffffffffu, wl, s));
    }

    const bool mine = lane >= HC / 4 && lane < 32 - HC / 4 && c0 <= Nx;
    if (!mine) return;
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
        const int y = yw + j;
        if (y < oy0 || y > oy1) continue;
        const bool edge = R == 2 && (c0 == 1 || c0 + 3 >= Nx || y == 1 || y == Ny);
        const float4 o = vec_of(v[j]);
        if (c0 + 3 <= Nx && !edge) {
            *reinterpret_cast<float4 *>(out + g.idx(c0, y)) = o;
        } else {
            const float o4[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
            for (int m = 0; m < 4; ++m)
                if (c0 + m <= Nx) store_node<R, float>(out, g, c0 + m, y, o4[m]);
        }
    }
}

}  // namespace
