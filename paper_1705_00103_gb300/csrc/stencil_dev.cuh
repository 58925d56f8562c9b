// Device arithmetic shared by the kernel translation units: the stencil evaluation in the
// fixed order of the FP64 reference (y-marching and direct forms), and the double-FP64 defect.
#pragma once

#include "cj_internal.h"
#include "grid_dev.cuh"

namespace {

template <typename T>
struct Ar;
template <>
struct Ar<double> {
    static __device__ __forceinline__ double add(double a, double b, double one) {
        return fma(a, one, b);
    }
    static __device__ __forceinline__ double fm(double a, double b, double c) { return fma(a, b, c); }
};

// Stencil coefficients of h^2 Delta_h (Table 3; Eq. 1 and Fig. 1 left; Eq. 2 and Fig. 1
// right), rounded once to the working type.
template <typename T>
struct Co;
template <>
struct Co<double> {
    static __device__ __forceinline__ double c5() { return -4.0; }
    static __device__ __forceinline__ double ax9() { return 4.0 / 6.0; }
    static __device__ __forceinline__ double dg9() { return 1.0 / 6.0; }
    static __device__ __forceinline__ double cc9() { return -20.0 / 6.0; }
    static __device__ __forceinline__ double a1() { return 64.0 / 72.0; }
    static __device__ __forceinline__ double a2() { return -4.0 / 72.0; }
    static __device__ __forceinline__ double d1() { return 16.0 / 72.0; }
    static __device__ __forceinline__ double d2() { return -1.0 / 72.0; }
    static __device__ __forceinline__ double cc17() { return -300.0 / 72.0; }
};

template <typename T>
__device__ __forceinline__ T ld(const T *p) {
    return __ldg(p);
}

// Walks rows j0..j1 of column i and calls op(j, r, u(i,j)) with r = (L u - b)(i, j).
template <int ST, typename T, class Op>
__device__ __forceinline__ void march(const T *__restrict__ u, const T *__restrict__ b,
                                      const Grid &g, int i, int j0, int j1, T one, Op &op) {
    using A = Ar<T>;
    using C = Co<T>;
    const long long P = g.pitch;
    const T *col = u + g.idx(i, 0);  // node (i, 0); row k at col + k * P
    const T *bcol = b + g.idx(i, 0);
    if (ST == 5) {
        T um = ld(col + (long long)(j0 - 1) * P);
        T uc = ld(col + (long long)j0 * P);
        for (int j = j0; j <= j1; ++j) {
            const T *row = col + (long long)j * P;
            T up = ld(row + P);
            T p0 = A::add(ld(row - 1), ld(row + 1), one);
            T v1 = A::add(um, up, one);
            T bk = ld(bcol + (long long)j * P);
            T a = A::add(p0, v1, one);
            T r = A::add(a, A::fm(C::c5(), uc, -bk), one);
            op(j, r, uc);
            um = uc;
            uc = up;
        }
    } else if (ST == 9) {
        const T *row = col + (long long)(j0 - 1) * P;
        T um = ld(row);
        T pm = A::add(ld(row - 1), ld(row + 1), one);
        row += P;
        T uc = ld(row);
        T pc = A::add(ld(row - 1), ld(row + 1), one);
        for (int j = j0; j <= j1; ++j) {
            row = col + (long long)(j + 1) * P;
            T up = ld(row);
            T pp = A::add(ld(row - 1), ld(row + 1), one);
            T bk = ld(bcol + (long long)j * P);
            T v1 = A::add(um, up, one);
            T a = A::add(pc, v1, one);
            T d = A::add(pm, pp, one);
            T r = A::fm(C::ax9(), a, A::fm(C::dg9(), d, A::fm(C::cc9(), uc, -bk)));
            op(j, r, uc);
            um = uc;
            uc = up;
            pm = pc;
            pc = pp;
        }
    } else {
        // rows j-2 .. j+1 in registers on entry to each iteration; row j+2 loaded in it
        T u_[4], p_[4], Q_[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const T *row = col + (long long)(j0 - 2 + k) * P;
            u_[k] = ld(row);
            p_[k] = A::add(ld(row - 1), ld(row + 1), one);
            Q_[k] = A::add(ld(row - 2), ld(row + 2), one);
        }
        for (int j = j0; j <= j1; ++j) {
            const T *row = col + (long long)(j + 2) * P;
            T u4 = ld(row);
            T p4 = A::add(ld(row - 1), ld(row + 1), one);
            T Q4 = A::add(ld(row - 2), ld(row + 2), one);
            T bk = ld(bcol + (long long)j * P);
            // u_[0..3] = rows j-2, j-1, j, j+1; u4 = row j+2
            T v1 = A::add(u_[1], u_[3], one);
            T v2 = A::add(u_[0], u4, one);
            T a1 = A::add(p_[2], v1, one);
            T a2 = A::add(Q_[2], v2, one);
            T d1 = A::add(p_[1], p_[3], one);
            T d2 = A::add(Q_[0], Q4, one);
            T r = A::fm(C::a1(), a1,
                        A::fm(C::a2(), a2,
                              A::fm(C::d1(), d1, A::fm(C::d2(), d2, A::fm(C::cc17(), u_[2], -bk)))));
            op(j, r, u_[2]);
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



// FP32 residual in second-difference form, L e - rk, from the horizontal and vertical second
// differences at spacing s, X_s(dy) = (e(s, dy) - e(0, dy)) - (e(0, dy) - e(-s, dy)) and
// Y_s = (e(0, s) - e_C) - (e_C - e(0, -s)): every value enters through a neighbour difference,
// so the smooth low modes keep their digits on fine grids where neighbour sums would cancel
// against the centre.  The forms are exact rewritings of the stencils: 5-point X_1(0) + Y_1;
// 9-point (Eq. 1) (X_1(-1) + X_1(1) + 4 X_1(0))/6 + Y_1 ([1 4 1; 4 -20 4; 1 4 1] is [1 4 1]
// across x times [1 4 1] across y, less 36 at the centre); 17-point (Eq. 2) 16/72 of the
// 9-point form times 6 less 1/72 of the same at spacing 2.  N(di, dj) returns the neighbour
// at offset (di, dj); the operation order is the FP32 reference's.
template <int ST, class F>
__device__ __forceinline__ float resid_diff32(F N, float uC, float rk) {
    auto X = [&](int sp, int dy) {
        const float c = N(0, dy);
        return (N(sp, dy) - c) - (c - N(-sp, dy));
    };
    const float Y1 = (N(0, 1) - uC) - (uC - N(0, -1));
    const float X1c = (N(1, 0) - uC) - (uC - N(-1, 0));
    if (ST == 5) return (X1c + Y1) - rk;
    const float X1s = X(1, -1) + X(1, 1);
    if (ST == 9) return fmaf(1.0f / 6.0f, X1s, fmaf(2.0f / 3.0f, X1c, Y1 - rk));
    const float Y2 = (N(0, 2) - uC) - (uC - N(0, -2));
    const float X2c = (N(2, 0) - uC) - (uC - N(-2, 0));
    const float X2s = X(2, -2) + X(2, 2);
    return fmaf(2.0f / 9.0f, X1s,
                fmaf(8.0f / 9.0f, X1c,
                     fmaf(4.0f / 3.0f, Y1,
                          fmaf(-1.0f / 72.0f, X2s, fmaf(-1.0f / 18.0f, X2c, fmaf(-1.0f / 12.0f, Y2, -rk))))));
}


// (L u - b)(i, j) evaluated directly from a node accessor U(di, dj), in the same order as
// march (so the two agree bit for bit).
template <int ST, typename T, class F>
__device__ __forceinline__ T resid_direct(F U, T bk) {
    const T uC = U(0, 0);
    const T v1 = U(0, -1) + U(0, 1);
    const T p0 = U(-1, 0) + U(1, 0);
    if (ST == 5) return (p0 + v1) + Ar<T>::fm(Co<T>::c5(), uC, -bk);
    const T pm = U(-1, -1) + U(1, -1);
    const T pp = U(-1, 1) + U(1, 1);
    if (ST == 9)
        return Ar<T>::fm(Co<T>::ax9(), p0 + v1,
                         Ar<T>::fm(Co<T>::dg9(), pm + pp, Ar<T>::fm(Co<T>::cc9(), uC, -bk)));
    const T v2 = U(0, -2) + U(0, 2);
    const T P0 = U(-2, 0) + U(2, 0);
    const T Pm = U(-2, -2) + U(2, -2);
    const T Pp = U(-2, 2) + U(2, 2);
    return Ar<T>::fm(Co<T>::a1(), p0 + v1,
                     Ar<T>::fm(Co<T>::a2(), P0 + v2,
                               Ar<T>::fm(Co<T>::d1(), pm + pp,
                                         Ar<T>::fm(Co<T>::d2(), Pm + Pp, Ar<T>::fm(Co<T>::cc17(), uC, -bk)))));
}

// s + e = a + b exactly: Knuth's TwoSum takes six FP64 operations; ordered by exponent on the integer
// pipe, Dekker's FastTwoSum takes three and finds the same e.
__device__ __forceinline__ void two_sum(double a, double b, double &s, double &e) {
    const bool ordered =
        ((unsigned)__double2hiint(a) & 0x7fffffffu) >= ((unsigned)__double2hiint(b) & 0x7fffffffu);
    const double big = ordered ? a : b, small = ordered ? b : a;
    const double x = a + b;
    e = small - (x - big);
    s = x;
}

// The cascade S + E of TwoSums, adding c h for a power of two c = +-2^K.  Each TwoSum is ordered as
// in two_sum above; c h is not formed: c goes into the fused multiply-adds, where its product is
// exact.  (Terms below 2^-1018 may be ordered wrongly; what that can change is below 2^-1070.)
struct Sum2 {
    double S, E = 0.0;
    double one;  // 1, as an argument: additions as fused multiply-adds
    template <int K, bool NEG>
    static __device__ __forceinline__ double c() {
        return (NEG ? -1.0 : 1.0) * (double)(1 << K);
    }
    template <int K, bool NEG = false>
    __device__ __forceinline__ void first(double h) {
        S = fma(h, c<K, NEG>(), 0.0);
    }
    template <int K, bool NEG = false>
    __device__ __forceinline__ void add(double h) {
        const double cc = c<K, NEG>();
        const double s = fma(h, cc, S);
        const bool ordered = ((unsigned)__double2hiint(S) & 0x7fffffffu) >=
                             ((unsigned)__double2hiint(h) & 0x7fffffffu) + ((unsigned)K << 20);
        const double big = ordered ? S : h, small = ordered ? h : S;
        const double cb = ordered ? 1.0 : cc, cs = ordered ? cc : 1.0;
        const double z = fma(big, -cb, s);  // what of the smaller term s holds
        E = fma(fma(small, cs, -z), one, E);
        S = s;
    }
};

// x / D, correctly rounded, for D = 6 or 72: x / D by the rounded reciprocal, corrected once by its
// exact remainder (Markstein's theorem on division by fused multiply-adds); the division where the
// remainder could underflow or nothing is finite.
template <int D>
__device__ __forceinline__ double div_const(double x) {
    if (((unsigned)__double2hiint(x) >> 20 & 0x7ffu) - 128u > 1900u) return x / (double)D;
    constexpr double y = 1.0 / D;
    const double q = x * y;
    return fma(fma(-(double)D, q, x), y, q);
}

// FP64 L u at (i, j) of the padded grid u in resid_direct's order (b = 0), additions as fused
// multiply-adds.
template <int ST>
__device__ __forceinline__ double plain_L(const double *u, const Grid &g, int i, int j, double one) {
    using C = Co<double>;
    const double *p = u + g.idx(i, j);
    const long long P = g.pitch;
    auto U = [&](int di, int dj) { return p[dj * P + di]; };
    auto add = [&](double a, double b) { return fma(a, one, b); };
    const double uC = U(0, 0);
    const double s = add(add(U(-1, 0), U(1, 0)), add(U(0, -1), U(0, 1)));
    if (ST == 5) return add(s, fma(C::c5(), uC, -0.0));
    const double d = add(add(U(-1, -1), U(1, -1)), add(U(-1, 1), U(1, 1)));
    if (ST == 9) return fma(C::ax9(), s, fma(C::dg9(), d, fma(C::cc9(), uC, -0.0)));
    const double s2 = add(add(U(-2, 0), U(2, 0)), add(U(0, -2), U(0, 2)));
    const double d2 = add(add(U(-2, -2), U(2, -2)), add(U(-2, 2), U(2, 2)));
    return fma(C::a1(), s, fma(C::a2(), s2, fma(C::d1(), d, fma(C::d2(), d2, fma(C::cc17(), uC, -0.0)))));
}

// R = L (uh + ul) - bk at node (i, j), rounded to FP64 (term order as documented above).  one: 1.
template <int ST>
__device__ __forceinline__ double resid_dd(const double *uh, const double *ul, const Grid &g, int i, int j, double bk,
                                           double one) {
    const double *p = uh + g.idx(i, j);
    const long long P = g.pitch;
    auto H = [&](int di, int dj) { return p[dj * P + di]; };
    const double uC = H(0, 0);
    Sum2 s;
    s.one = one;
    constexpr int D = ST == 5 ? 1 : ST == 9 ? 6 : 72;
    if (ST == 5) {
        s.first<0>(H(-1, 0));
        s.add<0>(H(1, 0));
        s.add<0>(H(0, -1));
        s.add<0>(H(0, 1));
        s.add<2, true>(uC);
        s.add<0, true>(bk);
    } else if (ST == 9) {
        s.first<2>(H(-1, 0));
        s.add<2>(H(1, 0));
        s.add<2>(H(0, -1));
        s.add<2>(H(0, 1));
        s.add<0>(H(-1, -1));
        s.add<0>(H(1, -1));
        s.add<0>(H(-1, 1));
        s.add<0>(H(1, 1));
        s.add<4, true>(uC);
        s.add<2, true>(uC);
        s.add<2, true>(bk);
        s.add<1, true>(bk);
    } else {
        s.first<6>(H(-1, 0));
        s.add<6>(H(1, 0));
        s.add<6>(H(0, -1));
        s.add<6>(H(0, 1));
        s.add<2, true>(H(-2, 0));
        s.add<2, true>(H(2, 0));
        s.add<2, true>(H(0, -2));
        s.add<2, true>(H(0, 2));
        s.add<4>(H(-1, -1));
        s.add<4>(H(1, -1));
        s.add<4>(H(-1, 1));
        s.add<4>(H(1, 1));
        s.add<0, true>(H(-2, -2));
        s.add<0, true>(H(2, -2));
        s.add<0, true>(H(-2, 2));
        s.add<0, true>(H(2, 2));
        s.add<8, true>(uC);
        s.add<5, true>(uC);
        s.add<3, true>(uC);
        s.add<2, true>(uC);
        s.add<6, true>(bk);
        s.add<3, true>(bk);
    }
    const double Llo = plain_L<ST>(ul, g, i, j, one);
    const double t = fma(s.S, one, fma(s.E, one, (double)D * Llo));
    if constexpr (D == 1)
        return t;
    else
        return div_const<D>(t);
}

}  // namespace
