// Factorisation of 16 x 16 blocks and their products by one warp, in float64: what the factorisations of
// larger blocks in shared memory (the leaf of the inverse, a head's block) are made of.
#pragma once

#include <math.h>

#include "common.cuh"

namespace ziplm {

// One warp: acc(16 x 16) += A(16 x 16) B(16 x 16), operands in shared memory;
// BT: B(k,n) = b[n][k], else b[k][n].
template <bool BT>
__device__ __forceinline__ void warp_mma16(double (&acc)[2][2][2], const double* a, int lda, const double* b, int ldb) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
        double fa[2], fb[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            fa[i] = a[(8 * i + (lane >> 2)) * lda + 4 * kk + (lane & 3)];
            fb[i] = BT ? b[(8 * i + (lane >> 2)) * ldb + 4 * kk + (lane & 3)]
                       : b[(4 * kk + (lane & 3)) * ldb + 8 * i + (lane >> 2)];
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j) dmma884(acc[i][j], fa[i], fb[j]);
    }
}

// One warp: c(16 x 16) = acc, or c -= acc.
template <bool SUB>
__device__ __forceinline__ void warp_put16(const double (&acc)[2][2][2], double* c, int ldc) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            double2* o = reinterpret_cast<double2*>(c + (8 * i + (lane >> 2)) * ldc + 8 * j + 2 * (lane & 3));
            double2 v = make_double2(acc[i][j][0], acc[i][j][1]);
            if (SUB) { const double2 x = *o; v.x = x.x - v.x; v.y = x.y - v.y; }
            *o = v;
        }
}

// 1 / x = y0 (1 + e + e^2 + ...), e = 1 - x y0, from the hardware's approximation y0 (relative error
// below 2^-20, so the terms left out are below 2^-60): y0 and e + e^2.
__device__ __forceinline__ void reciprocal_terms(double x, double& y0, double& s) {
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
    const double e = fma(-x, y0, 1.0);
    s = fma(e, e, e);
}

// One warp: the inverse of the Cholesky factor of an 8 x 8 block (full symmetric), in the lanes as the
// float64 mma's result: lane 4 i + c holds columns 2 c and 2 c + 1 of row i; lower, zero above.
// Elimination of [A | I] in place: at column k the rows i > k become
//     r_ij -= (r_ik / r_kk) r_kj   for all j != k,      r_ik = -r_ik / r_kk,
// which leaves the Schur complement in the columns j > k and row i of L^-1 (A = L D L^T) in the columns
// j < i; the result is D^-1/2 L^-1.  Returns the row's pivot.
// The chain is that of the pivots, p_{k+1} = a_{k+1,k+1} - a_{k+1,k}^2 / p_k: every lane runs it on its
// own, from the two entries as they were before column k, so that a column costs it a reciprocal and four
// FMAs and the shuffles of the rows run beside it.
__device__ __forceinline__ double warp_factor8(double (&r)[2]) {
    const int lane = threadIdx.x & 31, i = lane >> 2, c = lane & 3;
    double p = __shfl_sync(0xffffffffu, r[0], 0), piv = p;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        double y0, s;
        const double rik = __shfl_sync(0xffffffffu, r[k & 1], (lane & 28) + (k >> 1));
        reciprocal_terms(p, y0, s);
        double next = 1.0;
        if (k < 7) {
            const int n = k + 1;
            const double off = __shfl_sync(0xffffffffu, r[k & 1], 4 * n + (k >> 1));
            const double dia = __shfl_sync(0xffffffffu, r[n & 1], 4 * n + (n >> 1));
            const double t = off * y0;
            next = fma(-fma(t, s, t), off, dia);
        }
        const double t = i > k ? rik * y0 : 0.0;
        const double f = fma(t, s, t);
        const double rk0 = __shfl_sync(0xffffffffu, r[0], 4 * k + c);
        const double rk1 = __shfl_sync(0xffffffffu, r[1], 4 * k + c);
        r[0] = fma(-f, rk0, r[0]);
        r[1] = fma(-f, rk1, r[1]);
        if (c == (k >> 1) && i > k) r[k & 1] = -f;
        p = next;
        if (i == k + 1) piv = next;
    }
    const double sc = rsqrt(piv);
#pragma unroll
    for (int e = 0; e < 2; ++e) r[e] = 2 * c + e < i ? r[e] * sc : 2 * c + e == i ? sc : 0.0;
    return piv;
}

// One warp: d += x y^T of 8 x 8 blocks held as above.  The k order of the two mma steps is free, so
// columns 2 c go into the first and columns 2 c + 1 into the second, and no operand changes lanes.
__device__ __forceinline__ void warp_mma8(double (&d)[2], const double (&x)[2], const double (&y)[2]) {
    dmma884(d, x[0], y[0]);
    dmma884(d, x[1], y[1]);
}

// One warp: the inverse of the Cholesky factor of the 16 x 16 block at a (its lower triangle; the diagonal
// 8 x 8 blocks in full; pitch lda) -> out (lower, pitch PB; zero above).  Two 8 x 8 eliminations and seven
// 8 x 8 products in registers: the shuffles of a column are 5 instead of the 11 of a 16 x 16 elimination,
// whose columns took 308 clocks.
constexpr int PB = 20;
__device__ __forceinline__ int warp_factor16(const double* a, int lda, double* out) {
    const int lane = threadIdx.x & 31, i = lane >> 2, c = lane & 3;
    auto load = [&](double (&r)[2], int bi, int bj) {
        const double2 v = *reinterpret_cast<const double2*>(a + (8 * bi + i) * lda + 8 * bj + 2 * c);
        r[0] = v.x;
        r[1] = v.y;
    };
    auto store = [&](const double (&r)[2], int bi, int bj) {
        *reinterpret_cast<double2*>(out + (8 * bi + i) * PB + 8 * bj + 2 * c) = make_double2(r[0], r[1]);
    };
    double m1[2], a21[2], m2[2];
    load(m1, 0, 0);
    load(a21, 1, 0);
    load(m2, 1, 1);
    const double p1 = warp_factor8(m1);
    double l21[2] = {0.0, 0.0}, t[2] = {0.0, 0.0};
    warp_mma8(l21, a21, m1);                                 // L21 = A21 M11^T
    warp_mma8(t, l21, l21);                                  // A22 - L21 L21^T
    m2[0] -= t[0];
    m2[1] -= t[1];
    double m1t[2], x[2] = {0.0, 0.0}, m21[2] = {0.0, 0.0};
#pragma unroll
    for (int e = 0; e < 2; ++e) {                            // M11^T
        const double u = __shfl_sync(0xffffffffu, m1[0], 4 * (2 * c + e) + (i >> 1));
        const double v = __shfl_sync(0xffffffffu, m1[1], 4 * (2 * c + e) + (i >> 1));
        m1t[e] = i & 1 ? v : u;
    }
    warp_mma8(x, m1t, l21);                                  // (L21 M11)^T
    const double p2 = warp_factor8(m2);
    warp_mma8(m21, m2, x);                                   // M21 = -M22 (L21 M11)
    m21[0] = -m21[0];
    m21[1] = -m21[1];
    const double zero[2] = {0.0, 0.0};
    store(m1, 0, 0);
    store(zero, 0, 1);
    store(m21, 1, 0);
    store(m2, 1, 1);
    const unsigned bad1 = __ballot_sync(0xffffffffu, !(p1 > 0.0) || !isfinite(p1));
    const unsigned bad2 = __ballot_sync(0xffffffffu, !(p2 > 0.0) || !isfinite(p2));
    if (!(bad1 | bad2)) return 0;                            // the first bad pivot: not positive definite, or NaN
    const double bad = __shfl_sync(0xffffffffu, bad1 ? p1 : p2, __ffs(bad1 ? bad1 : bad2) - 1);
    return isfinite(bad) ? ZIPLM_ERR_NOT_PD : ZIPLM_ERR_NONFINITE;
}

}  // namespace ziplm
