// NOHAP solve of one staged column (arXiv 2203.00879, Sec. 3).
//
// A column holds (at least) the solve window win_lo .. win_hi of one (line,
// field) pair in shared memory, row r at col[(r - org) * LP].  Given the sub-domain's
// two end values (the equivalent explicit rows g_i = sum_j C_ij f_j of
// Eq. CS:fpCf_i, evaluated by the caller) the solve
//   1. evaluates any explicit wall-closure row inside the sub-domain,
//   2. runs the Thomas forward sweep over the implicit rows (tabulated factors,
//      the end values moved to the right-hand side), keeping the last 2W+1
//      inputs in registers and writing the forward values in place,
//   3. back-substitutes in place,
// leaving the derivative (or filtered value) of rows s .. e in place, times
// osc: the factor is folded into the right-hand-side weights, the end values and
// the explicit rows, and past the tabulated factors the reciprocal pivot into the
// weights as well, so that a row costs six multiplications and additions instead
// of eight (FP64 runs at 1/64 of the FP32 rate: its count decides the time).
#pragma once

#include "nopcs_internal.cuh"

namespace nopcs {

template <typename T>
__device__ __forceinline__ const T *coef_ptr(const LineOpDev &op);
template <>
__device__ __forceinline__ const double *coef_ptr<double>(const LineOpDev &op) { return op.coef64; }
template <>
__device__ __forceinline__ const float *coef_ptr<float>(const LineOpDev &op) { return op.coef32; }
template <typename T>
__device__ __forceinline__ const T *cp_ptr(const LineOpDev &op);
template <>
__device__ __forceinline__ const double *cp_ptr<double>(const LineOpDev &op) { return op.cp64; }
template <>
__device__ __forceinline__ const float *cp_ptr<float>(const LineOpDev &op) { return op.cp32; }
template <typename T>
__device__ __forceinline__ const T *inv_ptr(const LineOpDev &op);
template <>
__device__ __forceinline__ const double *inv_ptr<double>(const LineOpDev &op) { return op.inv64; }
template <>
__device__ __forceinline__ const float *inv_ptr<float>(const LineOpDev &op) { return op.inv32; }

// dot product of `len` taps with a column (stride LP), four partial sums
template <typename T>
__device__ __forceinline__ T dot_col(const T *c, const T *f, int len, int LP)
{
    T s0 = 0, s1 = 0, s2 = 0, s3 = 0;
    int k = 0;
    for (; k + 4 <= len; k += 4) {
        s0 += c[k] * f[(size_t)k * LP];
        s1 += c[k + 1] * f[(size_t)(k + 1) * LP];
        s2 += c[k + 2] * f[(size_t)(k + 2) * LP];
        s3 += c[k + 3] * f[(size_t)(k + 3) * LP];
    }
    for (; k < len; ++k) s0 += c[k] * f[(size_t)k * LP];
    return (s0 + s1) + (s2 + s3);
}

// org: the row at col[0]; gs / ge: the end values at rows s and e (ge unused
// when e == s); tcp / tiv: the first KC Thomas factors (the rest equal their
// limits cpL / invL); w: the right-hand-side weights times osc, and these times
// invL.  A single field takes them from there, kernel parameters, so that they
// need no registers: scaled in the kernel they cost it an eighth of its warps
// (400 x 9 x 400 along y 40.8 us, 35.1 now; 24 x 300 x 200 along x, order 3, 41.3
// and 35.1).  Sweeps of several fields scale them in the kernel: for these the
// parameters are slower (128^3 filter 980 against 954 us).
template <typename T, int MODE>
__device__ __forceinline__ void nohap_solve_column(const LineOpDev &op, const T (&w)[2][4], T *col, int LP, int org,
                                                   T gs, T ge, const T *tcp, const T *tiv, int KC, const int *rec,
                                                   T osc)
{
    constexpr int W = MODE == MODE_FILTER ? 3 : 2;     // right-hand-side half-width
    constexpr int NEXP = MODE == MODE_FILTER ? 3 : 2;  // explicit rows at each wall
    const int s = rec[0], e = rec[1], tlo = org;
    const int lene = rec[8];
    const int lo = rec[10], hi = rec[11];
    const int N = op.N;
    gs *= osc;
    ge *= osc;
    // explicit wall-closure rows strictly inside the sub-domain
    T exL[NEXP], exH[NEXP];
#pragma unroll
    for (int r = 0; r < NEXP; ++r) {
        exL[r] = 0;
        exH[r] = 0;
        if (r > s && r < e) {
            T acc = 0;
#pragma unroll
            for (int j = 0; j < 5; ++j)
                if (op.ex[r][j] != 0.0) acc += (T)op.ex[r][j] * col[(size_t)(j - tlo) * LP];
            exL[r] = osc * acc;
        }
        const int rh = N - 1 - r;
        if (rh > s && rh < e) {
            T acc = 0;
#pragma unroll
            for (int j = 0; j < 5; ++j)
                if (op.ex[r][j] != 0.0) acc += (T)op.ex[r][j] * col[(size_t)(N - 1 - j - tlo) * LP];
            exH[r] = osc * ((T)op.ex_sign * acc);
        }
    }
    // 2./3. Thomas over the implicit rows lo..hi; forward values overwrite
    // the staged inputs, which a register window of 2W+1 keeps
    if (lo <= hi) {
        const int m = hi - lo + 1;
        const T al = (T)op.alpha;
        const T gL = lo == s + 1 ? gs : exL[NEXP - 1];
        const T gR = hi == e - 1 ? ge : exH[NEXP - 1];
        constexpr bool SINGLE = MODE == MODE_FIELD || MODE == MODE_FIELD2;
        T b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) b[k] = SINGLE ? w[0][k] : osc * (T)op.rb[k];
        const T cL = (T)op.cpL, iL = (T)op.invL;
        T win[2 * W + 1];
        const T *pin = col + (size_t)(lo - W - tlo) * LP;
#pragma unroll
        for (int j = 0; j < 2 * W; ++j) win[j] = pin[(size_t)j * LP];
        pin += (size_t)(2 * W) * LP;                // row lo + W
        T *pout = col + (size_t)(lo - tlo) * LP;   // row lo
        T dprev = 0;
        // one forward row: right-hand side from the window, minus the
        // coupling `adj` to a known end value, then the elimination
        auto right = [&](const T(&b)[4]) {
            win[2 * W] = *pin;
            pin += LP;
            T rhs;
            if constexpr (MODE == MODE_FILTER)
                rhs = b[0] * win[3] + b[1] * (win[4] + win[2]) + b[2] * (win[5] + win[1]) + b[3] * (win[6] + win[0]);
            else if constexpr (MODE == MODE_FIELD2)
                rhs = b[0] * win[2] + b[1] * (win[3] + win[1]) + b[2] * (win[4] + win[0]);
            else
                rhs = b[0] * (win[3] - win[1]) + b[1] * (win[4] - win[0]);
#pragma unroll
            for (int j = 0; j < 2 * W; ++j) win[j] = win[j + 1];
            return rhs;
        };
        auto fwd = [&](T iv, T adj) {
            const T dp = (right(b) - adj - al * dprev) * iv;
            *pout = dp;
            pout += LP;
            dprev = dp;
        };
        // first row carries the left end value (and the right one if m == 1)
        fwd(tiv[0], al * gL + (m == 1 ? al * gR : T(0)));
        const int kmid = min(KC, m - 1);
        int r = 1;
#pragma unroll 4
        for (; r < kmid; ++r) fwd(tiv[r], T(0));
        if (r < m - 1) {
            T c[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) c[k] = SINGLE ? w[1][k] : b[k] * iL;
#pragma unroll 4
            for (; r < m - 1; ++r) {
                dprev = right(c) - cL * dprev;
                *pout = dprev;
                pout += LP;
            }
        }
        if (m > 1) fwd(m - 1 < KC ? tiv[m - 1] : iL, al * gR);
        // back substitution from row hi - 1 down to lo
        T x = dprev;
        pout -= 2 * (size_t)LP;  // row hi - 1
        r = m - 2;
#pragma unroll 4
        for (; r >= KC; --r) {
            x = *pout - cL * x;
            *pout = x;
            pout -= LP;
        }
#pragma unroll 4
        for (; r >= 0; --r) {
            x = *pout - tcp[r] * x;
            *pout = x;
            pout -= LP;
        }
    }
    // explicit values into their rows
    col[(size_t)(s - tlo) * LP] = gs;
    if (lene > 0) col[(size_t)(e - tlo) * LP] = ge;
#pragma unroll
    for (int r = 0; r < NEXP; ++r) {
        if (r > s && r < e) col[(size_t)(r - tlo) * LP] = exL[r];
        const int rh = N - 1 - r;
        if (rh > s && rh < e) col[(size_t)(rh - tlo) * LP] = exH[r];
    }
}

}  // namespace nopcs
