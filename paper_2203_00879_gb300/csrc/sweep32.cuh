// FP32 line sweeps without block-wide phases (arXiv 2203.00879, Sec. 3).
//
// Far from its ends a line's compact system (alpha, 1, alpha) g = B f factors
// into two first-order recurrences with constant coefficients,
//   d_i = t_i - c d_{i-1},   x_i = d_i - c x_{i+1},
// t the normalised right-hand side and c the limit of the Thomas factors
// (|c| = 0.46 for OUCS3, less for the filter and the second derivative).
// What lies k points away enters with weight c^k: 24 points give the 1e-8 at
// which the FP32 end rows of C = A^-1 B (Eqs. CS:fpCf, CS:fpCf_i) are cut as
// well.  So a piece of a line that starts its forward recurrence 24 rows
// early and its backward recurrence 24 rows late needs no end rows, and
// equals the NOHAP solve of any partition to FP32 rounding, as NOHAP solves of
// different partitions equal one another.  Next to a wall the recurrences
// start from the explicit closure rows with the tabulated factors and are
// those of the Thomas algorithm.
//
// Lines are independent, also where they hold infinities or NaN: whatever a
// kernel takes from a neighbouring thread or lane of another line is left out by
// selection, never by a factor of zero.  Within its line such a value reaches
// as far as the recurrence carries it: in a march the rest of its segment (a
// whole line where lines are not cut) and the 24 rows around, along x the three
// chunks of 8 on either side; explicit rows next to a wall only through their
// closure.
//
// Two kernels use this:
//   march_body (lines along y, z): a thread walks one line; consecutive
//     threads take consecutive lines, so loads and stores coalesce, and no
//     thread talks to another: no barrier anywhere.  Bound by HBM: at
//     1024 x 512 x 512 the y and z flux sweeps take 2.49 and 2.52 ms (60 B a
//     point, 0.95 and 0.94 of the measured copy bandwidth); the sub-domain
//     tiles with end rows and barriers took 3.56 and 3.62, held up by their
//     alternating load, solve and store phases.
//   scan_body (lines along x): a lane solves 8 consecutive points and takes
//     the recurrences' state from its three neighbour lanes by shuffles.
//     2.00 ms (40 B a point, 0.79 of the copy bandwidth; two thirds of the
//     issue slots and three quarters of the shared-memory cycles used) against
//     3.71 for whole lines in block-wide phases.
// One field at 512^3 (8 B a point), x, y, z: 239, 240, 243 us against 469, 546,
// 534 for the sub-domain tiles; compact viscous terms at 256^3, mean of the
// axes: gradients 0.148 ms against 0.207, divergence 0.165 against 0.193.
#pragma once

#include "nopcs_internal.cuh"

namespace nopcs {

// Rows after which the recurrences have forgotten their start (c^reach < 1e-8):
// 24 for the first derivative (c = 0.46), 16 for the second derivative (0.19)
// and the filter (0.14 at the paper's coefficient).
constexpr int sweep_reach(int mode) { return mode == MODE_FILTER || mode == MODE_FIELD2 ? 16 : 24; }
constexpr int SC_SHORT = 32;  // scan: lines shorter than this feel both walls
constexpr int SC_P = 8;       // scan: points of a lane
constexpr int SW_TAB = 20;    // rows tabulated next to a wall (the factors converge like c^(2r))

struct Sweep32Args {
    int n[3];
    int N;                 // points of a line
    int cols, seg, nseg;   // march: lines, rows per segment, segments per line
    int ring;              // march: groups of a thread's ring (4 or 8)
    const int *sub;        // march of a single field: sub-domain records (LineOpDev)
    int srow, sc;          // march: strides of a row and of the second line index
    int nch, tot;          // scan: 8-point chunks per line, chunks in all
    int kind;              // scan: 0 short lines, 1 single points, 2 four points a lane at a time
    int ga;                // gravity axis
    const float *in[5];
    float *out[5];
    const float *b0, *b1, *b2;  // base tables along gravity, as LineArgs
    float hp;              // gamma / (gamma - 1)
    float b[4];            // right-hand-side weights, normalised and scaled
    float c, g1;           // limit factor, 1 / (1 + c)
    float pw[SC_P], pw16;  // scan: (-c)^1 .. (-c)^8 and (-c)^16
    float kf[4];           // scan: low-wall correction of chunks 0 .. 3, c (-c)^(8 ch - NEXP)
    // by row from the low wall, the last entry for all rows beyond: the factor
    // (0 in explicit rows) and 1/pivot over its limit
    float cp[SW_TAB], rat[SW_TAB];
    float ex[3][5];        // explicit closure rows (scaled), taps from the wall inwards
    float exs;             // sign of the high wall's mirrored rows
};

template <int MODE>
struct SweepMode {
    static constexpr bool SINGLE = MODE == MODE_FIELD || MODE == MODE_FIELD2;
    static constexpr int NF = SINGLE ? 1 : (MODE == MODE_VGRAD || MODE == MODE_VDIV ? 4 : 5);
    static constexpr int NIN = SINGLE ? 1 : (MODE == MODE_VDIV ? 4 : 5);
    static constexpr int REACH = sweep_reach(MODE);
    static constexpr int HW = MODE == MODE_FILTER ? 3 : 2;    // right-hand-side half-width
    static constexpr int NEXP = MODE == MODE_FILTER ? 3 : 2;  // explicit rows at a wall
    static constexpr int NB = MODE == MODE_FLUX ? 2 : (MODE == MODE_VGRAD ? 3 : 0);  // base tables used
};
// explicit row r next to a wall has a tap at distance j from it
template <int MODE>
__host__ __device__ constexpr bool sweep_tap(int r, int j)
{
    return MODE == MODE_FILTER ? j == r : (MODE == MODE_FIELD2 ? j < (r ? 3 : 4) : (r ? true : j < 3));
}
// the sweeps that add to their output (the others store)
__host__ __device__ constexpr bool sweep_adds(int mode, int axis)
{
    return mode == MODE_VDIV || (mode == MODE_FLUX && axis != 0);
}

// The line quantities of one point from its inputs v and base values bb: the
// inviscid flux along AXIS (Eqs. ge3-ge5), u, v, w, T, or the inputs
// themselves.  The enthalpy H = H_b + gamma / (gamma - 1) p' + rho |V|^2 / 2 is
// formed here from the primitives: stored, it was a sixth field for the three
// sweeps to read and the stage kernel to write (1024 x 512 x 512: x, y, z 2.09,
// 2.63, 2.71 ms, stage 6.98; now 1.99, 2.49, 2.52 and 6.89), and its rounding
// is lost against that of H_b, which is thousands of times larger.  Fixed-order
// arithmetic: the same bits in every kernel.
template <int MODE, int AXIS>
__device__ __forceinline__ void sweep_point(const float *v, const float *bb, const float hp, float *f)
{
    if constexpr (MODE == MODE_FLUX) {
        const float rho = __fadd_rn(bb[0], v[0]);
        const float q = __fmaf_rn(v[3], v[3], __fmaf_rn(v[2], v[2], __fmul_rn(v[1], v[1])));
        const float H = __fadd_rn(bb[1], __fmaf_rn(hp, v[4], __fmul_rn(__fmul_rn(0.5f, rho), q)));
        const float ud = v[1 + AXIS], m = __fmul_rn(rho, ud);
        f[0] = m;
#pragma unroll
        for (int k = 0; k < 3; ++k) f[1 + k] = k == AXIS ? __fmaf_rn(m, v[1 + k], v[4]) : __fmul_rn(m, v[1 + k]);
        f[4] = __fmul_rn(H, ud);
    } else if constexpr (MODE == MODE_VGRAD) {
        f[0] = v[1];
        f[1] = v[2];
        f[2] = v[3];
        // T_b (1 + p'/p_b) / (1 + rho'/rho_b) on the deviations
        const float rr = __fmul_rn(v[0], bb[2]);
        f[3] = __fadd_rn(bb[0], __fdividef(__fmul_rn(bb[0], __fmaf_rn(v[4], bb[1], -rr)), __fadd_rn(1.0f, rr)));
    } else {
#pragma unroll
        for (int k = 0; k < SweepMode<MODE>::NF; ++k) f[k] = v[k];
    }
}

// normalised right-hand side of row i from w[0 .. 2 HW] = f_{i-HW} .. f_{i+HW}
template <int MODE>
__device__ __forceinline__ float sweep_rhs(const Sweep32Args &a, const float *w, int st)
{
    if constexpr (MODE == MODE_FILTER) {
        float t = __fmul_rn(a.b[0], w[3 * st]);
        t = __fmaf_rn(a.b[1], __fadd_rn(w[4 * st], w[2 * st]), t);
        t = __fmaf_rn(a.b[2], __fadd_rn(w[5 * st], w[st]), t);
        return __fmaf_rn(a.b[3], __fadd_rn(w[6 * st], w[0]), t);
    } else if constexpr (MODE == MODE_FIELD2) {
        // second differences: b0 = -2 (b1 + b2)
        const float e1 = __fadd_rn(__fadd_rn(w[3 * st], -w[2 * st]), -__fadd_rn(w[2 * st], -w[st]));
        const float e2 = __fadd_rn(__fadd_rn(w[4 * st], -w[2 * st]), -__fadd_rn(w[2 * st], -w[0]));
        return __fmaf_rn(a.b[1], e1, __fmul_rn(a.b[2], e2));
    } else {
        return __fmaf_rn(a.b[1], __fadd_rn(w[4 * st], -w[0]), __fmul_rn(a.b[0], __fadd_rn(w[3 * st], -w[st])));
    }
}

constexpr int SCAN_WARPS = 4;  // warps per block of a stand-alone scan

// Host: the operator's coefficients with `scale` folded in (false if its
// recurrences remember more than `reach` rows at 1e-8: a filter coefficient
// near 1/2), then the lines and pieces for a field of n points; a.N is set.
bool sweep32_operator(const LineOpDev &op, int reach, double scale, Sweep32Args &a);
void sweep32_geometry(int axis, const int n[3], Sweep32Args &a);
// the convective sweep of a box along `axis`: R (= or -=) L(flux(W)) / h
bool flux32_args(const LineOpDev &op, int axis, const BoxDev &bx, const float *W, float *R, Sweep32Args &a);
template <int MODE>
cudaError_t launch_sweep32(int axis, const Sweep32Args &a, cudaStream_t st);

// ---- lines along y and z ------------------------------------------------------
// A thread's forward values wait in shared memory until the backward
// recurrence has come far enough: a ring of R groups of 8 rows, private to the
// thread.  When it is full, at group n, the backward recurrence starts at the
// last row, runs back through groups n, n-1, n-2 (24 rows) and gives the final
// values of the groups before them.  The inputs of the next group are in
// flight meanwhile.  (Where the reach is 16 rows, two groups of start-up do.)
//
// A sweep of a box cuts its lines where that fills the GPU.  A single field's
// derivative cuts them at the sub-domains and reads nothing outside the rows
// [tlo, thi] that a sub-domain's end rows reach (a row beyond repeats the last
// one, 24 rows from any result): then a slab that holds these rows only gets
// the bits of the whole line.
constexpr int MR_G = 8;

// shared memory of a march block
constexpr size_t march_smem(int nf, int R, int threads) { return (size_t)R * MR_G * nf * threads * sizeof(float); }

// One block of a march: TPB lines of one segment.  tid: 0 .. TPB - 1; U (a
// divisor of 8): rows whose inputs are in flight; FAST: code of its own for the
// rows of constant coefficients.  Neither changes a result.
template <int MODE, int AXIS, bool GROW, int R, int TPB, int U = MR_G, bool FAST = true>
__device__ __forceinline__ void march_body(const Sweep32Args &a, const unsigned vblock, const int tid, float *sm)
{
    using M = SweepMode<MODE>;
    constexpr int NF = M::NF, NIN = M::NIN, HW = M::HW, NEXP = M::NEXP, NB = M::NB;
    constexpr int NV = NF >= 4 ? 4 : 0;  // fields kept as one 16-byte vector per row
    constexpr bool ADD = sweep_adds(MODE, AXIS);
    float4 *const ring4 = reinterpret_cast<float4 *>(sm) + tid;
    float *const ring1 = sm + (size_t)NV * R * MR_G * TPB + tid;
    const int q = (int)(vblock / (unsigned)a.nseg) * TPB + tid;
    if (q >= a.cols) return;
    const int x = q % a.n[0], cc = q / a.n[0];
    const int base = x + cc * a.sc;
    const int N = a.N, srow = a.srow;
    constexpr int LAG = M::REACH / MR_G;
    const int seg = (int)(vblock % (unsigned)a.nseg);
    const int hrow = N - 1 - NEXP;  // last implicit row
    int s, e, tlo = 0, thi = N - 1;
    bool low, high;
    if constexpr (M::SINGLE) {
        const int *rec = a.sub + seg * SUB_REC;
        s = rec[0], e = rec[1] + 1, tlo = rec[2], thi = rec[3];
        low = rec[14] != 0, high = rec[15] != 0;
    } else {
        s = seg * a.seg, e = min(N, s + a.seg);
        low = s == 0, high = e - 1 + M::REACH >= hrow;
    }
    const int r0 = low ? 0 : s - M::REACH;
    const int G = ((high ? hrow : e - 1 + M::REACH) - r0) / MR_G + 1;
    int next = (s - r0) / MR_G;  // next group to give results

    const int kc = a.ga == 0 ? x : cc;  // coordinate along gravity (gravity not along the sweep)
    float bc[3];
    if constexpr (NB > 0 && !GROW) {
        bc[0] = a.b0[kc];
        bc[1] = a.b1[kc];
        if constexpr (NB > 2) bc[2] = a.b2[kc];
    }
    auto load = [&](float *v, int row) {
        const int p = base + row * srow;
#pragma unroll
        for (int k = 0; k < NIN; ++k) v[k] = a.in[k][p];
    };
    auto convert = [&](const float *v, int row, float *f) {
        if constexpr (NB > 0 && GROW) {
            float bb[3] = {a.b0[row], a.b1[row], 0.0f};
            if constexpr (NB > 2) bb[2] = a.b2[row];
            sweep_point<MODE, AXIS>(v, bb, a.hp, f);
        } else {
            sweep_point<MODE, AXIS>(v, bc, a.hp, f);
        }
    };
    auto put = [&](int slot, const float *d) {
        if constexpr (NV == 4) ring4[slot * TPB] = make_float4(d[0], d[1], d[2], d[3]);
        if constexpr (NF > NV) ring1[slot * TPB] = d[NF - 1];
    };
    auto get = [&](int slot, float *d) {
        if constexpr (NV == 4) {
            const float4 t = ring4[slot * TPB];
            d[0] = t.x;
            d[1] = t.y;
            d[2] = t.z;
            d[3] = t.w;
        }
        if constexpr (NF > NV) d[NF - 1] = ring1[slot * TPB];
    };
    auto emit = [&](int row, const float *xv) {
        if (M::SINGLE && (row < s || row >= e)) return;
        const int p = base + row * srow;
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            // adding sweeps use a reduction performed in L2: every element
            // takes one addition per sweep, rounded as load + add + store
            if constexpr (ADD)
                atomicAdd(&a.out[k][p], xv[k]);
            else
                a.out[k][p] = xv[k];
        }
    };

    // F[u .. u + 2 HW]: the window of row i0 + U h + u in step h of a group
    float F[2 * HW + U][NF], v[U][NIN], dp[NF];
#pragma unroll
    for (int u = 0; u < 2 * HW; ++u) {
        const int row = min(max(r0 - HW + u, tlo), thi);
        float t[NIN];
        load(t, row);
        convert(t, row, F[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) load(v[u], min(max(r0 + HW + u, tlo), thi));
#pragma unroll
    for (int k = 0; k < NF; ++k) dp[k] = 0.0f;
#pragma unroll 1
    for (int n = 0; n < G; ++n) {
        const int i0 = r0 + MR_G * n;
        const int s0 = (n & (R - 1)) * MR_G;
        // ---- forward, U rows at a time, the next U rows' inputs in flight ----
#pragma unroll
        for (int h = 0; h < MR_G / U; ++h) {
            const int ih = i0 + U * h, nx = ih + U + HW;  // nx: next step's first input row
#pragma unroll
            for (int u = 0; u < U; ++u) convert(v[u], min(ih + HW + u, thi), F[2 * HW + u]);
            if (nx + U <= thi + 1 && (!M::SINGLE || nx >= tlo)) {
#pragma unroll
                for (int u = 0; u < U; ++u) load(v[u], nx + u);
            } else if (h + 1 < MR_G / U || n + 1 < G) {
#pragma unroll
                for (int u = 0; u < U; ++u) load(v[u], min(max(nx + u, tlo), thi));
            }
            if (FAST && (!low || i0 >= SW_TAB)) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
#pragma unroll
                    for (int k = 0; k < NF; ++k) dp[k] = __fmaf_rn(-a.c, dp[k], sweep_rhs<MODE>(a, &F[u][k], NF));
                    put(s0 + U * h + u, dp);
                }
            } else {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (U * h + u == NEXP && low && n == 0) {
                        // explicit rows of the low wall; the window holds rows 0 .. 2 HW
#pragma unroll
                        for (int r = 0; r < NEXP; ++r) {
#pragma unroll
                            for (int k = 0; k < NF; ++k) {
                                float t = 0.0f;
#pragma unroll
                                for (int j = 0; j < 5; ++j)
                                    if (sweep_tap<MODE>(r, j)) t = __fmaf_rn(a.ex[r][j], F[u + j][k], t);
                                dp[k] = t;
                            }
                            put(r, dp);
                        }
                    }
                    const int row = low ? min(ih + u, SW_TAB - 1) : SW_TAB - 1;
                    const float cp = a.cp[row], rt = a.rat[row];
#pragma unroll
                    for (int k = 0; k < NF; ++k)
                        dp[k] = __fmaf_rn(-cp, dp[k], __fmul_rn(rt, sweep_rhs<MODE>(a, &F[u][k], NF)));
                    if (!(U * h + u < NEXP && low && n == 0)) put(s0 + U * h + u, dp);
                }
            }
#pragma unroll
            for (int u = 0; u < 2 * HW; ++u)
#pragma unroll
                for (int k = 0; k < NF; ++k) F[u][k] = F[U + u][k];
        }
        // ---- backward, once R groups wait or the line ends ----
        const bool last = high && n == G - 1;
        if (n - next + 1 < R && n + 1 < G) continue;
        if (n - LAG < next && !last) continue;
        float X[NF];
        int emax = i0 - (LAG - 1) * MR_G;  // results: rows below emax
        if (last) {
            // explicit rows of the high wall, the last of which starts the
            // recurrence
            emax = min(e, hrow + 1);
            float f[5][NF];
#pragma unroll
            for (int j = 0; j < 5; ++j) {
                float t[NIN];
                load(t, N - 1 - j);
                convert(t, N - 1 - j, f[j]);
            }
#pragma unroll
            for (int r = 0; r < NEXP; ++r) {
#pragma unroll
                for (int k = 0; k < NF; ++k) {
                    float t = 0.0f;
#pragma unroll
                    for (int j = 0; j < 5; ++j)
                        if (sweep_tap<MODE>(r, j)) t = __fmaf_rn(a.ex[r][j], f[j][k], t);
                    X[k] = __fmul_rn(a.exs, t);
                }
                if (N - 1 - r >= s && N - 1 - r < e) emit(N - 1 - r, X);
            }
            if (hrow < i0 + MR_G - 1) {  // it sits in the group, with nothing after it
                put(s0 + hrow + 1 - i0, X);
#pragma unroll
                for (int k = 0; k < NF; ++k) X[k] = 0.0f;
#pragma unroll 1
                for (int i = hrow + 2; i < i0 + MR_G; ++i) put(s0 + i - i0, X);
            }
        } else {
            // as if the line went on unchanged
            get(s0 + MR_G - 1, X);
#pragma unroll
            for (int k = 0; k < NF; ++k) X[k] = __fmul_rn(X[k], a.g1);
        }
        if (FAST && !last && (!low || next * MR_G >= SW_TAB)) {
#pragma unroll 1
            for (int m = n; m > n - LAG; --m) {
#pragma unroll
                for (int u = MR_G - 1; u >= 0; --u) {
                    float d[NF];
                    get((m & (R - 1)) * MR_G + u, d);
#pragma unroll
                    for (int k = 0; k < NF; ++k) X[k] = __fmaf_rn(-a.c, X[k], d[k]);
                }
            }
#pragma unroll 1
            for (int m = n - LAG; m >= next; --m) {
#pragma unroll
                for (int u = MR_G - 1; u >= 0; --u) {
                    float d[NF];
                    get((m & (R - 1)) * MR_G + u, d);
#pragma unroll
                    for (int k = 0; k < NF; ++k) X[k] = __fmaf_rn(-a.c, X[k], d[k]);
                    emit(r0 + MR_G * m + u, X);
                }
            }
        } else {
#pragma unroll 1
            for (int m = n; m >= next; --m) {
                const int sb = (m & (R - 1)) * MR_G, ib = r0 + MR_G * m;
                const bool out = ib < emax, wall = low && m == 0;
#pragma unroll
                for (int u = MR_G - 1; u >= 0; --u) {
                    float d[NF];
                    get(sb + u, d);
                    const float cp = a.cp[low ? min(ib + u, SW_TAB - 1) : SW_TAB - 1];
                    // an explicit row (factor 0) has its own value whatever the
                    // rows above it hold
#pragma unroll
                    for (int k = 0; k < NF; ++k)
                        X[k] = u < NEXP && wall ? d[k] : __fmaf_rn(-cp, X[k], d[k]);
                    if (out && ib + u < emax) emit(ib + u, X);
                }
            }
        }
        next = n - LAG + 1;
    }
}

// ---- lines along x --------------------------------------------------------------
// A line is cut into chunks of 8 points; lane l of a warp holds chunk
// 26 w + l - 3 of the sequence of all lines' chunks and gives the results of
// lanes 3 .. 28 (three chunks are the 24 points the recurrences reach).  The
// points are loaded and stored coalesced, 32 at a time, and change places
// through a shared-memory tile that the warp has to itself.
constexpr int SC_H = 3;                       // halo lanes on either side (24 points)
constexpr int SC_USE = 32 - 2 * SC_H;         // lanes that give results
constexpr int SC_FS = 4 + 8 * 36 + 4;         // floats of a field's tile: 32 points and 4 pad words, 8 times, halo words
inline size_t scan_smem(int nf, int warps) { return (size_t)SC_FS * nf * warps * sizeof(float); }

// One warp's chunks: wid = w, sm = the warp's tile (NF x SC_FS floats).
// VEC: N and the field stride are multiples of 4 and the pointers 16-byte
// aligned, so a lane loads and stores 4 points at a time.  SHORT: lines of
// fewer than SC_SHORT points, which feel both walls; they take the tabulated
// factors row by row.  Longer lines take constant coefficients throughout,
// and what the low wall's first factors would have changed is added
// afterwards: started from the explicit value d_e = g_e next to the implicit
// rows, the recurrences give x_e = g_e - c x_{e+1} instead of g_e, and the
// solution that corrects it is c x_{e+1} (-c)^k, k rows in.
template <int MODE, bool VEC, bool SHORT>
__device__ __forceinline__ void scan_body(const Sweep32Args &a, const int wid, float *sm)
{
    using M = SweepMode<MODE>;
    constexpr int NF = M::NF, NIN = M::NIN, HW = M::HW, NEXP = M::NEXP, NB = M::NB, P = SC_P;
    constexpr bool ADD = sweep_adds(MODE, 0);
    constexpr unsigned ALL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int N = a.N;
    const int id = wid * SC_USE + lane - SC_H;
    const bool ok = id >= 0 && id < a.tot;
    const int line = ok ? id / a.nch : 0, ch = ok ? id - line * a.nch : 0;
    const int g0 = ch * P;                    // first row of the chunk
    const int cnt = ok ? min(P, N - g0) : 0;  // its rows
    const int addr = line * N + g0;
    float *const tile = sm + 4;

    // ---- stage: E consecutive points per lane, KB times 32 E in flight ----
    constexpr int E = VEC ? 4 : 1, KS = 256 / (32 * E), KB = VEC ? 2 : 4;
    // lane's points of pass k: chunk src of the warp, from point el on
    auto src_of = [&](int k) { return (32 * E * k + E * lane) >> 3; };
    const int el = (E * lane) & 7;
    float bl[3] = {0.0f, 0.0f, 0.0f};  // base values of the lane's own chunk (gravity not along x)
    if constexpr (NB > 0) {
        if (a.ga != 0) {
            const int gk = a.ga == 1 ? line % a.n[1] : line / a.n[1];
            bl[0] = a.b0[gk];
            bl[1] = a.b1[gk];
            if constexpr (NB > 2) bl[2] = a.b2[gk];
        }
    }
    // SHORT: four more points on either side of the warp's (lanes 0 .. 3 load
    // those before, lanes 4 .. 7 those after), for the end lanes' stencils.
    // Longer lines leave the end lanes' outermost rows, which would need them,
    // out of what they pass on (22 rows or more from a result).  Either way a
    // result does not depend on where in a warp its chunk sits: equal lines
    // give equal bits, and a slab's lines those of the whole box.
    float eu[NIN];
    float ey[3] = {0.0f, 0.0f, 0.0f};
    bool ein = false;
    if constexpr (SHORT) {
        const int src = lane < 4 ? 0 : 31, d = lane < 4 ? lane - 4 : lane + 4;
        const int A = __shfl_sync(ALL, addr, src), g = __shfl_sync(ALL, g0, src) + d, C = __shfl_sync(ALL, cnt, src);
        ein = lane < 8 && C > 0 && g >= 0 && g < N;
        const int p = ein ? A + d : addr;
#pragma unroll
        for (int m = 0; m < NIN; ++m) eu[m] = a.in[m][p];
        if constexpr (NB > 0) {
            const int ge = ein ? g : 0;
#pragma unroll
            for (int i = 0; i < NB; ++i) ey[i] = __shfl_sync(ALL, bl[i], src);
            if (a.ga == 0) {
                ey[0] = a.b0[ge];
                ey[1] = a.b1[ge];
                if constexpr (NB > 2) ey[2] = a.b2[ge];
            }
        }
    }
#pragma unroll
    for (int kb = 0; kb < KS; kb += KB) {
        float v[KB][NIN][E], bb[KB][E][3];
        bool in[KB];
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const int src = src_of(kb + k);
            const int A = __shfl_sync(ALL, addr, src), C = __shfl_sync(ALL, cnt, src);
            in[k] = el < C;
            const int p = in[k] ? A + el : A;  // a chunk's first points stand in for missing ones
#pragma unroll
            for (int m = 0; m < NIN; ++m) {
                if constexpr (VEC) {
                    const float4 t = *reinterpret_cast<const float4 *>(a.in[m] + p);
                    v[k][m][0] = t.x, v[k][m][1] = t.y, v[k][m][2] = t.z, v[k][m][3] = t.w;
                } else {
                    v[k][m][0] = a.in[m][p];
                }
            }
            if constexpr (NB > 0) {
                if (a.ga != 0) {
#pragma unroll
                    for (int i = 0; i < NB; ++i) {
                        const float y = __shfl_sync(ALL, bl[i], src);
#pragma unroll
                        for (int e = 0; e < E; ++e) bb[k][e][i] = y;
                    }
                } else {
                    const int gs = __shfl_sync(ALL, g0, src), kk = in[k] ? gs + el : 0;
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        bb[k][e][0] = a.b0[kk + e];
                        bb[k][e][1] = a.b1[kk + e];
                        if constexpr (NB > 2) bb[k][e][2] = a.b2[kk + e];
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            float f[E][NF];
#pragma unroll
            for (int e = 0; e < E; ++e) {
                float u[NIN];
#pragma unroll
                for (int m = 0; m < NIN; ++m) u[m] = v[k][m][e];
                sweep_point<MODE, 0>(u, bb[k][e], a.hp, f[e]);
            }
            const int pos = 32 * E * (kb + k) + E * lane;
            float *const t = tile + pos + 4 * (pos >> 5);
#pragma unroll
            for (int m = 0; m < NF; ++m) {
#pragma unroll
                for (int e = 0; e < E; ++e) f[e][m] = in[k] ? f[e][m] : 0.0f;
                if constexpr (VEC)
                    *reinterpret_cast<float4 *>(t + m * SC_FS) = make_float4(f[0][m], f[1][m], f[2][m], f[3][m]);
                else
                    t[m * SC_FS] = f[0][m];
            }
        }
    }
    if (lane < 8) {
        float f[NF];
#pragma unroll
        for (int m = 0; m < NF; ++m) f[m] = 0.0f;
        if constexpr (SHORT) {
            if (ein) sweep_point<MODE, 0>(eu, ey, a.hp, f);
        }
        float *const t = tile + (lane < 4 ? lane - 4 : 288 + lane - 4);
#pragma unroll
        for (int m = 0; m < NF; ++m) t[m * SC_FS] = f[m];
    }
    __syncwarp();

    // ---- solve ----
    const int po = 8 * lane + 4 * (lane >> 2);                              // own points
    const int pl = lane ? (8 * lane - 4) + 4 * ((8 * lane - 4) >> 5) : -4;  // 4 before
    const int pr = (8 * lane + 8) + 4 * ((8 * lane + 8) >> 5);              // 4 after
    const float c = a.c;
    // explicit row N - 1 - r sits at point hj - r of this lane's chunk
    const int hj = N - 1 - g0;
    const bool lo = ok && ch == 0, hi = ok && hj - (NEXP - 1) < P;
    const bool anylo = __any_sync(ALL, lo), anyhi = __any_sync(ALL, hi);
    // neighbours on the lane's left and right that hold chunks of its own line.
    // Values of the others are left out by selection: a weight of zero would
    // let a NaN or an infinity of one line through to the next.
    const int left = ok ? min(ch, lane) : 0, right = ok ? min(a.nch - 1 - ch, 31 - lane) : 0;
    // weights of the second and third neighbours' end values in the state that
    // enters the lane (the first one's is 1)
    float wl1 = a.pw[P - 1], wl2 = a.pw16, wr1 = a.pw[P - 1], wr2 = a.pw16;
    // SHORT: factor of a row, its pivot's ratio to the limit (0 for explicit
    // rows), weight at a row of the state entering from the left and right
    float cp[P], rt[P], pf[P], ps[P];
    if constexpr (SHORT) {
#pragma unroll
        for (int j = 0; j < P; ++j) {
            const int g = g0 + j, row = min(g, SW_TAB - 1);
            cp[j] = g < N - NEXP ? a.cp[row] : 0.0f;
            rt[j] = g < N - NEXP ? a.rat[row] : 0.0f;
            pf[j] = j ? __fmul_rn(-cp[j], pf[j ? j - 1 : 0]) : -cp[j];
        }
#pragma unroll
        for (int j = P - 1; j >= 0; --j) ps[j] = j < P - 1 ? __fmul_rn(-cp[j], ps[j < P - 1 ? j + 1 : j]) : -cp[j];
        wl1 = __shfl_up_sync(ALL, pf[P - 1], 1), wl2 = wl1 * __shfl_up_sync(ALL, pf[P - 1], 2);
        wr1 = __shfl_down_sync(ALL, ps[0], 1), wr2 = wr1 * __shfl_down_sync(ALL, ps[0], 2);
    }
    const bool near_lo = ok && ch <= SC_H;  // chunks that the low wall's first factors reach
    const float kf = near_lo ? a.kf[ch] : 0.0f;
#pragma unroll 1
    for (int m = 0; m < NF; ++m) {
        float *const t = tile + m * SC_FS;
        float w[P + 8];  // w[4 + j]: point j
        {
            const float4 q1 = *reinterpret_cast<const float4 *>(t + po), q2 = *reinterpret_cast<const float4 *>(t + po + 4);
            w[4] = q1.x, w[5] = q1.y, w[6] = q1.z, w[7] = q1.w;
            w[8] = q2.x, w[9] = q2.y, w[10] = q2.z, w[11] = q2.w;
            if constexpr (HW > 2) w[1] = t[pl + 1], w[14] = t[pr + 2];
            const float2 q0 = *reinterpret_cast<const float2 *>(t + pl + 2), q3 = *reinterpret_cast<const float2 *>(t + pr);
            w[2] = q0.x, w[3] = q0.y;
            w[12] = q3.x, w[13] = q3.y;
            if constexpr (SHORT) {
                // the next line's points, in the stencils of rows beyond this
                // line's end
                if (ok && ch == a.nch - 1) w[12] = w[13] = 0.0f;
                if constexpr (HW > 2) w[14] = ok && ch == a.nch - 1 ? 0.0f : w[14];
            }
        }
        float d[P], gl[NEXP], gh[NEXP];
#pragma unroll
        for (int j = 0; j < P; ++j) {
            d[j] = sweep_rhs<MODE>(a, w + 4 + j - HW, 1);
            if constexpr (SHORT) d[j] = __fmul_rn(rt[j], d[j]);
        }
        if (anylo) {
#pragma unroll
            for (int r = 0; r < NEXP; ++r) {
                gl[r] = 0.0f;
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (sweep_tap<MODE>(r, j)) gl[r] = __fmaf_rn(a.ex[r][j], w[4 + j], gl[r]);
                // the last explicit value starts the recurrence
                if (lo) d[r] = SHORT || r == NEXP - 1 ? gl[r] : 0.0f;
            }
        }
        if (anyhi) {
            if (hi) {
#pragma unroll
                for (int r = 0; r < NEXP; ++r) {
                    gh[r] = 0.0f;
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        // points left of lane 0 are not in the tile (lane 0
                        // gives no results)
                        const int q = max(8 * lane + hj - i, 0);
                        if (sweep_tap<MODE>(r, i)) gh[r] = __fmaf_rn(a.ex[r][i], t[q + 4 * (q >> 5)], gh[r]);
                    }
                    gh[r] = __fmul_rn(a.exs, gh[r]);
                }
                if constexpr (SHORT) {
#pragma unroll
                    for (int r = 0; r < NEXP; ++r)
#pragma unroll
                        for (int j = 0; j < P; ++j)
                            if (j == hj - r) d[j] = gh[r];
                }
            }
        }
        // what a lane passes on to its third neighbour: without its outermost
        // rows, whose stencils reach outside the lane
        float dq = 0.0f, xq = 0.0f;
        if constexpr (!SHORT) {
            dq = d[HW];
#pragma unroll
            for (int j = HW + 1; j < P; ++j) dq = __fmaf_rn(-c, dq, d[j]);
        }
#pragma unroll
        for (int j = 1; j < P; ++j) d[j] = __fmaf_rn(SHORT ? -cp[j] : -c, d[j - 1], d[j]);
        {
            const float d1 = __shfl_up_sync(ALL, d[P - 1], 1), d2 = __shfl_up_sync(ALL, d[P - 1], 2),
                        d3 = __shfl_up_sync(ALL, SHORT ? d[P - 1] : dq, 3);
            float y = left > 0 ? d1 : 0.0f;
            if (left > 1) y = __fmaf_rn(wl1, d2, y);
            if (left > 2) y = __fmaf_rn(wl2, d3, y);
#pragma unroll
            for (int j = 0; j < P; ++j) d[j] = __fmaf_rn(SHORT ? pf[j] : a.pw[j], y, d[j]);
        }
        if (!SHORT && anyhi && hi) {
            // the backward recurrence starts from the last explicit value
#pragma unroll
            for (int j = 0; j < P; ++j) {
                if (j == hj - (NEXP - 1)) d[j] = gh[NEXP - 1];
                if (j > hj - (NEXP - 1)) d[j] = 0.0f;
            }
        }
        if constexpr (!SHORT) {
            xq = d[P - HW - 1];
#pragma unroll
            for (int j = P - HW - 2; j >= 0; --j) xq = __fmaf_rn(-c, xq, d[j]);
        }
#pragma unroll
        for (int j = P - 2; j >= 0; --j) d[j] = __fmaf_rn(SHORT ? -cp[j] : -c, d[j + 1], d[j]);
        {
            const float x1 = __shfl_down_sync(ALL, d[0], 1), x2 = __shfl_down_sync(ALL, d[0], 2),
                        x3 = __shfl_down_sync(ALL, SHORT ? d[0] : xq, 3);
            float z = right > 0 ? x1 : 0.0f;
            if (right > 1) z = __fmaf_rn(wr1, x2, z);
            if (right > 2) z = __fmaf_rn(wr2, x3, z);
#pragma unroll
            for (int j = 0; j < P; ++j) d[j] = __fmaf_rn(SHORT ? ps[j] : a.pw[P - 1 - j], z, d[j]);
        }
        if constexpr (!SHORT) {
            if (anylo) {
                const float x0 = __shfl_sync(ALL, d[NEXP], max(lane - ch, 0));
                const float y = near_lo ? __fmul_rn(kf, x0) : 0.0f;
#pragma unroll
                for (int j = 0; j < P; ++j) d[j] = __fmaf_rn(a.pw[j], y, d[j]);
                if (lo) {
#pragma unroll
                    for (int r = 0; r < NEXP; ++r) d[r] = gl[r];
                }
            }
            if (anyhi && hi) {
#pragma unroll
                for (int r = 0; r < NEXP - 1; ++r)
#pragma unroll
                    for (int j = 0; j < P; ++j)
                        if (j == hj - r) d[j] = gh[r];
            }
        }
        __syncwarp();  // the neighbours have read their halo points
        *reinterpret_cast<float4 *>(t + po) = make_float4(d[0], d[1], d[2], d[3]);
        *reinterpret_cast<float4 *>(t + po + 4) = make_float4(d[4], d[5], d[6], d[7]);
        if constexpr (SHORT) {
            // explicit rows have their own values, whatever the others hold
#pragma unroll
            for (int r = 0; r < NEXP; ++r) {
                if (lo) t[po + r] = gl[r];
                if (hi && hj >= r && hj - r < P) t[po + hj - r] = gh[r];
            }
        }
    }
    __syncwarp();

    // ---- store ----
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const int src = src_of(k);
        const int A = __shfl_sync(ALL, addr, src), C = __shfl_sync(ALL, cnt, src);
        if (el < C && src >= SC_H && src < 32 - SC_H) {
            const int pos = 32 * E * k + E * lane;
            const float *const t = tile + pos + 4 * (pos >> 5);
#pragma unroll
            for (int m = 0; m < NF; ++m) {
                float *const o = a.out[m] + A + el;
                if constexpr (VEC && !ADD) {
                    *reinterpret_cast<float4 *>(o) = *reinterpret_cast<const float4 *>(t + m * SC_FS);
                } else {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        if constexpr (ADD)
                            atomicAdd(o + e, t[m * SC_FS + e]);
                        else
                            o[e] = t[m * SC_FS + e];
                    }
                }
            }
        }
    }
}

// the variant for the lines and fields at hand
template <int MODE>
__device__ __forceinline__ void scan_any(const Sweep32Args &a, const int wid, float *sm)
{
    if (a.kind == 2)
        scan_body<MODE, true, false>(a, wid, sm);
    else if (a.kind == 1)
        scan_body<MODE, false, false>(a, wid, sm);
    else
        scan_body<MODE, false, true>(a, wid, sm);
}

}  // namespace nopcs
