// Device bodies of the NOHAP line sweeps (arXiv 2203.00879, Sec. 3): the
// sub-domain sweep (line_body) and the whole-line x sweep (xline_body), each
// for one block given as a block index of its launch grid.  The header comment
// of line_kernels.cu describes the algorithm.
#pragma once

#include "line_solve.cuh"

namespace nopcs {

template <typename T>
struct LineArgs {
    int n[3];
    int lines;      // lines per block (LINES)
    int ntile_a;    // tiles along the line-tile axis
    int rt;         // staged-row capacity (op.max_tile): tile rows along x
    int rw;         // solve-window capacity (op.max_win): tile rows along y, z
    // one base pointer per field, so a node is one 32-bit index away from a
    // kernel parameter (fields hold < 2^31 points)
    const T *in[6]; // FIELD: f; FLUX: W (6 fields); FILTER: Q (5 fields);
                    // VGRAD: W (first 5 fields); VDIV: 4 flux fields
    T *out[5];      // FIELD: df; FLUX: R (5 fields); FILTER: Qout (5 fields);
                    // VGRAD: 4 gradient fields; VDIV: R[1..4]
    T scale;        // 1/h for FIELD, FLUX, VGRAD and VDIV
    int first;      // FLUX: store (1) or subtract (0)
    int ga;         // gravity axis
    const T *b0;    // FLUX: rho_b, FILTER: rho_b, VGRAD: T_b (FP32) / rho_b (FP64)
    const T *b1;    // FLUX: H_b,   FILTER: E_b,   VGRAD: 1/p_b (FP32) / p_b (FP64)
    const T *b2;    // VGRAD: 1/rho_b (FP32)
    T gm2;          // VGRAD: gamma M^2 (FP64)
    T w[2][4];      // sub-domain sweep: right-hand-side weights (nohap_solve_column)
};

// the factor on a sweep's results: 1 / h, and the flux's sign
template <typename T, int MODE>
__host__ __device__ __forceinline__ T line_factor(const LineArgs<T> &a)
{
    return MODE == MODE_FILTER ? T(1) : (MODE == MODE_FLUX ? -a.scale : a.scale);
}

// One block of the sub-domain sweep: block `vblock` of the launch grid
// (sub-domain vblock % nsub of line tile vblock / nsub), in the block's
// dynamic shared memory.  The shared array is declared here rather than passed
// in.
template <typename T, int MODE, int AXIS>
__device__ __forceinline__ void line_body(const LineOpDev &op, const LineArgs<T> &a, const unsigned vblock)
{
    extern __shared__ __align__(32) unsigned char smraw[];
    const int NT = (int)blockDim.x;
    constexpr bool SINGLE = MODE == MODE_FIELD || MODE == MODE_FIELD2;  // one field in, one out
    constexpr bool VISC = MODE == MODE_VGRAD || MODE == MODE_VDIV;      // four fields out
    constexpr int NF = SINGLE ? 1 : (VISC ? 4 : 5);
    constexpr int NIN = SINGLE ? 1 : (MODE == MODE_FLUX ? 6 : (MODE == MODE_VDIV ? 4 : 5));
    // rows in flight per thread and staging pass: four along x, three along y
    // and z (the y and z flux sweeps ran 3% and 1% faster with three than
    // with four; x 4% slower; more rows than four cost occupancy)
    constexpr int U = AXIS == 0 ? 4 : 3;
    // STREAM: the end-row dot products are summed while staging and only the
    // solve window is kept (four blocks per SM instead of three for the flux
    // sweeps); along x a warp walks one line and reduces its lanes' sums with
    // shuffles.  The single-field derivative along x keeps the whole staged
    // tile and takes the dot products in the solve (faster there).
    constexpr bool STREAM = AXIS != 0 || !SINGLE;
    const int LINES = a.lines, LP = a.lines + 1, RW = STREAM ? a.rw : a.rt;
    const int KC = sizeof(T) == 8 ? op.kconv64 : op.kconv32;
    // row groups sharing a line while staging along y, z (one warp along x)
    const int RG = STREAM ? (AXIS == 0 ? 1 : NT / LINES) : 0;
    // shared memory: end-row taps (2 x max_taps), Thomas factors (2 x KC),
    // end-row partial sums [RG][2][NF][LINES], tile [NF][RW][LP]
    T *cs = reinterpret_cast<T *>(smraw);
    T *ce = cs + op.max_taps;
    T *tcp = ce + op.max_taps;
    T *tiv = tcp + KC;
    T *part = tiv + KC;
    T *sm = part + (size_t)RG * 2 * NF * LINES;
    const int nx = a.n[0], ny = a.n[1];

    // unsigned block index: the compiler then knows the tile coordinates are
    // non-negative (with a signed index the z sweep ran 5% slower)
    const int b = vblock % (unsigned)op.nsub;
    const int tile = vblock / (unsigned)op.nsub;
    const int ta = tile % a.ntile_a;
    const int cc = tile / a.ntile_a;
    const int a0 = ta * LINES;
    const int Na = AXIS == 0 ? ny : nx;
    const int nl = min(LINES, Na - a0);

    const int *rec = op.sub + b * SUB_REC;
    const int s = rec[0], e = rec[1], tlo = rec[2], thi = rec[3];
    const int j0s = rec[4], lens = rec[5], j0e = rec[7], lene = rec[8];
    const int org = STREAM ? rec[12] : tlo, last = STREAM ? rec[13] : thi;  // tile rows
    const int nrows = thi - tlo + 1;
    const int srow = AXIS == 0 ? 1 : (AXIS == 1 ? nx : nx * ny);
    const int sa = AXIS == 0 ? nx : 1;
    const int sc = AXIS == 2 ? nx : nx * ny;
    const int gbase = cc * sc + a0 * sa + tlo * srow;
    // which of (row, line, cc) is the coordinate along the gravity axis
    const int gsel = a.ga == AXIS ? 0 : (a.ga == (AXIS == 0 ? 1 : 0) ? 1 : 2);
    const size_t fs = (size_t)RW * LP;

    // ---- block constants: end-row taps and the unconverged Thomas factors ----
    // (STREAM reads the taps from the global table while staging: no barrier
    // between these loads and the staging loads)
    const T *coef = coef_ptr<T>(op);
    {
        if (!STREAM) {
            for (int k = threadIdx.x; k < lens; k += NT) cs[k] = coef[rec[6] + k];
            for (int k = threadIdx.x; k < lene; k += NT) ce[k] = coef[rec[9] + k];
        }
        const T *cpp = cp_ptr<T>(op), *ivp = inv_ptr<T>(op);
        for (int k = threadIdx.x; k < KC; k += NT) {
            tcp[k] = cpp[k];
            tiv[k] = ivp[k];
        }
    }

    // ---- stage rows [tlo, thi] of nl lines --------------------------------------
    // Rows [org, last] go to the tile [field][row][line].  STREAM: every
    // staged row also feeds the two end-row dot products
    // g_i = sum_j C_ij f_j (Eq. CS:fpCf_i) as it passes, so the end-row
    // supports outside the solve window need no shared memory.
    // x: a warp walks the rows of one line (coalesced along x, transposed into
    // the odd line pitch); y, z: consecutive threads take consecutive lines.
    {
        int r0, rstep, l0, lstep;
        if (AXIS == 0) {
            r0 = threadIdx.x & 31;
            rstep = 32;
            l0 = (int)threadIdx.x >> 5;
            lstep = NT >> 5;
        } else {
            l0 = threadIdx.x % LINES;
            lstep = LINES;  // one line per thread
            r0 = threadIdx.x / LINES;
            rstep = RG;
            if (r0 >= RG) l0 = LINES;  // threads beyond RG x LINES do not stage
        }
        for (int l = l0; l < (AXIS == 0 ? nl : LINES); l += lstep) {
            const int src = gbase + l * sa;
            const int gl = gsel == 1 ? a0 + l : cc;
            T ps[NF], pe[NF];
#pragma unroll
            for (int f = 0; f < NF; ++f) ps[f] = pe[f] = T(0);
            for (int r = r0; l < nl && r < nrows; r += U * rstep) {
                T v[U][NIN];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int rr = r + u * rstep;
                    if (rr < nrows) {
                        const int p = src + rr * srow;
#pragma unroll
                        for (int k = 0; k < NIN; ++k) v[u][k] = a.in[k][p];
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int rr = r + u * rstep;
                    if (rr >= nrows) continue;
                    const int g = tlo + rr;
                    T val[NF];
                    if constexpr (SINGLE) {
                        val[0] = v[u][0];
                    } else if constexpr (MODE == MODE_FLUX) {
                        const int gk = gsel == 0 ? g : gl;
                        const T rho = a.b0[gk] + v[u][0];
                        const T uu = v[u][1], vv = v[u][2], ww = v[u][3], pp = v[u][4];
                        const T H = a.b1[gk] + v[u][5];
                        const T ud = AXIS == 0 ? uu : (AXIS == 1 ? vv : ww);
                        const T m = rho * ud;
                        val[0] = m;
                        val[1] = m * uu + (AXIS == 0 ? pp : T(0));
                        val[2] = m * vv + (AXIS == 1 ? pp : T(0));
                        val[3] = m * ww + (AXIS == 2 ? pp : T(0));
                        val[4] = H * ud;
                    } else if constexpr (MODE == MODE_VGRAD) {
                        // u, v, w and T = gamma M^2 p / rho of the stage state
                        const int gk = gsel == 0 ? g : gl;
                        val[0] = v[u][1];
                        val[1] = v[u][2];
                        val[2] = v[u][3];
                        if constexpr (sizeof(T) == 4) {
                            // T_b (1 + p'/p_b) / (1 + rho'/rho_b) on the deviations
                            const T rr = v[u][0] * a.b2[gk];
                            val[3] = a.b0[gk] + __fdividef(a.b0[gk] * (v[u][4] * a.b1[gk] - rr), 1.0f + rr);
                        } else {
                            val[3] = a.gm2 * (a.b1[gk] + v[u][4]) / (a.b0[gk] + v[u][0]);
                        }
                    } else if constexpr (MODE == MODE_VDIV) {
#pragma unroll
                        for (int f = 0; f < 4; ++f) val[f] = v[u][f];
                    } else {  // FILTER on Q - base (no base tables: the input is a deviation already)
                        const int gk = gsel == 0 ? g : gl;
                        val[0] = a.b0 ? v[u][0] - a.b0[gk] : v[u][0];
                        val[1] = v[u][1];
                        val[2] = v[u][2];
                        val[3] = v[u][3];
                        val[4] = a.b1 ? v[u][4] - a.b1[gk] : v[u][4];
                    }
                    if (!STREAM || (g >= org && g <= last)) {
                        T *d = sm + (size_t)(g - org) * LP + l;
#pragma unroll
                        for (int f = 0; f < NF; ++f) d[f * fs] = val[f];
                    }
                    if constexpr (STREAM) {
                        const unsigned ks = (unsigned)(g - j0s), ke = (unsigned)(g - j0e);
                        if (ks < (unsigned)lens) {
                            const T c = __ldg(coef + rec[6] + ks);
#pragma unroll
                            for (int f = 0; f < NF; ++f) ps[f] += c * val[f];
                        }
                        if (ke < (unsigned)lene) {
                            const T c = __ldg(coef + rec[9] + ke);
#pragma unroll
                            for (int f = 0; f < NF; ++f) pe[f] += c * val[f];
                        }
                    }
                }
            }
            if constexpr (STREAM) {
                if constexpr (AXIS == 0) {
                    // sum over the lanes, halving the sums a lane carries with
                    // their number of addends: 16 additions for the ten sums
                    // instead of 50 in a butterfly of each (FP64,
                    // 128^3: 0.42 -> 0.31 ms, with the shorter solve)
                    __syncwarp();
                    T sv[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) sv[k] = k < NF ? ps[k < NF ? k : 0] : (k < 2 * NF ? pe[k < 2 * NF ? k - NF : 0] : T(0));
#pragma unroll
                    for (int o = 16; o >= 2; o >>= 1) {
                        const bool up = (r0 & o) != 0;
                        const int half = o / 2;  // sums kept
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            if (k >= half) continue;
                            const T give = up ? sv[k] : sv[k + half], keep = up ? sv[k + half] : sv[k];
                            sv[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                        }
                    }
                    sv[0] += __shfl_xor_sync(0xffffffffu, sv[0], 1);
                    // lane 2 k holds sum k
                    if (!(r0 & 1) && (r0 >> 1) < 2 * NF) part[(size_t)(r0 >> 1) * LINES + l] = sv[0];
                } else {
                    T *pp = part + l + (size_t)r0 * 2 * NF * LINES;  // [k][which][f][line]
#pragma unroll
                    for (int f = 0; f < NF; ++f) {
                        pp[(size_t)f * LINES] = ps[f];
                        pp[(size_t)(NF + f) * LINES] = pe[f];
                    }
                }
            }
        }
    }
    __syncthreads();

    // ---- per-(line, field) NOHAP solve ----------------------------------------
    {
        const int l = threadIdx.x % LINES;
        const int fld = threadIdx.x / LINES;
        if (l < nl && fld < NF) {
            T *col = sm + (size_t)fld * fs + l;
            T gs = 0, ge = 0;
            if constexpr (STREAM) {
                for (int k = 0; k < RG; ++k) {
                    gs += part[((size_t)k * 2 * NF + fld) * LINES + l];
                    ge += part[((size_t)k * 2 * NF + NF + fld) * LINES + l];
                }
            } else {
                gs = dot_col(cs, col + (size_t)(j0s - org) * LP, lens, LP);
                if (lene > 0) ge = dot_col(ce, col + (size_t)(j0e - org) * LP, lene, LP);
            }
            nohap_solve_column<T, MODE>(op, a.w, col, LP, org, gs, ge, tcp, tiv, KC, rec, line_factor<T, MODE>(a));
        }
    }
    __syncthreads();

    // ---- write the sub-domain's own rows ---------------------------------------
    {
        const int nown = e - s + 1;
        int r0, rstep, l0, lstep;
        if (AXIS == 0) {
            r0 = threadIdx.x & 31;
            rstep = 32;
            l0 = (int)threadIdx.x >> 5;
            lstep = NT >> 5;
        } else {
            l0 = (int)threadIdx.x % LINES;
            lstep = LINES;
            r0 = threadIdx.x / LINES;
            rstep = NT / LINES;
        }
        const int obase = gbase + (s - tlo) * srow;
        for (int ll = l0; ll < nl; ll += lstep) {
            const int dstg = obase + ll * sa;
            const T *srcs = sm + (size_t)(s - org) * LP + ll;
            const int gl = gsel == 1 ? a0 + ll : cc;
            for (int r = r0; r < nown; r += U * rstep) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int rr = r + u * rstep;
                    if (rr >= nown) continue;
                    const T *src = srcs + (size_t)rr * LP;
                    const int o = dstg + rr * srow;
                    if constexpr (SINGLE) {
                        a.out[0][o] = src[0];
                    } else if constexpr (MODE == MODE_FLUX) {
#pragma unroll
                        for (int f = 0; f < 5; ++f) {
                            const T v = src[f * fs];
                            // later sweeps add through a reduction performed
                            // in L2 (the old value never travels to the SM,
                            // so the store phase waits on no load); every
                            // element takes exactly one addition per sweep,
                            // the same rounding as load + add + store
                            if (a.first)
                                a.out[f][o] = v;
                            else
                                atomicAdd(&a.out[f][o], v);
                        }
                    } else if constexpr (MODE == MODE_VGRAD) {
#pragma unroll
                        for (int f = 0; f < 4; ++f) a.out[f][o] = src[f * fs];
                    } else if constexpr (MODE == MODE_VDIV) {
                        // one addition per element and sweep, as for the flux
#pragma unroll
                        for (int f = 0; f < 4; ++f) atomicAdd(&a.out[f][o], src[f * fs]);
                    } else {
                        const int gk = gsel == 0 ? s + rr : gl;
                        a.out[0][o] = a.b0 ? src[0] + a.b0[gk] : src[0];
                        a.out[1][o] = src[fs];
                        a.out[2][o] = src[2 * fs];
                        a.out[3][o] = src[3 * fs];
                        a.out[4][o] = a.b1 ? src[4 * fs] + a.b1[gk] : src[4 * fs];
                    }
                }
            }
        }
    }
}

// ---- whole-line sweep along x -------------------------------------------------
// Along x a grid line is contiguous in memory and short enough (N x 5 fields
// x 8 B = 40 KB at N = 1024) for a block to stage a whole line at once.
// Every point is then loaded once -- a sub-domain tile also reads the 2 x 48
// end-row support points of its neighbours, 2.5 times its own points at
// sub-domains of 64 -- and the end rows read their supports from the staged
// line instead of summing partial products across a warp.  Each thread
// solves one (field, sub-domain) column in three phases separated by
// barriers, so that no column reads a row another column has overwritten:
//   A. the two end values g_i = sum_j C_ij f_j (Eq. CS:fpCf_i) and any
//      explicit wall row, from the staged inputs;
//   B. the Thomas solve of the implicit rows in place: it reads rows s-1 ..
//      e+1, and the only rows of other columns among them (s-1 and e+1) are
//      their end rows, which phase B never writes;
//   C. the end and wall values into their rows.
// The layout is [field][row] with one pad word per 32 rows and a field
// pitch chosen on the host (LineOpDev::xpitch) so that the columns a warp's
// threads take (neighbouring sub-domains, then the next field) fall in
// different banks.  The line's end-row taps (a few KB) are copied to shared
// memory once per block: the threads of a warp read the taps of different
// sub-domains, which from global memory would touch a cache line each.
__host__ __device__ __forceinline__ int xrow(int g) { return g + (g >> 5); }

// Inviscid flux along x (Eq. ge3) of one point's stage primitives
// v = (rho - rho_b, u, v, w, p, H - H_b) into the tile rows d[k FS], k = 0..4;
// gk is the point's coordinate along gravity.
template <typename T>
__device__ __forceinline__ void xline_flux_point(const LineArgs<T> &a, T *d, const size_t FS, const T v[6],
                                                 const int gk)
{
    const T rho = a.b0[gk] + v[0];
    const T uu = v[1], vv = v[2], ww = v[3], pp = v[4];
    const T H = a.b1[gk] + v[5];
    const T m = rho * uu;
    d[0] = m;
    d[FS] = m * uu + pp;
    d[2 * FS] = m * vv;
    d[3 * FS] = m * ww;
    d[4 * FS] = H * uu;
}

template <typename T>
__device__ __forceinline__ void xline_solve_store(const LineOpDev &op, const LineArgs<T> &a, T *sm,
                                                  const T *ctab, const T *tcp, const T *tiv, const int base);

// One block of the whole-line x sweep: one line (= y + ny z), in the block's
// dynamic shared memory.
template <typename T>
__device__ __forceinline__ void xline_body(const LineOpDev &op, const LineArgs<T> &a, const int line)
{
    extern __shared__ __align__(32) unsigned char smraw[];
    constexpr int NF = 5, NIN = 6;
    constexpr int U = 4;     // staged points in flight per thread and field
    const int N = op.N;      // = nx
    const int ny = a.n[1];
    const size_t FS = a.rt;  // field pitch (padded)
    const int KC = sizeof(T) == 8 ? op.kconv64 : op.kconv32;
    T *sm = reinterpret_cast<T *>(smraw);
    T *ctab = sm + NF * FS;  // end-row taps
    T *tcp = ctab + op.ncoef;
    T *tiv = tcp + KC;
    const int base = line * N;
    {
        const T *cpp = cp_ptr<T>(op), *ivp = inv_ptr<T>(op), *cf = coef_ptr<T>(op);
        for (int k = threadIdx.x; k < KC; k += blockDim.x) {
            tcp[k] = cpp[k];
            tiv[k] = ivp[k];
        }
        for (int k = threadIdx.x; k < op.ncoef; k += blockDim.x) ctab[k] = cf[k];
    }
    // ---- stage the line: consecutive threads take consecutive points ----
    const int gl = a.ga == 1 ? line % ny : line / ny;  // coordinate along gravity (y or z)
    for (int g0 = threadIdx.x; g0 < N; g0 += U * blockDim.x) {
        T v[U][NIN];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int g = g0 + u * (int)blockDim.x;
            if (g < N) {
#pragma unroll
                for (int k = 0; k < NIN; ++k) v[u][k] = a.in[k][base + g];
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int g = g0 + u * (int)blockDim.x;
            if (g >= N) continue;
            xline_flux_point(a, sm + xrow(g), FS, v[u], a.ga == 0 ? g : gl);
        }
    }
    __syncthreads();
    xline_solve_store<T>(op, a, sm, ctab, tcp, tiv, base);
}

// The solve and the store of the whole-line x sweep, once the line is staged in
// sm (and a barrier has passed): the columns, thread c solving sub-domain
// c % nsub of field c / nsub, in phases A-C, then the rows scaled by 1/h into the
// outputs, from element base on.
template <typename T>
__device__ __forceinline__ void xline_solve_store(const LineOpDev &op, const LineArgs<T> &a, T *sm,
                                                  const T *ctab, const T *tcp, const T *tiv, const int base)
{
    constexpr int NF = 5;
    constexpr int NEXP = 2;  // explicit rows at each wall (derivative)
    const int N = op.N;      // = nx
    const size_t FS = a.rt;
    const int KC = sizeof(T) == 8 ? op.kconv64 : op.kconv32;
    const int nsub = op.nsub;
    const int c = threadIdx.x;
    const bool active = c < nsub * NF;
    const int b = c % nsub, f = c / nsub;
    const int *rec = op.sub + b * SUB_REC;
    T *col = sm + (size_t)f * FS;
    const int s = rec[0], e = rec[1], lo = rec[10], hi = rec[11];
    T gs = 0, ge = 0;
    T exL[NEXP], exH[NEXP];
#pragma unroll
    for (int r = 0; r < NEXP; ++r) exL[r] = exH[r] = T(0);
    // A. end values and explicit wall rows from the staged inputs
    if (active) {
        const T *coef = ctab;
        auto dot = [&](const T *cf, int j0, int len) {
            T s0 = 0, s1 = 0, s2 = 0, s3 = 0;
            int k = 0;
            for (; k + 4 <= len; k += 4) {
                s0 += cf[k] * col[xrow(j0 + k)];
                s1 += cf[k + 1] * col[xrow(j0 + k + 1)];
                s2 += cf[k + 2] * col[xrow(j0 + k + 2)];
                s3 += cf[k + 3] * col[xrow(j0 + k + 3)];
            }
            for (; k < len; ++k) s0 += cf[k] * col[xrow(j0 + k)];
            return (s0 + s1) + (s2 + s3);
        };
        gs = dot(coef + rec[6], rec[4], rec[5]);
        if (rec[8] > 0) ge = dot(coef + rec[9], rec[7], rec[8]);
#pragma unroll
        for (int r = 0; r < NEXP; ++r) {
            if (r > s && r < e) {
                T acc = 0;
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (op.ex[r][j] != 0.0) acc += (T)op.ex[r][j] * col[xrow(j)];
                exL[r] = acc;
            }
            const int rh = N - 1 - r;
            if (rh > s && rh < e) {
                T acc = 0;
#pragma unroll
                for (int j = 0; j < 5; ++j)
                    if (op.ex[r][j] != 0.0) acc += (T)op.ex[r][j] * col[xrow(N - 1 - j)];
                exH[r] = (T)op.ex_sign * acc;
            }
        }
    }
    __syncthreads();
    // B. Thomas over the implicit rows lo..hi, forward values in place; a
    // register window keeps the inputs rows i-2 .. i+2 that row i reads
    if (active && lo <= hi) {
        const int m = hi - lo + 1;
        const T al = (T)op.alpha;
        const T gL = lo == s + 1 ? gs : exL[NEXP - 1];
        const T gR = hi == e - 1 ? ge : exH[NEXP - 1];
        const T r0 = (T)op.rb[0], r1 = (T)op.rb[1];
        const T cL = (T)op.cpL, iL = (T)op.invL;
        T win[5];
#pragma unroll
        for (int j = 0; j < 4; ++j) win[j] = col[xrow(lo - 2 + j)];
        int gin = lo + 2, gout = lo;
        T dprev = 0;
        auto fwd = [&](T iv, T adj) {
            win[4] = col[xrow(gin)];
            ++gin;
            const T rhs = r0 * (win[3] - win[1]) + r1 * (win[4] - win[0]);
            const T dp = (rhs - adj - al * dprev) * iv;
            col[xrow(gout)] = dp;
            ++gout;
            dprev = dp;
#pragma unroll
            for (int j = 0; j < 4; ++j) win[j] = win[j + 1];
        };
        fwd(tiv[0], al * gL + (m == 1 ? al * gR : T(0)));
        const int kmid = min(KC, m - 1);
        int r = 1;
#pragma unroll 4
        for (; r < kmid; ++r) fwd(tiv[r], T(0));
#pragma unroll 4
        for (; r < m - 1; ++r) fwd(iL, T(0));
        if (m > 1) fwd(m - 1 < KC ? tiv[m - 1] : iL, al * gR);
        // back substitution from row hi - 1 down to lo
        T x = dprev;
        int g = hi - 1;
        r = m - 2;
#pragma unroll 4
        for (; r >= KC; --r, --g) {
            x = col[xrow(g)] - cL * x;
            col[xrow(g)] = x;
        }
#pragma unroll 4
        for (; r >= 0; --r, --g) {
            x = col[xrow(g)] - tcp[r] * x;
            col[xrow(g)] = x;
        }
    }
    __syncthreads();
    // C. end values and wall rows into their rows
    if (active) {
        col[xrow(s)] = gs;
        if (rec[8] > 0) col[xrow(e)] = ge;
#pragma unroll
        for (int r = 0; r < NEXP; ++r) {
            if (r > s && r < e) col[xrow(r)] = exL[r];
            const int rh = N - 1 - r;
            if (rh > s && rh < e) col[xrow(rh)] = exH[r];
        }
    }
    __syncthreads();
    // ---- store (scaled by 1/h; the flux sweep stores -dF/dx into R) ----
    for (int g = threadIdx.x; g < N; g += blockDim.x) {
        const int o = base + g;
        const int q = xrow(g);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const T v = -sm[(size_t)k * FS + q] * a.scale;
            if (a.first)
                a.out[k][o] = v;
            else
                atomicAdd(&a.out[k][o], v);
        }
    }
}


// ---- launch geometry (host) ----------------------------------------------------
constexpr size_t SMEM_BUDGET = 200 * 1024;
constexpr size_t XLINE_SMEM = 100 * 1024;  // whole-line x flux sweep: most shared memory of a block

inline int pick_lines(int pref, int rw, int nf, size_t esz)
{
    int L = pref;
    while (L > 1 && (size_t)nf * rw * (L + 1) * esz > SMEM_BUDGET) L /= 2;
    return L;
}

struct LineGrid {
    long long nblk = 0;  // blocks
    int threads = 0;
    size_t smem = 0;     // dynamic shared memory per block
    bool xline = false;  // the whole-line x kernel runs
};

// Geometry of one sweep along AXIS: fills a.lines, a.ntile_a, a.rt, a.rw.  The
// whole-line x kernel (FLUX along x only) needs one thread per (line, field,
// sub-domain) column.  False if no configuration fits.
template <typename T, int MODE, int AXIS>
bool line_grid(const LineOpDev &op, LineArgs<T> &a, int pref_lines, LineGrid &g)
{
    constexpr bool SINGLE = MODE == MODE_FIELD || MODE == MODE_FIELD2;
    constexpr int NF = SINGLE ? 1 : (MODE == MODE_VGRAD || MODE == MODE_VDIV ? 4 : 5);
    const int kc = sizeof(T) == 8 ? op.kconv64 : op.kconv32;
    g = LineGrid();
    // The whole-line kernel saves the tiles' second reading of end rows, but a
    // warp of its solve costs the same however many of its lanes have a (field,
    // sub-domain) column.  Nx x 96 x 96, ms, tiles and whole lines; columns of
    // the lanes of their warps:
    //   sub-domains of 64: Nx = 512  0.738 0.859 (40 of 64), 768  1.096 1.008 (60 of 64),
    //     832 1.180 1.334 (65 of 96), 1024  1.440 1.551 (80 of 96), 1536  2.143 2.091 (120 of 128)
    //   of 32: 256  0.520 0.539 (40 of 64), 512  1.019 0.948 (80 of 96), 1024  2.022 1.703 (160 of 160)
    //   of 128: 1024  1.310 1.555 (40 of 64)
    // so whole lines where nine lanes in ten work, or four in five with short
    // sub-domains, whose tiles read the most rows twice; not with long ones, nor
    // with fewer than 50 columns (none measured faster).
    const int columns = op.nsub * NF, lanes = (columns + 31) / 32 * 32;
    const bool filled = op.N < 48 * op.nsub ? 5 * columns >= 4 * lanes
                                            : op.N < 96 * op.nsub && 10 * columns >= 9 * lanes;
    if (AXIS == 0 && MODE == MODE_FLUX && columns >= 50 && filled) {
        const size_t bytes = ((size_t)NF * op.xpitch + (size_t)op.ncoef + 2 * (size_t)kc) * sizeof(T);
        if (bytes <= XLINE_SMEM && columns <= 1024) {
            a.lines = 1;
            a.rt = op.xpitch;
            g.threads = lanes < 128 ? 128 : lanes;
            g.smem = bytes;
            g.xline = true;
            g.nblk = (long long)a.n[1] * a.n[2];
            return g.nblk <= 0x7fffffffLL;
        }
    }
    a.rt = op.max_tile;
    a.rw = op.max_win;
    const int rows = (AXIS != 0 || !SINGLE) ? a.rw : a.rt;
    a.lines = pick_lines(pref_lines, rows, NF, sizeof(T));
    const int Na = AXIS == 0 ? a.n[1] : a.n[0];
    const int Nc = AXIS == 2 ? a.n[1] : a.n[2];
    a.ntile_a = (Na + a.lines - 1) / a.lines;
    g.nblk = (long long)op.nsub * a.ntile_a * Nc;
    if (g.nblk > 0x7fffffffLL) return false;
    // extra threads beyond the lines x fields of the solve only stage and
    // store, which keeps more loads in flight per SM (8 per line for the five
    // flux fields, 4 per line for one field: the fastest on GB300)
    int threads = a.lines * NF;
    threads = (threads + 31) / 32 * 32;
    const int per_line = NF == 1 ? 4 : 8;
    if (threads < per_line * a.lines) threads = per_line * a.lines;
    if (threads < 128) threads = 128;
    if (threads > 1024) threads = (a.lines * NF + 31) / 32 * 32;
    if (threads > 1024) return false;
    const int rg = (AXIS != 0 || !SINGLE) ? (AXIS == 0 ? 1 : threads / a.lines) : 0;
    g.threads = threads;
    g.smem = ((size_t)NF * rows * (a.lines + 1) + 2 * (size_t)op.max_taps + 2 * (size_t)kc +
              (size_t)rg * 2 * NF * a.lines) *
             sizeof(T);
    return g.smem <= 227 * 1024;
}

// The whole-line x flux kernel lives in its own translation unit
// (xline_kernels.cu).
template <typename T>
cudaError_t launch_xline_flux(const LineOpDev &op, const LineArgs<T> &a, long long nblk, int threads, size_t smem,
                              cudaStream_t st);
template <typename T>
cudaError_t init_xline_flux();

}  // namespace nopcs
