// Point-wise and stencil kernels of one RK stage (arXiv 2203.00879, Sec. 2 and
// Sec. 4): primitive recovery, the second-order explicit viscous terms with
// bulk viscosity, the gravity source, the classical RK4 stage update in FP64,
// the no-slip adiabatic wall conditions, the initial state and the
// diagnostics reduction.
#include <math.h>

#include "fp_bits.cuh"
#include "wall_body.cuh"

namespace nopcs {

namespace {


__device__ __forceinline__ void coords(const BoxDev &bx, long long p, int c[3])
{
    c[0] = (int)(p % bx.n[0]);
    long long q = p / bx.n[0];
    c[1] = (int)(q % bx.n[1]);
    c[2] = (int)(q / bx.n[1]);
}

// ---------------------------------------------------------------------------
// Primitive recovery (Eqs. ge12, ge13, nondimensional): from the FP64 state to
// W = (rho - rho_b, u, v, w, p - p_b, E + p - H_b) in the compute precision,
// with (rho_b, p_b, H_b) the hydrostatic base in the base-subtracted form and
// zero in the plain form.  The mixed form takes the two large differences
// rho - rho_b and E - E_b in FP64 and the rest in FP32, using
// p - p_b = (gamma - 1)(E - E_b - rho |V|^2 / 2); it keeps the first five.
// ---------------------------------------------------------------------------
// The base state at gravity coordinate kg (mixed form), read where it is used, or
// ahead, with a point's other loads: the integer conversions branch, and no load
// moves across a branch (filter of 64 x 64 x 2048: 830 us with the base read where it
// is used, 622 ahead; of no use to rows that fill their blocks).
struct BaseAt {
    const BoxDev &bx;
    int kg;
    __device__ __forceinline__ double rho() const { return bx.rho_b64[kg]; }
    __device__ __forceinline__ double E() const { return bx.E_b64[kg]; }
    __device__ __forceinline__ float rho32() const { return bx.rho_b32[kg]; }
};
struct BaseAhead {
    double r, e;
    float r32;
    __device__ __forceinline__ BaseAhead(const BoxDev &bx, int kg)
        : r(bx.rho_b64[kg]), e(bx.E_b64[kg]), r32(bx.rho_b32[kg])
    {
    }
    __device__ __forceinline__ double rho() const { return r; }
    __device__ __forceinline__ double E() const { return e; }
    __device__ __forceinline__ float rho32() const { return r32; }
};

// W (and the deviation D_n, mixed form) of one point of the FP64 state.  CVT:
// hardware conversions to binary32 (the same results).
template <typename T, bool CVT, class Base>
__device__ __forceinline__ void prep_point(const BoxDev &bx, long long p, int kg, const Base &b, double r, double mx,
                                           double my, double mz, double E, T *__restrict__ W, float *__restrict__ Dn)
{
    const long long np = bx.np;
    if constexpr (sizeof(T) == 8) {
        const double u = mx / r, v = my / r, w = mz / r;
        const double pr = (bx.gamma - 1.0) * (E - 0.5 * (mx * u + my * v + mz * w));
        W[p] = r - bx.rho_b64[kg];
        W[np + p] = u;
        W[2 * np + p] = v;
        W[3 * np + p] = w;
        W[4 * np + p] = pr - bx.p_b64[kg];
        W[5 * np + p] = E + pr - bx.H_b64[kg];
    } else {
        // deviation of the state from the hydrostatic base (mixed form), then
        // the primitives from it exactly as the stage kernels form them
        auto f32 = [](double d) { return CVT ? (float)d : narrow_f64(d); };
        const float D[5] = {f32(r - b.rho()), f32(mx), f32(my), f32(mz), f32(E - b.E())};
        float Wv[5];
        prim_from_deviation(b.rho32(), (float)(bx.gamma - 1.0), D, Wv);
#pragma unroll
        for (int k = 0; k < 5; ++k) W[k * np + p] = Wv[k];
        if (Dn) {
#pragma unroll
            for (int k = 0; k < 5; ++k) Dn[k * np + p] = D[k];
        }
    }
}

// grid-stride over (y, z) rows, threads along x: no 64-bit division per point.
// Mixed form: hardware conversions (CVT) for rows of up to 64 points, which leave
// most of a block's threads idle, and for fewer rows than SMs: there the latency of
// a row counts and not the FP64 pipe.  set_state, us, hardware and integer
// conversions: 9 x 400 x 400 165 and 192, 64 x 256 x 256 141 and 150, 96 189 and 187, 128
// 236 and 226, 192 331 and 320, 321 x 257 x 203 550 and 525; 4000 x 5 x 5 30 and 35.
constexpr int PREP_SHORT = 64, PREP_ROWS = 152;
template <typename T, bool CVT>
__global__ void prep_kernel(const BoxDev bx, const double *__restrict__ Q, T *__restrict__ W,
                            float *__restrict__ Dn)
{
    const long long np = bx.np;
    const int nx = bx.n[0], ny = bx.n[1], rows = bx.n[1] * bx.n[2];
    for (int rw = blockIdx.x; rw < rows; rw += gridDim.x) {
        const int y = rw % ny, z = rw / ny;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            const long long p = (long long)rw * nx + x;
            const int kg = bx.ga == 0 ? x : (bx.ga == 1 ? y : z);
            prep_point<T, CVT>(bx, p, kg, BaseAt{bx, kg}, Q[p], Q[np + p], Q[2 * np + p], Q[3 * np + p], Q[4 * np + p], W, Dn);
        }
    }
}

// Mixed-form filter (Sec. 4): the FP32 deviation D_n was filtered into Fd;
// the state takes the change Fd - D_n in FP64, so its low-order bits survive,
// and W0 and D_n are recomputed from the new state.  A point's fifteen loads are
// issued before the first conversion, whose branch loads do not move across.
__global__ void filter_update_kernel(const BoxDev bx, double *__restrict__ Q, const float *__restrict__ Fd,
                                     float *__restrict__ W, float *__restrict__ Dn)
{
    const long long np = bx.np;
    const int nx = bx.n[0], ny = bx.n[1], rows = bx.n[1] * bx.n[2];
    for (int rw = blockIdx.x; rw < rows; rw += gridDim.x) {
        const int y = rw % ny, z = rw / ny;
        for (int x = threadIdx.x; x < nx; x += blockDim.x) {
            const long long p = (long long)rw * nx + x;
            const int kg = bx.ga == 0 ? x : (bx.ga == 1 ? y : z);
            const BaseAhead b(bx, kg);
            double q[5];
            float fd[5], dn[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) q[k] = Q[k * np + p], fd[k] = Fd[k * np + p], dn[k] = Dn[k * np + p];
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                q[k] += widen_f32(fd[k] - dn[k]);
                Q[k * np + p] = q[k];
            }
            prep_point<float, false>(bx, p, kg, b, q[0], q[1], q[2], q[3], q[4], W, Dn);
        }
    }
}

__global__ void wall_kernel(const BoxDev bx, double *Q, float *Dn, float *Wf, float *Ww)
{
    if (blockIdx.x == 0) {
        corner_block(bx, threadIdx.x, Q, Dn, Wf, Ww);
        return;
    }
    const unsigned tot = wall_count(bx);
    for (unsigned t = (blockIdx.x - 1) * blockDim.x + threadIdx.x; t < tot; t += (gridDim.x - 1) * blockDim.x)
        wall_node(bx, t, Q, Dn, Wf, Ww);
}

// ---------------------------------------------------------------------------
// Initial state (Sec. 2, Fig. 1): quiescent hydrostatic two-temperature box
// plus a uniform velocity perturbation from SplitMix64 (Steele, Lea & Flood,
// 2014) used as a counter-based generator, value 3 p + component.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long splitmix64_at(unsigned long long seed, unsigned long long c)
{
    unsigned long long z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__global__ void initial_state_kernel(const BoxDev bx, unsigned long long seed, double amp, double *Q)
{
    const long long np = bx.np;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < np;
         p += (long long)gridDim.x * blockDim.x) {
        int c[3];
        coords(bx, p, c);
        const int kg = c[bx.ga];
        const double rho = bx.rho_h64[kg], pr = bx.p_h64[kg];
        double V[3] = {0.0, 0.0, 0.0};
        const bool wall = c[0] == 0 || c[0] == bx.n[0] - 1 || c[1] == 0 || c[1] == bx.n[1] - 1 || c[2] == 0 ||
                          c[2] == bx.n[2] - 1;
        if (!wall && amp != 0.0) {
            for (int k = 0; k < 3; ++k) {
                const unsigned long long z = splitmix64_at(seed, 3ull * (unsigned long long)p + k);
                const double U = (double)(z >> 11) * (1.0 / 9007199254740992.0);
                V[k] = amp * (2.0 * U - 1.0);
            }
        }
        Q[p] = rho;
        Q[np + p] = rho * V[0];
        Q[2 * np + p] = rho * V[1];
        Q[3 * np + p] = rho * V[2];
        Q[4 * np + p] = pr / (bx.gamma - 1.0) + 0.5 * rho * (V[0] * V[0] + V[1] * V[1] + V[2] * V[2]);
    }
}

// ---------------------------------------------------------------------------
// Diagnostics: per-block partials (fixed grid, fixed order), then one block.
// partial record: mass, mx, my, mz, energy, max|V|^2, max|dp|, max Mach^2, bad
// ---------------------------------------------------------------------------
constexpr int DIAG_THREADS = 256;
constexpr int DIAG_REC = 10;

// BLOCKS: blocks per SM it is compiled for.  A row keeps nx of a block's threads
// busy, so short rows want four blocks (64 registers); long ones run faster with
// the 72 registers the compiler takes for three.  After eight steps, us, three
// and four blocks: 9 x 400 x 400 675 and 492, 101 x 1001 x 51 328 and 279,
// 128 x 256 x 256 416 and 342, 160 431 and 408, 192 480 and 479, 224 508 and 551,
// 256 553 and 623: four up to 160 points.
constexpr int DIAG_SHORT = 160;
template <int BLOCKS>
__global__ void __launch_bounds__(DIAG_THREADS, BLOCKS)
diag_partial_kernel(const BoxDev bx, const double *__restrict__ Q, double *partial, uint4 *seen)
{
    __shared__ double sh[DIAG_REC][DIAG_THREADS];
    const long long np = bx.np;
    const int nx = bx.n[0], ny = bx.n[1], rows = bx.n[1] * bx.n[2];
    const double gm1 = bx.gamma - 1.0, igam = 1.0 / bx.gamma;
    // maxima of |V|^2 and Mach^2 are kept and their square roots taken once
    // in the final kernel (the square root is monotone).  The FP64 work per
    // point is what decides this kernel's time (GB300 runs FP64 at 1/64 of the
    // FP32 rate): the sums are FP64 at every point; the maxima are evaluated
    // in FP64 (1/rho by two Newton steps instead of a division, the Mach^2
    // division only where it can raise the maximum) only at the points that a
    // binary32 screen cannot rule out; the gravity-axis terms are taken once
    // per row where gravity is not along x.
    double v[DIAG_REC] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    double v7t = 0.0;  // v[7] * 0.999999
    // FP32 screen for the maxima: a point goes through the FP64 evaluation
    // below only if its binary32 estimates, with margins well above their
    // rounding error, could reach the current maxima (or are not numbers);
    // the maxima are those of the FP64 values of the points that could raise
    // them, so they are the same as evaluating every point in FP64.  The
    // thresholds are those of all warps (seen, zero at launch): a warp evaluates
    // when any lane passes, so lanes each finding maxima of their own kept it
    // evaluating nearly every point of boxes up to 256^3 (1.49 ms there after
    // eight steps, 0.55 now).  A warp that has points reads them once a row, with
    // one load that is in flight with the row's own: every warp reads the same
    // line, L2 serves 2.7 such reads a ns, and three loads a row by every warp
    // took longer than short rows themselves (9 x 400 x 400: 1.11 ms, 0.49 now;
    // 0.75 with thresholds of each thread)
    float v5f = 0.0f, v6f = 0.0f, v7f = 0.0f;
    bool screening = true;
    int nseen = 0, ncand = 0;
    const float gm1f = (float)gm1, igamf = (float)igam;
    for (int rw = (int)(threadIdx.x & ~31u) < nx ? blockIdx.x : rows; rw < rows; rw += gridDim.x) {
        const uint4 all = __ldcg(seen);
        const int y = rw % ny, z = rw / ny;
        const long long base = (long long)rw * nx;
        // coordinate along gravity of the row (gravity along y or z)
        const int kr = bx.ga == 1 ? y : z;
        const double kgh_r = kr * bx.h[bx.ga];
        const double ph_r = bx.ga != 0 ? bx.p_h64[kr] : 0.0;
        // screen of |p - p_h|: p - p_h = (gamma - 1)(E - E_b - kinetic) + c
        // with c = (gamma - 1) E_b - p_h, so that the binary32 estimate resolves
        // disturbances far smaller than p itself
        const double Eb_r = bx.ga != 0 && bx.E_b64 ? bx.E_b64[kr] : 0.0;
        const float cf_r = narrow_f64(gm1 * Eb_r - ph_r);
        for (int xw = threadIdx.x & ~31; xw < nx; xw += blockDim.x) {
            const int x = xw + (int)(threadIdx.x & 31);
            bool cand = false, rise = false;
            float n5f = 0.0f, n6f = 0.0f, n7f = 0.0f;
            if (x < nx) {
                const long long p = base + x;
                const double kgh = bx.ga == 0 ? x * bx.h[0] : kgh_r;
                const double ph = bx.ga == 0 ? bx.p_h64[x] : ph_r;
                const double r = Q[p], mx = Q[np + p], my = Q[2 * np + p], mz = Q[3 * np + p], E = Q[4 * np + p];
                // not finite: exponent field all ones (infinity or NaN), tested on
                // the high words by integer operations instead of FP64 compares
                auto nonfinite = [](double q) { return ((unsigned)__double2hiint(q) & 0x7ff00000u) == 0x7ff00000u; };
                const bool bad = nonfinite(r) || nonfinite(mx) || nonfinite(my) || nonfinite(mz) || nonfinite(E);
                if (bad) v[8] = 1.0;
                v[0] += r;
                v[1] += mx;
                v[2] += my;
                v[3] += mz;
                v[4] += E + r * bx.g * kgh;
                // screen: |V|^2 to ~1e-6 relative; p to tol absolute (a few
                // binary32 ulps of |E| + |kinetic| + |p_h|, with room to spare),
                // so Mach^2 only where p is known to 1e-4 relative
                cand = true;
                v5f = fmaxf(v5f, __uint_as_float(all.x));
                v6f = fmaxf(v6f, __uint_as_float(all.y));
                v7f = fmaxf(v7f, __uint_as_float(all.z));
                if (screening) {
                    const double Eb = bx.ga == 0 ? (bx.E_b64 ? bx.E_b64[x] : 0.0) : Eb_r;
                    const float cf = bx.ga == 0 ? narrow_f64(gm1 * Eb - ph) : cf_r;
                    const float rf = narrow_f64(r), mxf = narrow_f64(mx), myf = narrow_f64(my), mzf = narrow_f64(mz);
                    const float Ef = narrow_f64(E), phf = narrow_f64(ph), dEf = narrow_f64(E - Eb);
                    const float irf = __fdividef(1.0f, rf);
                    const float s2f = (mxf * mxf + myf * myf + mzf * mzf) * (irf * irf);
                    const float kinf = 0.5f * rf * s2f;
                    const float prf = gm1f * (Ef - kinf);
                    const float tol = 2e-6f * (fabsf(Ef) + fabsf(kinf) + fabsf(phf));
                    // the disturbance pressure to 2e-6 of its own terms, plus 1e-14
                    // of E and p_h for the rounding of the FP64 evaluation it
                    // stands for
                    const float dpf = fabsf(gm1f * (dEf - kinf) + cf);
                    const float tol_dp =
                        2e-6f * (fabsf(dEf) + fabsf(kinf) + fabsf(cf)) + 1e-14f * (fabsf(Ef) + fabsf(phf));
                    const float machf = __fdividef(s2f * rf * igamf, prf);
                    cand = !(s2f < v5f) || !(dpf + tol_dp < v6f) || !(fabsf(prf) > 1e4f * tol) ||
                           !(machf * 1.0003f < v7f);
                    // a state whose maxima sit at the FP64 rounding floor (a box at
                    // rest) passes every point: the thread then stops screening
                    ncand += cand ? 1 : 0;
                    if (++nseen == 256) screening = 2 * ncand < nseen;
                }
                if (cand) {
                    const double ir = recip_newton(r);
                    const double u = mx * ir, vv = my * ir, w = mz * ir;
                    const double s2 = u * u + vv * vv + w * w;
                    const double pr = gm1 * (E - 0.5 * r * s2);
                    v[5] = fmax(v[5], s2);
                    v[6] = fmax(v[6], fabs(pr - ph));
                    // Mach^2 = num / pr can raise the maximum only where num
                    // exceeds v7 pr (for pr > 0; the factor 0.999999 keeps every
                    // point whose rounded quotient could exceed v7).  Elsewhere the
                    // quotient is at most v7, or not a number, and the maximum
                    // stays as it is.
                    const double num = s2 * r * igam;
                    if (num > v7t * pr) {
                        v[7] = fmax(v[7], num / pr);
                        v7t = v[7] * 0.999999;
                    }
                    // thresholds a little below the maxima; none while a maximum
                    // is too small for the binary32 estimates to resolve
                    const float m5 = narrow_f64(v[5]), m7 = narrow_f64(v[7]);
                    n5f = m5 > 1e-30f ? m5 * 0.99999f : 0.0f;
                    n6f = narrow_f64(v[6]) * 0.99999f;
                    n7f = m7 > 1e-30f ? m7 * 0.9999f : 0.0f;
                    rise = n5f > v5f || n6f > v6f || n7f > v7f;
                }
            }
            if (__any_sync(0xffffffffu, rise)) {
                // those of the warp (not negative, so their bit patterns are
                // ordered as the values are)
                auto raise = [&](float &t, float f, unsigned *to) {
                    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(f));
                    if (__uint_as_float(m) > t) {
                        t = __uint_as_float(m);
                        if ((threadIdx.x & 31) == 0) atomicMax(to, m);
                    }
                };
                raise(v5f, n5f, &seen->x);
                raise(v6f, n6f, &seen->y);
                raise(v7f, n7f, &seen->z);
            }
        }
    }
    for (int k = 0; k < DIAG_REC; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = DIAG_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
            for (int k = 5; k < 9; ++k) sh[k][threadIdx.x] = fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x < DIAG_REC) partial[(size_t)blockIdx.x * DIAG_REC + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void diag_final_kernel(const BoxDev bx, const double *partial, int nblk, double *out)
{
    // one block: each thread folds a fixed stride of partial records, then a
    // fixed-shape tree; the reduction order never changes between calls
    __shared__ double sh[DIAG_REC][DIAG_THREADS];
    double v[DIAG_REC] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) {
        const double *q = partial + (size_t)b * DIAG_REC;
        for (int k = 0; k < 5; ++k) v[k] += q[k];
        for (int k = 5; k < 9; ++k) v[k] = fmax(v[k], q[k]);
    }
    for (int k = 0; k < DIAG_REC; ++k) sh[k][threadIdx.x] = v[k];
    __syncthreads();
    for (int w = DIAG_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            for (int k = 0; k < 5; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
            for (int k = 5; k < 9; ++k) sh[k][threadIdx.x] = fmax(sh[k][threadIdx.x], sh[k][threadIdx.x + w]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double dV = bx.h[0] * bx.h[1] * bx.h[2];
        for (int k = 0; k < 5; ++k) out[k] = sh[k][0] * dV;
        out[5] = sqrt(sh[5][0]);
        out[6] = sh[6][0];
        out[7] = sqrt(sh[7][0]);
        out[8] = sh[8][0];
        out[9] = 0.0;
    }
}

int grid_for(long long work, int threads)
{
    long long b = (work + threads - 1) / threads;
    const long long cap = 152LL * 16;  // grid-stride beyond 16 blocks per SM
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

static int row_grid(const BoxDev &bx)
{
    const int rows = bx.n[1] * bx.n[2];
    return rows < 152 * 16 ? rows : 152 * 16;
}

template <typename T>
cudaError_t launch_prep(const BoxDev &bx, const double *Q, T *W, float *Dn, cudaStream_t st)
{
    if (sizeof(T) == 4 && (bx.n[0] <= PREP_SHORT || bx.n[1] * bx.n[2] < PREP_ROWS))
        prep_kernel<T, sizeof(T) == 4><<<row_grid(bx), 256, 0, st>>>(bx, Q, W, Dn);
    else
        prep_kernel<T, false><<<row_grid(bx), 256, 0, st>>>(bx, Q, W, Dn);
    return cudaGetLastError();
}

cudaError_t launch_filter_update(const BoxDev &bx, double *Q, const float *Fd, float *W, float *Dn, cudaStream_t st)
{
    filter_update_kernel<<<row_grid(bx), 256, 0, st>>>(bx, Q, Fd, W, Dn);
    return cudaGetLastError();
}

cudaError_t launch_wall_bc(const BoxDev &bx, double *Q, float *Dn, float *Wf, float *Ww, cudaStream_t st)
{
    wall_kernel<<<1 + grid_for(wall_count(bx), 128), 128, 0, st>>>(bx, Q, Dn, Wf, Ww);
    return cudaGetLastError();
}

cudaError_t launch_initial_state(const BoxDev &bx, unsigned long long seed, double amp, double *Q,
                                 cudaStream_t st)
{
    initial_state_kernel<<<grid_for(bx.np, 256), 256, 0, st>>>(bx, seed, amp, Q);
    return cudaGetLastError();
}

int diag_blocks(long long np)
{
    (void)np;
    return 152 * 8;  // grid-stride over (y, z) rows: 8 blocks per SM
}

cudaError_t launch_diagnostics(const BoxDev &bx, const double *Q, double *partial, int nblk, double *out,
                               cudaStream_t st)
{
    // the warps' common thresholds, after the partial records and the result
    // (16-byte aligned: an even number of doubles from the allocation's start)
    uint4 *seen = reinterpret_cast<uint4 *>(partial + (size_t)nblk * DIAG_REC + 10);
    cudaError_t e = cudaMemsetAsync(seen, 0, sizeof(uint4), st);
    if (e != cudaSuccess) return e;
    if (bx.n[0] <= DIAG_SHORT)
        diag_partial_kernel<4><<<nblk, DIAG_THREADS, 0, st>>>(bx, Q, partial, seen);
    else
        diag_partial_kernel<3><<<nblk, DIAG_THREADS, 0, st>>>(bx, Q, partial, seen);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    diag_final_kernel<<<1, DIAG_THREADS, 0, st>>>(bx, partial, nblk, out);
    return cudaGetLastError();
}

template cudaError_t launch_prep<float>(const BoxDev &, const double *, float *, float *, cudaStream_t);
template cudaError_t launch_prep<double>(const BoxDev &, const double *, double *, float *, cudaStream_t);
}  // namespace nopcs
