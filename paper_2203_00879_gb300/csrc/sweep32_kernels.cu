// Stand-alone launches of the FP32 line sweeps (bodies: sweep32.cuh).
#include <math.h>

#include "sweep32.cuh"

namespace nopcs {

namespace {

template <int MODE, int AXIS, bool GROW, int R, int TPB>
__global__ void __launch_bounds__(TPB) march_kernel(const __grid_constant__ Sweep32Args a)
{
    extern __shared__ __align__(16) float march_sm[];
    march_body<MODE, AXIS, GROW, R, TPB>(a, blockIdx.x, (int)threadIdx.x, march_sm);
}

template <int MODE, bool VEC, bool SHORT>
__global__ void __launch_bounds__(SCAN_WARPS * 32) scan_kernel(const __grid_constant__ Sweep32Args a)
{
    __shared__ __align__(16) float scan_sm[SCAN_WARPS * SweepMode<MODE>::NF * SC_FS];
    const int w = (int)(threadIdx.x >> 5);
    scan_body<MODE, VEC, SHORT>(a, (int)blockIdx.x * SCAN_WARPS + w, scan_sm + w * SweepMode<MODE>::NF * SC_FS);
}

template <int MODE, int AXIS, int R, int TPB>
cudaError_t launch_march_r(const Sweep32Args &a, cudaStream_t st)
{
    const unsigned nblk = (unsigned)((a.cols + TPB - 1) / TPB) * (unsigned)a.nseg;
    constexpr size_t sm = march_smem(SweepMode<MODE>::NF, R, TPB);
    const bool grow = SweepMode<MODE>::NB > 0 && a.ga == AXIS;
    const void *f = grow ? (const void *)march_kernel<MODE, AXIS, SweepMode<MODE>::NB != 0, R, TPB>
                         : (const void *)march_kernel<MODE, AXIS, false, R, TPB>;
    if constexpr (sm > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (e != cudaSuccess) return e;
    }
    void *args[] = {(void *)&a};
    return cudaLaunchKernel(f, dim3(nblk), dim3(TPB), args, sm, st);
}

template <int MODE, int AXIS>
cudaError_t launch_march(const Sweep32Args &a, cudaStream_t st)
{
    if constexpr (SweepMode<MODE>::SINGLE) {
        // 512^3, sub-domains of 64, y and z: 240 and 243 us; a ring of 4 groups
        // 234 and 248, but 48^3 8.3 us instead of 6.5
        return launch_march_r<MODE, AXIS, 8, 64>(a, st);
    } else {
        if (a.ring == 8) return launch_march_r<MODE, AXIS, 8, 32>(a, st);
        return launch_march_r<MODE, AXIS, 4, 64>(a, st);
    }
}

}  // namespace

bool sweep32_operator(const LineOpDev &op, int reach, double scale, Sweep32Args &a)
{
    const double al = op.alpha;
    const double c = al == 0.0 ? 0.0 : (1.0 - sqrt(1.0 - 4.0 * al * al)) / (2.0 * al);
    if (pow(fabs(c), reach) > 1e-8) return false;
    const double inv = 1.0 / (1.0 - al * c);
    a.N = op.N;
    a.c = (float)c;
    a.g1 = (float)(1.0 / (1.0 + c));
    for (int k = 0; k < 4; ++k) a.b[k] = (float)(op.rb[k] * inv * scale);
    double pw = 1.0, cp = 0.0;
    for (int j = 0; j < SC_P; ++j) a.pw[j] = (float)(pw *= -c);
    a.pw16 = (float)(pw * pw);
    for (int k = 0; k < 4; ++k) a.kf[k] = c == 0.0 ? 0.0f : (float)(c * pow(-c, SC_P * k - op.nexp));
    for (int i = 0; i < SW_TAB; ++i) {
        const int r = i - op.nexp;
        const double den = 1.0 - (r > 0 ? al * cp : 0.0);
        cp = r < 0 ? 0.0 : (i == SW_TAB - 1 ? c : al / den);
        a.cp[i] = (float)cp;
        a.rat[i] = r < 0 ? 0.0f : (i == SW_TAB - 1 ? 1.0f : (float)(1.0 / den / inv));
    }
    for (int r = 0; r < 3; ++r)
        for (int j = 0; j < 5; ++j) a.ex[r][j] = (float)(op.ex[r][j] * scale);
    a.exs = (float)op.ex_sign;
    return true;
}

void sweep32_geometry(int axis, const int n[3], Sweep32Args &a)
{
    for (int d = 0; d < 3; ++d) a.n[d] = n[d];
    if (axis == 0) {
        // four points at a time where the lines and every field allow
        // 16-byte accesses
        bool vec = a.N % 4 == 0;
        for (const float *p : a.in) vec = vec && (uintptr_t)p % 16 == 0;
        for (const float *p : a.out) vec = vec && (uintptr_t)p % 16 == 0;
        a.kind = a.N < SC_SHORT ? 0 : (vec ? 2 : 1);
        a.nch = (a.N + SC_P - 1) / SC_P;
        a.tot = a.nch * n[1] * n[2];
        return;
    }
    a.cols = n[0] * n[axis == 1 ? 2 : 1];
    a.srow = axis == 1 ? n[0] : n[0] * n[1];
    a.sc = axis == 1 ? n[0] * n[1] : n[0];
    // A ring of 8 groups runs the backward recurrence over its 24 rows of
    // start-up less often, one of 4 leaves room for twice the threads: while
    // the lines are too few to fill two blocks per SM the longer ring is
    // faster (48^3: y 12.1 against 13.5 us, z 13.0 against 14.4), beyond that
    // the shorter (512^3: 1.36 against 1.41 ms, 1.40 against 1.47).
    a.ring = (a.cols + 31) / 32 < 2 * 152 ? 8 : 4;
    // Segments, of 32 rows at least, while all of them run at once (5 blocks
    // per SM): every further one costs 52 rows of overlap.  201 x 263 x 171,
    // y: one segment 0.134 ms, two 0.155; boxes of 32 to 128 points, z: one
    // 26.4 us, as many as fit 22.2.
    const int tile = a.ring == 8 ? 32 : 64;
    const int nct = (a.cols + tile - 1) / tile;
    const int ns = 152 * 5 / nct > 1 ? 152 * 5 / nct : 1;
    int seg = (a.N + ns - 1) / ns;
    seg = (seg + MR_G - 1) / MR_G * MR_G;
    if (seg < 32) seg = 32;
    a.seg = seg;
    a.nseg = (a.N + seg - 1) / seg;
}

bool flux32_args(const LineOpDev &op, int axis, const BoxDev &bx, const float *W, float *R, Sweep32Args &a)
{
    if (!sweep32_operator(op, sweep_reach(MODE_FLUX), -bx.inv_h[axis], a)) return false;
    for (int k = 0; k < 5; ++k) a.in[k] = W + (size_t)k * bx.np;
    for (int k = 0; k < 5; ++k) a.out[k] = R + (size_t)k * bx.np;
    a.ga = bx.ga;
    a.b0 = bx.rho_b32;
    a.b1 = bx.H_b32;
    a.hp = (float)(bx.gamma / (bx.gamma - 1.0));
    sweep32_geometry(axis, bx.n, a);
    return true;
}

template <int MODE>
cudaError_t launch_sweep32(int axis, const Sweep32Args &a, cudaStream_t st)
{
    switch (axis) {
    case 0: {
        const int per = SC_USE * SCAN_WARPS;
        const unsigned nblk = (unsigned)((a.tot + per - 1) / per);
        switch (a.kind) {
        case 0: scan_kernel<MODE, false, true><<<nblk, SCAN_WARPS * 32, 0, st>>>(a); break;
        case 1: scan_kernel<MODE, false, false><<<nblk, SCAN_WARPS * 32, 0, st>>>(a); break;
        default: scan_kernel<MODE, true, false><<<nblk, SCAN_WARPS * 32, 0, st>>>(a);
        }
        return cudaGetLastError();
    }
    case 1: return launch_march<MODE, 1>(a, st);
    case 2: return launch_march<MODE, 2>(a, st);
    }
    return cudaErrorInvalidValue;
}

template cudaError_t launch_sweep32<MODE_FLUX>(int, const Sweep32Args &, cudaStream_t);
template cudaError_t launch_sweep32<MODE_FIELD>(int, const Sweep32Args &, cudaStream_t);
template cudaError_t launch_sweep32<MODE_FIELD2>(int, const Sweep32Args &, cudaStream_t);
template cudaError_t launch_sweep32<MODE_FILTER>(int, const Sweep32Args &, cudaStream_t);
template cudaError_t launch_sweep32<MODE_VGRAD>(int, const Sweep32Args &, cudaStream_t);
template cudaError_t launch_sweep32<MODE_VDIV>(int, const Sweep32Args &, cudaStream_t);

}  // namespace nopcs
