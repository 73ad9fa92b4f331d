// Viscous terms, gravity source and the classical RK4 stage update, fused in
// one z-marching kernel (arXiv 2203.00879: Eqs. ge6-ge8a, ge19, ge20, bv1-bv3;
// Sec. 4: second-order explicit viscous terms, four-stage RK4).
//
// The viscous right-hand side at a node is the second-order explicit
// divergence of nodal viscous fluxes, and each nodal flux needs second-order
// explicit gradients of u, v, w, T at its node: a +-2 stencil (+-3 next to a
// wall, where both operators are one-sided).  A block owns a TX x TY column
// tile, a thread per node of a plane, and marches along z.  In step j
//   1. E_v, F_v and G_v of plane j are evaluated from one stencil in the ring of
//      primitives (u, v, w, T; four planes with a two-node x/y halo in shared
//      memory, each primitive loaded once per block and plane), E_v also on the
//      x halo and F_v on the y halo; G_v stays in the thread's registers;
//   2. plane j - 1, whose z divergence is now complete, gets the gravity source
//      on top of the convective right-hand side accumulated by the sweeps,
//      zero momentum on wall nodes (no-slip) and the RK4 stage;
//   3. plane j + 2 goes into the ring, and after the step's only barrier
//   4. the x and y divergence of plane j is taken from E_v and F_v in shared
//      memory (two planes, so that the next step can write while others read).
// The loads of steps 2 and 3 are issued before step 1, and L2 is asked for
// those of the next step.
//
// Tiles never start past n - TX, so every tile is at least min(n, TX) wide and
// the one-sided wall stencils stay inside it; a tile that had to be shifted
// back writes only the columns it owns.
//
// Bound by issue slots and latency (stage 2 at 256^3: 56% of the issue slots,
// 568 instructions a node, 57% of the HBM cycles; 24 warps an SM, held by 80
// registers).  Mean over the stages at 1024 x 512 x 512: 6.89 ms (133 B a
// point, 0.76 of the measured copy bandwidth) against 8.04 with a five-plane
// ring, G_v in shared memory and two barriers per plane; at 256^3 0.526
// against 0.594, at 48^3 17 us against 31.  Measured slower: two rows a thread
// in 32 x 16 tiles (128 registers, 16 warps: 431 instructions a node, but 7.58
// ms); four blocks per SM (spills, 12.6); the next plane's inputs copied to
// shared memory with cp.async (9.8: 4-byte copies saturate the memory pipe);
// plane base + 32-bit offset addresses (more instructions).  Stage 4 at 256^3:
// 0.736 ms against 0.827; its binary32/binary64 conversions had been issued to
// the FP64 pipe for every value (49% busy, now 26%).
#include "visc_body.cuh"

namespace nopcs {

namespace {

// S fixes the stage and the gravity axis at compile time (Spec) or leaves
// them to the arguments.
template <typename T, class S>
__global__ void __launch_bounds__(VT, visc_occupancy<T>()) visc_rk_kernel(const __grid_constant__ VArgs<T> a)
{
    extern __shared__ __align__(32) unsigned char smraw[];
    visc_rk_block<T, S>(a, blockIdx.x, blockIdx.y, blockIdx.z, smraw);
}

// Compact viscous terms, step 2 of 3: the nodal viscous fluxes from the
// gradients that the VGRAD sweeps left in G, written over them in place
// (field 4 d + q = d(prim q)/dx_d in, field 4 d + c = component c of the flux
// along d out; a node's twelve values are read before any is written).
template <typename T>
__global__ void __launch_bounds__(256) visc_flux_kernel(const VArgs<T> a, T *__restrict__ G)
{
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const size_t np = (size_t)a.np;
    for (long long q = blockIdx.x * blockDim.x + threadIdx.x; q < a.np; q += gridDim.x * blockDim.x) {
        const int p = (int)q;  // boxes hold < 2^31 points
        T g[3][4];  // g[d][q] = d(prim q)/dx_d, prim = u, v, w, T
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int q = 0; q < 4; ++q) g[d][q] = G[(4 * d + q) * np + p];
        const int x = p % nx, y = (p / nx) % ny, z = p / (nx * ny);
        const int kg = a.ga == 0 ? x : (a.ga == 1 ? y : z);
        const T u = a.W[1][p], v = a.W[2][p], w = a.W[3][p];
        T mu, mub;
        visc_coeffs(a, node_temperature(a, kg, a.W[0][p], a.W[4][p]), mu, mub);
        const T k43 = (T(4) / T(3) * mu + mub) * a.iRe, k23 = (T(-2) / T(3) * mu + mub) * a.iRe, ks = mu * a.iRe;
        // stress tensor, Eqs. ge19, bv1-bv3 (d u_i / d x_j = g[j][i])
        const T txx = k43 * g[0][0] + k23 * (g[1][1] + g[2][2]);
        const T tyy = k43 * g[1][1] + k23 * (g[0][0] + g[2][2]);
        const T tzz = k43 * g[2][2] + k23 * (g[0][0] + g[1][1]);
        const T txy = ks * (g[1][0] + g[0][1]);
        const T txz = ks * (g[2][0] + g[0][2]);
        const T tyz = ks * (g[2][1] + g[1][2]);
        // heat flux, Eq. ge20; its normal component is zero on an adiabatic wall
        const T mk = -mu * a.kq;
        const T qx = (x == 0 || x == nx - 1) ? T(0) : mk * g[0][3];
        const T qy = (y == 0 || y == ny - 1) ? T(0) : mk * g[1][3];
        const T qz = (z == 0 || z == nz - 1) ? T(0) : mk * g[2][3];
        const T f[12] = {txx, txy, txz, u * txx + v * txy + w * txz - qx,
                         txy, tyy, tyz, u * txy + v * tyy + w * tyz - qy,
                         txz, tyz, tzz, u * txz + v * tyz + w * tzz - qz};
#pragma unroll
        for (int k = 0; k < 12; ++k) G[k * np + p] = f[k];
    }
}

// Compact viscous terms, step 3 of 3 (after the VDIV sweeps added the
// divergence into R): gravity source, no-slip walls and the RK stage.
template <typename T>
__global__ void __launch_bounds__(256) source_rk_kernel(const VArgs<T> a)
{
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    for (long long q = blockIdx.x * blockDim.x + threadIdx.x; q < a.np; q += gridDim.x * blockDim.x) {
        const int p = (int)q;  // boxes hold < 2^31 points
        T r[5];
        float kd[5], dn[5];
        double qn[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) r[k] = a.R[k][p];
        if constexpr (sizeof(T) == 4) {
            if (a.stage >= 2) {
#pragma unroll
                for (int k = 0; k < 5; ++k) kd[k] = a.Kacc[k][p];
            }
            if (a.stage >= 1 && a.stage <= 3) {
#pragma unroll
                for (int k = 0; k < 5; ++k) dn[k] = a.Dn[k][p];
            }
            if (a.stage == 4) {
#pragma unroll
                for (int k = 0; k < 5; ++k) qn[k] = a.Qn[k][p];
            }
        }
        const int x = p % nx, y = (p / nx) % ny, z = p / (nx * ny);
        const int kg = a.ga == 0 ? x : (a.ga == 1 ? y : z);
        const bool wall = x == 0 || x == nx - 1 || y == 0 || y == ny - 1 || z == 0 || z == nz - 1;
        source_and_stage(a, p, kg, wall, a.W[0][p], a.W[1 + a.ga][p], r, kd, dn, qn);
    }
}

// pointwise kernels: a grid of 8 blocks of 256 per SM striding over the box
unsigned pointwise_blocks(long long np)
{
    long long b = (np + 255) / 256;
    if (b > 152LL * 8) b = 152LL * 8;
    return (unsigned)(b < 1 ? 1 : b);
}

// The stage kernel for (stage, gravity axis): the FP32 ones are specialised
// per stage, and for gravity along z; the FP64 one is generic.
template <typename T>
const void *visc_kernel_for(int stage, int ga)
{
    if constexpr (sizeof(T) == 4) {
        const bool z = ga == 2;
        switch (stage) {
        case 0: return z ? (const void *)visc_rk_kernel<float, Spec<0, 2>> : (const void *)visc_rk_kernel<float, Spec<0, -1>>;
        case 1: return z ? (const void *)visc_rk_kernel<float, Spec<1, 2>> : (const void *)visc_rk_kernel<float, Spec<1, -1>>;
        case 2: return z ? (const void *)visc_rk_kernel<float, Spec<2, 2>> : (const void *)visc_rk_kernel<float, Spec<2, -1>>;
        case 3: return z ? (const void *)visc_rk_kernel<float, Spec<3, 2>> : (const void *)visc_rk_kernel<float, Spec<3, -1>>;
        default: return z ? (const void *)visc_rk_kernel<float, Spec<4, 2>> : (const void *)visc_rk_kernel<float, Spec<4, -1>>;
        }
    } else {
        return (const void *)visc_rk_kernel<T, RunSpec>;
    }
}

}  // namespace

cudaError_t init_visc_kernels()
{
    for (int ga = 0; ga < 3; ga += 2)
        for (int s = 0; s <= 4; ++s) {
            cudaError_t e = cudaFuncSetAttribute(visc_kernel_for<float>(s, ga),
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)visc_smem<float>());
            if (e != cudaSuccess) return e;
        }
    return cudaFuncSetAttribute(visc_kernel_for<double>(0, 0), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)visc_smem<double>());
}

template <typename T>
cudaError_t launch_visc_update(const BoxDev &bx, const T *W, const T *R, int stage, const StageRegs<T> &g,
                               cudaStream_t st)
{
    VArgs<T> a = make_vargs(bx, W, R, stage, g);
    const dim3 grid = visc_grid<T>(bx, a.zc);
    void *args[] = {&a};
    return cudaLaunchKernel(visc_kernel_for<T>(stage, bx.ga), grid, dim3(VT), args, visc_smem<T>(), st);
}

template <typename T>
cudaError_t launch_visc_flux(const BoxDev &bx, const T *W, T *G, cudaStream_t st)
{
    const VArgs<T> a = make_vargs(bx, W, (const T *)nullptr, 0, StageRegs<T>{});
    visc_flux_kernel<T><<<pointwise_blocks(bx.np), 256, 0, st>>>(a, G);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_source_update(const BoxDev &bx, const T *W, const T *R, int stage, const StageRegs<T> &g,
                                 cudaStream_t st)
{
    const VArgs<T> a = make_vargs(bx, W, R, stage, g);
    source_rk_kernel<T><<<pointwise_blocks(bx.np), 256, 0, st>>>(a);
    return cudaGetLastError();
}

template cudaError_t launch_visc_flux<float>(const BoxDev &, const float *, float *, cudaStream_t);
template cudaError_t launch_visc_flux<double>(const BoxDev &, const double *, double *, cudaStream_t);
template cudaError_t launch_source_update<float>(const BoxDev &, const float *, const float *, int,
                                                 const StageRegs<float> &, cudaStream_t);
template cudaError_t launch_source_update<double>(const BoxDev &, const double *, const double *, int,
                                                  const StageRegs<double> &, cudaStream_t);
template cudaError_t launch_visc_update<float>(const BoxDev &, const float *, const float *, int,
                                              const StageRegs<float> &, cudaStream_t);
template cudaError_t launch_visc_update<double>(const BoxDev &, const double *, const double *, int,
                                               const StageRegs<double> &, cudaStream_t);

}  // namespace nopcs
