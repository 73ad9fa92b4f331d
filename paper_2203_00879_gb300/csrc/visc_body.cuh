// Device body of the fused viscous / source / RK stage kernel (arXiv
// 2203.00879: Eqs. ge6-ge8a, ge19, ge20, bv1-bv3; Sec. 4), one block given as
// (bx, by, bz), with its argument block (VArgs, make_vargs) and shared-memory
// size, so that the stand-alone kernel (visc_kernel.cu) and the batched
// persistent kernel (batch_kernel.cu) run the same code.  The header comment of
// visc_kernel.cu describes the algorithm.
#pragma once

#include <math.h>

#include "fp_bits.cuh"
#include "nopcs_internal.cuh"

namespace nopcs {

namespace {

// A block's tile: TX x TY nodes of a plane, one thread each, in a ring of
// planes with a two-node halo.
constexpr int TX = 32, TY = 8, HALO = 2, VT = TX * TY;
constexpr int PX = TX + 2 * HALO, PY = TY + 2 * HALO, PLANE = PX * PY;
constexpr int RING = 4;                 // planes in the ring
constexpr int PN = (PLANE + VT - 1) / VT;  // ring nodes of a thread
// resident blocks per SM the kernels are compiled for
template <typename T>
constexpr int visc_occupancy() { return sizeof(T) == 4 ? 3 : 1; }

// Every field array is passed as its own base pointer, so a node's address is
// one 32-bit index away from a kernel parameter (boxes hold < 2^31 points).
template <typename T>
struct VArgs {
    int n[3];
    int np;
    T ih2[3];             // 1 / (2 h)
    int ga, zc;           // gravity axis, planes per block
    T gm2, iRe, kq, S1, S, c0, c1, g;
    const T *W[5];
    const T *rho_b, *p_b;                 // base tables (zeros in the plain form)
    const float *T_b, *ip_b, *ir_b;       // mixed form: T_b, 1/p_b, 1/rho_b
    const T *R[5];
    int stage;
    double dt;
    double dt6, dt3, dt2;                 // dt/6, dt/3, dt/2 (host-computed: no FP64 division per node)
    float cdt2, cdt1;                     // FP32 dt/2 and dt (mixed-form stage states)
    T *Rout[5];                           // stage 0: right-hand side out
    double *Qn[5], *acc[5], *Qout[5];     // FP64 stage registers
    float *Kacc[5], *Dn[5];               // mixed form: slope sum, deviation of Q_n
    T *Wn[5];                             // mixed form: next stage's W
    const double *rho_b64, *E_b64;        // mixed form: base state for the deviation of Q_n
    float gm1;                            // gamma - 1
};

// Compile-time specialisation of the stage kernel: the RK stage (0..4) and
// the gravity axis (0..2) fixed at compile time, or -1 to take them from the
// arguments at run time.  The benchmark's stages run specialised: no per-node
// tests of the stage or the gravity axis, and no dead code of other stages.
template <int STAGE, int GA>
struct Spec {
    static constexpr int stage_c = STAGE, ga_c = GA;
};
using RunSpec = Spec<-1, -1>;
template <class S, typename A>
__device__ __forceinline__ int st_of(const A &a)
{
    return S::stage_c >= 0 ? S::stage_c : a.stage;
}
template <class S, typename A>
__device__ __forceinline__ int ga_of(const A &a)
{
    return S::ga_c >= 0 ? S::ga_c : a.ga;
}

// T = gamma M^2 p / rho of a stage state from its primitives W0 = rho - rho_b
// and W4 = p - p_b at gravity coordinate kg (FP32: T_b (1 + p'/p_b) /
// (1 + rho'/rho_b), which keeps the deviations' digits)
template <typename T>
__device__ __forceinline__ T node_temperature(const VArgs<T> &a, int kg, T w0, T w4)
{
    if constexpr (sizeof(T) == 4) {
        // fixed-order arithmetic, like the fluxes: every kernel that forms a
        // node's temperature gets the same bits
        const float rr = __fmul_rn(w0, a.ir_b[kg]);
        return __fadd_rn(a.T_b[kg], __fdividef(__fmul_rn(a.T_b[kg], __fmaf_rn(w4, a.ip_b[kg], -rr)),
                                               __fadd_rn(1.0f, rr)));
    } else {
        return a.gm2 * (a.p_b[kg] + w4) / (a.rho_b[kg] + w0);
    }
}

// ---- four ring fields per node ------------------------------------------------
// A ring node holds (u, v, w, T) as one 16-byte (FP32) or 32-byte (FP64)
// vector, so the gradient of all four fields along an axis is two vector
// loads; the FP32 arithmetic on such vectors runs as packed FP32x2 operations.
struct alignas(32) dbl4 {
    double x, y, z, w;
};
template <typename T>
struct V4T;
template <>
struct V4T<float> {
    using type = float4;
};
template <>
struct V4T<double> {
    using type = dbl4;
};
template <typename T>
using V4 = typename V4T<T>::type;

// Scalar arithmetic in a fixed order (no contraction into FMAs the compiler
// might choose differently in different places): a flux evaluated at the same
// node from the same inputs gives the same bits in every block that needs it.
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

__device__ __forceinline__ float2 lo2(const float4 &a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ float2 hi2(const float4 &a) { return make_float2(a.z, a.w); }
__device__ __forceinline__ float4 cat4(float2 l, float2 h) { return make_float4(l.x, l.y, h.x, h.y); }

// a - b (as fma(b, -1, a): one rounding, the same as a subtraction)
__device__ __forceinline__ float4 v_sub(const float4 &a, const float4 &b)
{
    const float2 m1 = make_float2(-1.0f, -1.0f);
    return cat4(__ffma2_rn(lo2(b), m1, lo2(a)), __ffma2_rn(hi2(b), m1, hi2(a)));
}
__device__ __forceinline__ float4 v_add(const float4 &a, const float4 &b)
{
    return cat4(__fadd2_rn(lo2(a), lo2(b)), __fadd2_rn(hi2(a), hi2(b)));
}
__device__ __forceinline__ float4 v_mul(const float4 &a, float s)
{
    const float2 s2 = make_float2(s, s);
    return cat4(__fmul2_rn(lo2(a), s2), __fmul2_rn(hi2(a), s2));
}
// a s + c
__device__ __forceinline__ float4 v_fma(const float4 &a, float s, const float4 &c)
{
    const float2 s2 = make_float2(s, s);
    return cat4(__ffma2_rn(lo2(a), s2, lo2(c)), __ffma2_rn(hi2(a), s2, hi2(c)));
}
__device__ __forceinline__ dbl4 v_sub(const dbl4 &a, const dbl4 &b)
{
    return dbl4{__dadd_rn(a.x, -b.x), __dadd_rn(a.y, -b.y), __dadd_rn(a.z, -b.z), __dadd_rn(a.w, -b.w)};
}
__device__ __forceinline__ dbl4 v_add(const dbl4 &a, const dbl4 &b)
{
    return dbl4{__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y), __dadd_rn(a.z, b.z), __dadd_rn(a.w, b.w)};
}
__device__ __forceinline__ dbl4 v_mul(const dbl4 &a, double s)
{
    return dbl4{__dmul_rn(a.x, s), __dmul_rn(a.y, s), __dmul_rn(a.z, s), __dmul_rn(a.w, s)};
}
__device__ __forceinline__ dbl4 v_fma(const dbl4 &a, double s, const dbl4 &c)
{
    return dbl4{__fma_rn(a.x, s, c.x), __fma_rn(a.y, s, c.y), __fma_rn(a.z, s, c.z), __fma_rn(a.w, s, c.w)};
}

// second-order differences of a ring vector: central (p+ - p-) / (2h) and the
// one-sided (-3 p0 + 4 p1 - p2) / (2h) at a low wall, (3 p0 - 4 p-1 + p-2) /
// (2h) at a high wall (ih = 1 / (2h))
template <typename V, typename T>
__device__ __forceinline__ V d_central(const V &pp, const V &pm, T ih)
{
    return v_mul(v_sub(pp, pm), ih);
}
template <typename V, typename T>
__device__ __forceinline__ V d_low(const V &p0, const V &p1, const V &p2, T ih)
{
    return v_mul(v_sub(v_fma(p1, T(4), v_mul(p0, T(-3))), p2), ih);
}
template <typename V, typename T>
__device__ __forceinline__ V d_high(const V &p0, const V &pm1, const V &pm2, T ih)
{
    return v_mul(v_add(v_fma(pm1, T(-4), v_mul(p0, T(3))), pm2), ih);
}

// Ask L2 for data that a load will need a plane later: it takes the HBM latency
// off the load and, unlike a load, holds no register.
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// The ring nodes of a thread: node t is ring node threadIdx.x + t VT, read from
// element goff of a plane (a node outside the box stands for the nearest one
// inside: it is in no stencil).
template <typename T, class S>
struct RingNodes {
    int goff[PN], kgxy[PN];
    T w[PN][5];
    __device__ __forceinline__ void init(const VArgs<T> &a, int x0, int y0)
    {
#pragma unroll
        for (int t = 0; t < PN; ++t) {
            const int idx = min((int)threadIdx.x + t * VT, PLANE - 1);
            const int gx = min(max(x0 - HALO + idx % PX, 0), a.n[0] - 1);
            const int gy = min(max(y0 - HALO + idx / PX, 0), a.n[1] - 1);
            goff[t] = gx + a.n[0] * gy;
            kgxy[t] = ga_of<S>(a) == 0 ? gx : gy;
        }
    }
    __device__ __forceinline__ void put(const VArgs<T> &a, V4<T> *ring, int z, int t, const T q[5]) const
    {
        const int idx = (int)threadIdx.x + t * VT;
        if ((t + 1) * VT > PLANE && idx >= PLANE) return;
        const int kg = ga_of<S>(a) == 2 ? z : kgxy[t];
        ring[(z & (RING - 1)) * PLANE + idx] = V4<T>{q[1], q[2], q[3], node_temperature(a, kg, q[0], q[4])};
    }
    // planes z .. z + NP - 1 straight into the ring, all loads at once
    template <int NP>
    __device__ __forceinline__ void load(const VArgs<T> &a, V4<T> *ring, int z) const
    {
        const int nxy = a.n[0] * a.n[1];
        T q[NP][PN][5];
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int t = 0; t < PN; ++t)
#pragma unroll
                for (int k = 0; k < 5; ++k) q[i][t][k] = a.W[k][nxy * (z + i) + goff[t]];
#pragma unroll
        for (int i = 0; i < NP; ++i)
#pragma unroll
            for (int t = 0; t < PN; ++t) put(a, ring, z + i, t, q[i][t]);
    }
    // the same for one plane in two halves, so that the loads are in flight
    // while the thread does other work
    __device__ __forceinline__ void issue(const VArgs<T> &a, int z)
    {
        const int zo = a.n[0] * a.n[1] * z;
#pragma unroll
        for (int t = 0; t < PN; ++t)
#pragma unroll
            for (int k = 0; k < 5; ++k) w[t][k] = a.W[k][zo + goff[t]];
    }
    __device__ __forceinline__ void settle(const VArgs<T> &a, V4<T> *ring, int z) const
    {
#pragma unroll
        for (int t = 0; t < PN; ++t) put(a, ring, z, t, w[t]);
    }
    __device__ __forceinline__ void prefetch(const VArgs<T> &a, int z) const
    {
        const int zo = a.n[0] * a.n[1] * z;
#pragma unroll
        for (int t = 0; t < PN; ++t) {
            if ((t + 1) * VT > PLANE && (int)threadIdx.x + t * VT >= PLANE) continue;
#pragma unroll
            for (int k = 0; k < 5; ++k) prefetch_l2(a.W[k] + zo + goff[t]);
        }
    }
};

// The inputs of a node's RK update: right-hand side, rho - rho_b and (mixed
// form) K, D_n and Q_n, as far as the stage reads them.
template <typename T, class S>
struct UpdateIn {
    T r[5], w0;
    float kd[5], dn[5];
    double qn[5];
    static constexpr bool MIXED = sizeof(T) == 4;
    static __device__ __forceinline__ bool has_k(int stage) { return MIXED && stage >= 2; }
    static __device__ __forceinline__ bool has_d(int stage) { return MIXED && stage >= 1 && stage <= 3; }
    static __device__ __forceinline__ bool has_q(int stage) { return MIXED && stage == 4; }
    __device__ __forceinline__ void load(const VArgs<T> &a, int p)
    {
        const int stage = st_of<S>(a);
#pragma unroll
        for (int k = 0; k < 5; ++k) r[k] = a.R[k][p];
        w0 = a.W[0][p];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            if (has_k(stage)) kd[k] = a.Kacc[k][p];
            if (has_d(stage)) dn[k] = a.Dn[k][p];
            if (has_q(stage)) qn[k] = a.Qn[k][p];
        }
    }
    static __device__ __forceinline__ void prefetch(const VArgs<T> &a, int p)
    {
        const int stage = st_of<S>(a);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            prefetch_l2(a.R[k] + p);
            if (has_k(stage)) prefetch_l2(a.Kacc[k] + p);
            if (has_d(stage)) prefetch_l2(a.Dn[k] + p);
            if (has_q(stage)) prefetch_l2(a.Qn[k] + p);
        }
    }
};

// Second-order explicit derivatives of (u, v, w, T) at one node of the ring:
// central inside, one-sided (-3, 4, -1)/(2h) on a wall.  mode 0: central, 1:
// low wall (forward), 2: high wall (backward).  EDGE is false for blocks whose
// nodes are all at least one node away from the x and y walls, so only the z
// mode (uniform over a plane) is tested there.  (Planes j - 2 and j + 2 share a
// ring slot; only the one inside the box is read, on a z wall.)
template <typename T, bool EDGE>
struct Stencil {
    const V4<T> *b0, *bm1, *bp1, *b2;  // bases of planes j, j-1, j+1, j-2 or j+2
    int off;                           // ly * PX + lx
    int xm, ym, zm;
    T ihx, ihy, ihz;                   // 1 / (2 h)
    __device__ __forceinline__ V4<T> val() const { return b0[off]; }
    __device__ __forceinline__ V4<T> dx() const
    {
        const V4<T> *p = b0 + off;
        if (!EDGE || xm == 0) return d_central(p[1], p[-1], ihx);
        if (xm == 1) return d_low(p[0], p[1], p[2], ihx);
        return d_high(p[0], p[-1], p[-2], ihx);
    }
    __device__ __forceinline__ V4<T> dy() const
    {
        const V4<T> *p = b0 + off;
        if (!EDGE || ym == 0) return d_central(p[PX], p[-PX], ihy);
        if (ym == 1) return d_low(p[0], p[PX], p[2 * PX], ihy);
        return d_high(p[0], p[-PX], p[-2 * PX], ihy);
    }
    __device__ __forceinline__ V4<T> dz() const
    {
        if (zm == 0) return d_central(bp1[off], bm1[off], ihz);
        if (zm == 1) return d_low(b0[off], bp1[off], b2[off], ihz);
        return d_high(b0[off], bm1[off], b2[off], ihz);
    }
};

__device__ __forceinline__ int wall_mode(int c, int n) { return c == 0 ? 1 : (c == n - 1 ? 2 : 0); }

// Sutherland's law and Eq. reg (over mu_s), in a fixed order
template <typename T>
__device__ __forceinline__ void visc_coeffs(const VArgs<T> &a, T Tn, T &mu, T &mub)
{
    if constexpr (sizeof(T) == 4)
        mu = __fdividef(r_mul(r_mul(r_mul(Tn, Tn), rsqrtf(Tn)), a.S1), r_add(Tn, a.S));  // FP32 intrinsics
    else
        mu = r_mul(r_mul(Tn, sqrt(Tn)), a.S1) / r_add(Tn, a.S);
    mub = r_fma(a.c0, Tn, a.c1);
}

// the three viscosity factors of the stress (Eqs. ge19, bv1-bv3) divided by Re
template <typename T>
struct ViscK {
    T k43, k23, ks, mk;  // (4/3 mu + mu_b)/Re, (-2/3 mu + mu_b)/Re, mu/Re, -mu kq
    __device__ __forceinline__ ViscK(const VArgs<T> &a, T Tn)
    {
        T mu, mub;
        visc_coeffs(a, Tn, mu, mub);
        k43 = r_mul(r_fma(T(4) / T(3), mu, mub), a.iRe);
        k23 = r_mul(r_fma(T(-2) / T(3), mu, mub), a.iRe);
        ks = r_mul(mu, a.iRe);
        mk = r_mul(-mu, a.kq);
    }
};

// Viscous fluxes at a node from its values q = (u, v, w, T) and the
// gradients gx, gy, gz of (u, v, w, T) (Eqs. ge6-ge8, ge19, ge20, bv1-bv3).
// The heat flux normal to an adiabatic wall is zero on the wall node (wq = 0).
template <typename T>
__device__ __forceinline__ V4<T> flux_E(const ViscK<T> &k, const V4<T> &q, const V4<T> &gx, const V4<T> &gy,
                                        const V4<T> &gz, bool wq)
{
    const T txx = r_fma(k.k43, gx.x, r_mul(k.k23, r_add(gy.y, gz.z)));
    const T txy = r_mul(k.ks, r_add(gy.x, gx.y));
    const T txz = r_mul(k.ks, r_add(gz.x, gx.z));
    const T qx = wq ? r_mul(k.mk, gx.w) : T(0);
    return V4<T>{txx, txy, txz, r_add(r_fma(q.z, txz, r_fma(q.y, txy, r_mul(q.x, txx))), -qx)};
}
template <typename T>
__device__ __forceinline__ V4<T> flux_F(const ViscK<T> &k, const V4<T> &q, const V4<T> &gx, const V4<T> &gy,
                                        const V4<T> &gz, bool wq)
{
    const T tyy = r_fma(k.k43, gy.y, r_mul(k.k23, r_add(gx.x, gz.z)));
    const T txy = r_mul(k.ks, r_add(gy.x, gx.y));
    const T tyz = r_mul(k.ks, r_add(gz.y, gy.z));
    const T qy = wq ? r_mul(k.mk, gy.w) : T(0);
    return V4<T>{txy, tyy, tyz, r_add(r_fma(q.z, tyz, r_fma(q.y, tyy, r_mul(q.x, txy))), -qy)};
}
template <typename T>
__device__ __forceinline__ V4<T> flux_G(const ViscK<T> &k, const V4<T> &q, const V4<T> &gx, const V4<T> &gy,
                                        const V4<T> &gz, bool wq)
{
    const T tzz = r_fma(k.k43, gz.z, r_mul(k.k23, r_add(gx.x, gy.y)));
    const T txz = r_mul(k.ks, r_add(gz.x, gx.z));
    const T tyz = r_mul(k.ks, r_add(gz.y, gy.z));
    const T qz = wq ? r_mul(k.mk, gz.w) : T(0);
    return V4<T>{txz, tyz, tzz, r_add(r_fma(q.z, tzz, r_fma(q.y, tyz, r_mul(q.x, txz))), -qz)};
}



// primitives of a stage state from its FP32 deviation D = (rho', m_x, m_y, m_z, E')
__device__ __forceinline__ void prim_from_dev(const VArgs<float> &a, int p, int kg, const float D[5])
{
    float Wv[5];
    prim_from_deviation(a.rho_b[kg], a.gm1, D, Wv);
#pragma unroll
    for (int k = 0; k < 5; ++k) a.Wn[k][p] = Wv[k];
}

// Mixed form of the classical RK4 stage.  The slopes are FP32 (they are FP32
// right-hand sides); K = k1 + 2 k2 + 2 k3 + k4 is accumulated in FP32 and added
// to the FP64 state once, Q_n += dt/6 K, in FP64.  The stage states
// Q_n + c dt k are formed as FP32 deviations from the hydrostatic base, the
// same quantities the primitive recovery of the FP64 form rounds to FP32.
template <class S>
__device__ __forceinline__ void mixed_update(const VArgs<float> &a, int p, int kg, const float r[5],
                                             const float kold[5], const float dn[5], const double qn[5])
{
    const int s = st_of<S>(a);
    float K[5];
    if (s == 1) {
#pragma unroll
        for (int k = 0; k < 5; ++k) K[k] = r[k];
    } else {
        const float w = s == 4 ? 1.0f : 2.0f;
#pragma unroll
        for (int k = 0; k < 5; ++k) K[k] = __fmaf_rn(w, r[k], kold[k]);
    }
    float D[5];
    if (s < 4) {
#pragma unroll
        for (int k = 0; k < 5; ++k) a.Kacc[k][p] = K[k];
        const float c = s == 3 ? a.cdt1 : a.cdt2;
#pragma unroll
        for (int k = 0; k < 5; ++k) D[k] = __fmaf_rn(c, r[k], dn[k]);
    } else {
        const double w6 = a.dt6;
        double q[5];
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            q[k] = __fma_rn(w6, widen_f32(K[k]), qn[k]);
            a.Qn[k][p] = q[k];
        }
        D[0] = narrow_f64(q[0] - a.rho_b64[kg]);
        D[1] = narrow_f64(q[1]);
        D[2] = narrow_f64(q[2]);
        D[3] = narrow_f64(q[3]);
        D[4] = narrow_f64(q[4] - a.E_b64[kg]);
#pragma unroll
        for (int k = 0; k < 5; ++k) a.Dn[k][p] = D[k];
    }
    prim_from_dev(a, p, kg, D);
}

// Gravity source (Eq. ge8a), no-slip walls and the RK4 stage at node p, whose
// right-hand side r holds every other term.  w0 = rho - rho_b, ug = the
// velocity along gravity; kd, dn, qn (mixed form) = the node's K, D_n and, in
// stage 4, Q_n.
template <typename T, class S = RunSpec>
__device__ __forceinline__ void source_and_stage(const VArgs<T> &a, int p, int kg, bool wall, T w0, T ug, T r[5],
                                                 const float kd[5], const float dn[5], const double qn[5])
{
    const int ga = ga_of<S>(a), stage = st_of<S>(a);
    // fixed-order arithmetic: the same bits whether the stage and the gravity
    // axis are compile-time constants (Spec) or not
    const T rho = r_add(a.rho_b[kg], w0);
    const T sg = r_mul(w0, a.g);
    if (ga == 0) r[1] = r_add(r[1], -sg);
    if (ga == 1) r[2] = r_add(r[2], -sg);
    if (ga == 2) r[3] = r_add(r[3], -sg);
    r[4] = r_add(r[4], -r_mul(r_mul(rho, ug), a.g));
    // no-slip walls
    if (wall) r[1] = r[2] = r[3] = 0;
    if (stage == 0) {
#pragma unroll
        for (int k = 0; k < 5; ++k) a.Rout[k][p] = r[k];
    } else if constexpr (sizeof(T) == 4) {
        mixed_update<S>(a, p, kg, r, kd, dn, qn);
    } else {
        // classical RK4: acc collects Q_n + dt (k1 + 2 k2 + 2 k3 + k4) / 6
        const double bw = (stage == 1 || stage == 4) ? a.dt6 : a.dt3;
        const double cw = stage == 3 ? a.dt : a.dt2;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const double rk = (double)r[k];
            if (stage == 1) {
                const double q = a.Qn[k][p];
                a.acc[k][p] = __fma_rn(bw, rk, q);
                a.Qout[k][p] = __fma_rn(cw, rk, q);
            } else if (stage < 4) {
                a.acc[k][p] = __fma_rn(bw, rk, a.acc[k][p]);
                a.Qout[k][p] = __fma_rn(cw, rk, a.Qn[k][p]);
            } else {
                a.Qout[k][p] = __fma_rn(bw, rk, a.acc[k][p]);
            }
        }
    }
}


// shared memory of a block, in elements of T: ring, E_v and F_v (two planes
// each)
constexpr size_t VISC_ELEMENTS = 4 * ((size_t)RING * PLANE + 2 * TY * (TX + 2) + 2 * (TY + 2) * TX);

// One block marching through the planes z0 .. z1 - 1 of its tile.
template <typename T, bool EDGE, class S>
__device__ __forceinline__ void visc_rk_body(const VArgs<T> &a, const unsigned bx, const unsigned by,
                                             const unsigned bz, unsigned char *smraw)
{
    const int ga = ga_of<S>(a);
    using V = V4<T>;
    constexpr int EW = TX + 2, FH = TY + 2;  // E_v row width, F_v rows (one-node halos)
    const int nx = a.n[0], ny = a.n[1], nz = a.n[2];
    const int xs = bx * TX, ys = by * TY;
    const int x0 = min(xs, max(nx - TX, 0)), y0 = min(ys, max(ny - TY, 0));
    V *const ring = reinterpret_cast<V *>(smraw);
    V *const EV = ring + RING * PLANE;  // [2][TY][EW], local x + 1
    V *const FV = EV + 2 * TY * EW;     // [2][FH][TX], local y + 1
    const int z0 = bz * a.zc, z1 = min(nz, z0 + a.zc);
    const int tx = (int)(threadIdx.x % TX), ty = (int)(threadIdx.x / TX);
    const int x = x0 + tx, y = y0 + ty;
    // a block off the x and y walls (EDGE false) is never shifted back and
    // owns all its nodes, halo nodes included, inside the box
    const bool in_dom = !EDGE || (x < nx && y < ny);
    const bool own = !EDGE || (in_dom && x >= xs && y >= ys);
    const T ihx = a.ih2[0], ihy = a.ih2[1], ihz = a.ih2[2];
    const int xm = EDGE ? wall_mode(x, nx) : 0, ym = EDGE ? wall_mode(y, ny) : 0;
    const int p0 = x + nx * y, nxy = nx * ny;
    // first and last plane whose fluxes are evaluated: one beyond the output
    // planes, and three at least next to a wall, where the z divergence is
    // one-sided; planes [ulo, uhi) are updated inside the loop
    const int jb = max(0, z1 == nz ? min(z0 - 1, nz - 3) : z0 - 1);
    const int je = min(nz - 1, z0 == 0 ? max(z1, 2) : z1);
    const int ulo = max(z0, 1), uhi = min(z1, nz - 1), top = min(je + 1, nz - 1);

    auto stencil_at = [&](int lx, int ly, int j) {
        Stencil<T, EDGE> St;
        auto plane = [&](int z) { return (const V *)(ring + (z & (RING - 1)) * PLANE); };
        St.b0 = plane(j);
        St.bm1 = plane(j - 1);
        St.bp1 = plane(j + 1);
        St.b2 = plane(j + 2);
        St.off = (ly + HALO) * PX + (lx + HALO);
        St.xm = EDGE ? wall_mode(x0 + lx, nx) : 0;
        St.ym = EDGE ? wall_mode(y0 + ly, ny) : 0;
        St.zm = wall_mode(j, nz);
        St.ihx = ihx;
        St.ihy = ihy;
        St.ihz = ihz;
        return St;
    };
    // divergence dv added, gravity source, RK stage of the node of plane o,
    // whose velocity along gravity is ug
    auto update = [&](UpdateIn<T, S> &in, int o, const V &dv, T ug) {
        in.r[1] = r_add(in.r[1], dv.x);
        in.r[2] = r_add(in.r[2], dv.y);
        in.r[3] = r_add(in.r[3], dv.z);
        in.r[4] = r_add(in.r[4], dv.w);
        const int kg = ga == 0 ? x : (ga == 1 ? y : o);
        const bool wall = (EDGE && (x == 0 || x == nx - 1 || y == 0 || y == ny - 1)) || o == 0 || o == nz - 1;
        source_and_stage<T, S>(a, p0 + nxy * o, kg, wall, in.w0, ug, in.r, in.kd, in.dn, in.qn);
    };
    auto ug_of = [&](int o) {
        const V &q = ring[(o & (RING - 1)) * PLANE + (ty + HALO) * PX + tx + HALO];
        return ga == 0 ? q.x : (ga == 1 ? q.y : q.z);
    };

    RingNodes<T, S> rn;
    rn.init(a, x0, y0);
    // planes jb - 1 .. jb + 1, or 0 .. 2 at the bottom wall
    const int zf = max(jb - 1, 0);
    rn.template load<3>(a, ring, zf);
    int lhi = zf + 2;  // last plane in the ring
    __syncthreads();
    // G_v of planes j, j - 1, j - 2; x and y divergence of plane j - 1; of the
    // bottom wall, whose plane leaves the ring before its update: the energy
    // component and the velocity along gravity
    V g0{}, g1{}, g2{}, dxy{};
    T dwall = T(0), uwall = T(0);
#pragma unroll 1
    for (int j = jb; j <= je; ++j) {
        V *const ev = EV + (j & 1) * TY * EW, *const fv = FV + (j & 1) * FH * TX;
        const int o = j - 1;
        const bool load = j + 2 > lhi && j + 2 <= top, upd = o >= ulo && o < uhi && own;
        UpdateIn<T, S> in;
        if (load) rn.issue(a, j + 2);
        if (upd) in.load(a, p0 + nxy * o);
        if (j + 3 <= top) rn.prefetch(a, j + 3);
        if (j < uhi && own) UpdateIn<T, S>::prefetch(a, p0 + nxy * j);
        // ---- viscous fluxes of plane j ----
        g2 = g1;
        g1 = g0;
        if (in_dom) {
            const Stencil<T, EDGE> St = stencil_at(tx, ty, j);
            const V q = St.val(), gx = St.dx(), gy = St.dy(), gz = St.dz();
            const ViscK<T> k(a, q.w);
            ev[ty * EW + tx + 1] = flux_E(k, q, gx, gy, gz, St.xm == 0);
            fv[(ty + 1) * TX + tx] = flux_F(k, q, gx, gy, gz, St.ym == 0);
            g0 = flux_G(k, q, gx, gy, gz, St.zm == 0);
        }
        // F_v on the y halo (warps 0 and 1) and E_v on the x halo (warp 2):
        // the same arithmetic as in the tile that owns the node, so the same
        // bits
        if (threadIdx.x < 2 * TX) {
            const int side = threadIdx.x / TX, hx = threadIdx.x % TX;
            const int ly = side ? TY : -1;
            const int gx_ = x0 + hx, gy_ = y0 + ly;
            if (!EDGE || (gy_ >= 0 && gy_ < ny && gx_ < nx)) {
                const Stencil<T, EDGE> St = stencil_at(hx, ly, j);
                const V q = St.val(), gx = St.dx(), gy = St.dy(), gz = St.dz();
                fv[(ly + 1) * TX + hx] = flux_F(ViscK<T>(a, q.w), q, gx, gy, gz, St.ym == 0);
            }
        } else if (threadIdx.x < 2 * TX + 2 * TY) {
            const int t = threadIdx.x - 2 * TX;
            const int side = t / TY, hy = t % TY;
            const int lx = side ? TX : -1;
            const int gx_ = x0 + lx, gy_ = y0 + hy;
            if (!EDGE || (gx_ >= 0 && gx_ < nx && gy_ < ny)) {
                const Stencil<T, EDGE> St = stencil_at(lx, hy, j);
                const V q = St.val(), gx = St.dx(), gy = St.dy(), gz = St.dz();
                ev[hy * EW + lx + 1] = flux_E(ViscK<T>(a, q.w), q, gx, gy, gz, St.xm == 0);
            }
        }
        // ---- RK update of plane j - 1, and the ring's plane j + 2 ----
        if (upd) update(in, o, v_add(dxy, d_central(g0, g2, ihz)), ug_of(o));
        if (z0 == 0 && j == 2 && own) {  // the bottom wall (its momentum stays zero)
            in.load(a, p0);
            V d{};
            d.w = r_add(dwall, d_low(g2, g1, g0, ihz).w);
            update(in, 0, d, uwall);
        }
        if (load) {
            // into the slot of plane j - 2, which no thread reads any more
            rn.settle(a, ring, j + 2);
            lhi = j + 2;
        }
        __syncthreads();
        // ---- x and y divergence of plane j ----
        if (own) {
            const V *e = ev + ty * EW + tx + 1;
            const V *f = fv + (ty + 1) * TX + tx;
            V dvx, dvy;
            if (xm == 0)
                dvx = d_central(e[1], e[-1], ihx);
            else if (xm == 1)
                dvx = d_low(e[0], e[1], e[2], ihx);
            else
                dvx = d_high(e[0], e[-1], e[-2], ihx);
            if (ym == 0)
                dvy = d_central(f[TX], f[-TX], ihy);
            else if (ym == 1)
                dvy = d_low(f[0], f[TX], f[2 * TX], ihy);
            else
                dvy = d_high(f[0], f[-TX], f[-2 * TX], ihy);
            dxy = v_add(dvx, dvy);
            if (j == 0) {
                dwall = dxy.w;
                uwall = ug_of(0);
            }
        }
    }
    if (z1 == nz && own) {  // the top wall
        UpdateIn<T, S> in;
        in.load(a, p0 + nxy * (nz - 1));
        update(in, nz - 1, v_add(dxy, d_high(g0, g1, g2, ihz)), ug_of(nz - 1));
    }
}

// One block (bx, by, bz) of the fused viscous / source / RK stage kernel:
// blocks whose x and y ranges (with the one-node flux halo) stay off the walls
// take the branch-free stencils.
template <typename T, class S = RunSpec>
__device__ __forceinline__ void visc_rk_block(const VArgs<T> &a, const unsigned bx, const unsigned by,
                                              const unsigned bz, unsigned char *smraw)
{
    const int nx = a.n[0], ny = a.n[1];
    const int x0 = min(bx * TX, max(nx - TX, 0)), y0 = min(by * TY, max(ny - TY, 0));
    const bool edge = x0 - 1 <= 0 || x0 + TX >= nx - 1 || y0 - 1 <= 0 || y0 + TY >= ny - 1;
    if (edge)
        visc_rk_body<T, true, S>(a, bx, by, bz, smraw);
    else
        visc_rk_body<T, false, S>(a, bx, by, bz, smraw);
}

template <typename T>
constexpr size_t visc_smem() { return VISC_ELEMENTS * sizeof(T); }

// Blocks in x, y and z, and planes per block zc: the least waves x planes, a
// block spending about three planes' time on its first planes and on the two
// planes of fluxes beyond its own.  Chunks of 32 instead of 64 planes: 7.01
// against 6.98 ms at 1024 x 512 x 512, 0.526 against 0.549 at 256^3 (two and a
// half waves of 64); of 8 at least: 25 instead of 17 us at 48^3.
template <typename T>
dim3 visc_grid(const BoxDev &bx, int &zc)
{
    const int gx = (bx.n[0] + TX - 1) / TX, gy = (bx.n[1] + TY - 1) / TY, nz = bx.n[2];
    const long long slots = 152LL * visc_occupancy<T>();
    long long best = -1;
    for (int c = 2; c <= 64; ++c) {
        const long long blocks = (long long)gx * gy * ((nz + c - 1) / c);
        const long long cost = (blocks + slots - 1) / slots * (c + 3);
        if (best < 0 || cost < best) {
            best = cost;
            zc = c;
        }
    }
    return dim3(gx, gy, (nz + zc - 1) / zc);
}

template <typename T>
VArgs<T> make_vargs(const BoxDev &bx, const T *W, const T *R, int stage, const StageRegs<T> &g)
{
    VArgs<T> a{};
    for (int d = 0; d < 3; ++d) {
        a.n[d] = bx.n[d];
        a.ih2[d] = (T)(0.5 * bx.inv_h[d]);
    }
    a.np = (int)bx.np;
    a.ga = bx.ga;
    a.gm2 = (T)bx.gm2;
    a.iRe = (T)(1.0 / bx.Re);
    a.kq = (T)bx.kq;
    a.S1 = (T)(1.0 + bx.suth_S);
    a.S = (T)bx.suth_S;
    a.c0 = (T)bx.mub_coef0;
    a.c1 = (T)bx.mub_coef1;
    a.g = (T)bx.g;
    for (int k = 0; k < 5; ++k) a.W[k] = W + (size_t)k * bx.np;
    if constexpr (sizeof(T) == 8) {
        a.rho_b = (const T *)bx.rho_b64;
        a.p_b = (const T *)bx.p_b64;
    } else {
        a.rho_b = (const T *)bx.rho_b32;
    }
    a.T_b = bx.T_b32;
    a.ip_b = bx.ip_b32;
    a.ir_b = bx.ir_b32;
    for (int k = 0; k < 5; ++k) a.R[k] = R + (size_t)k * bx.np;
    a.stage = stage;
    a.dt = bx.dt;
    a.dt6 = bx.dt / 6.0;
    a.dt3 = bx.dt / 3.0;
    a.dt2 = 0.5 * bx.dt;
    a.cdt2 = (float)(0.5 * bx.dt);
    a.cdt1 = (float)bx.dt;
    auto fp = [&](auto *base, int k) { return base ? base + (size_t)k * bx.np : base; };
    for (int k = 0; k < 5; ++k) {
        a.Rout[k] = fp(g.Rout, k);
        a.Qn[k] = fp(g.Qn, k);
        a.acc[k] = fp(g.acc, k);
        a.Qout[k] = fp(g.Qout, k);
        a.Kacc[k] = fp(g.Kacc, k);
        a.Dn[k] = fp(g.Dn, k);
    }
    for (int k = 0; k < 5; ++k) a.Wn[k] = fp(g.Wn, k);
    a.rho_b64 = bx.rho_b64;
    a.E_b64 = bx.E_b64;
    a.gm1 = (float)(bx.gamma - 1.0);
    return a;
}

}  // namespace

}  // namespace nopcs
