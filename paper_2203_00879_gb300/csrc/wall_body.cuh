// Device side of the no-slip adiabatic wall conditions (a reading of Sec. 2,
// Fig. 1), shared by the stand-alone wall kernels (rk_kernels.cu) and the
// batched persistent kernel (batch_kernel.cu).
#pragma once

#include "nopcs_internal.cuh"

namespace nopcs {

namespace {

// ---------------------------------------------------------------------------
// No-slip adiabatic walls: momentum zero on every wall node (kept by the
// update), T_w = (4 T_1 - T_2) / 3 along the inward normal, averaged over the
// normals of edge and corner nodes, where T_1 and T_2 are wall temperatures
// themselves (edges from the faces, corners from the edges).
// E_w = rho_w T_w / (gamma (gamma-1) M^2).
//
// Faces and edges are set in one pass: an edge node works out the four face
// temperatures it needs from the four interior nodes behind them instead of
// waiting for them, so nothing reads what another thread writes (the density of
// a wall node is not written).  A corner reads the two nodes next to it on each
// of its edges, so one block sets the 48 such edge nodes of a box and then, after
// a barrier, its corners.
// Bound by latency at all but the largest sizes: every load of a node is issued
// before its first use, and a stage has one launch.  Between two events on the
// stream at 48^3 and 256^3: 28 and 70 us as three launches (faces, edges,
// corners) with branches between the loads, 20 and 57 with the faces and edges
// in one, now 14 and 45.  (Edges and corners recursing to the interior, nothing
// shared: 50 us at 48^3.)
// ---------------------------------------------------------------------------

// On the FP64 state (refreshing D_n and W when given).  A value is a
// temperature.
struct WallState {
    using T = double;
    const BoxDev &bx;
    double *Q;
    float *Dn, *Wf;
    __device__ __forceinline__ double temp(double r, double mx, double my, double mz, double E) const
    {
        const double ke = 0.5 * (mx * mx + my * my + mz * mz) / r;
        return bx.gm2 * (bx.gamma - 1.0) * (E - ke) / r;
    }
    // value of a stored node
    __device__ __forceinline__ double node(long long i, int) const
    {
        const long long np = bx.np;
        return temp(Q[i], Q[np + i], Q[2 * np + i], Q[3 * np + i], Q[4 * np + i]);
    }
    // extrapolation to a wall node from the nodes one and two inside
    __device__ __forceinline__ double extrapolate(int, int, double t1, int, double t2) const
    {
        return (4.0 * t1 - t2) / 3.0;
    }
    // value of a wall node that extrapolates to tw (through the energy it stores)
    __device__ __forceinline__ double wall(long long i, int, double tw) const
    {
        const double r = Q[i];
        return temp(r, 0.0, 0.0, 0.0, r * tw * bx.cE);
    }
    __device__ __forceinline__ void store(long long i, int kg, double tw) const
    {
        const long long np = bx.np;
        const double r = Q[i], E = r * tw * bx.cE;
        Q[np + i] = Q[2 * np + i] = Q[3 * np + i] = 0.0;
        Q[4 * np + i] = E;
        if (Dn) {
            const float Dv[5] = {(float)(r - bx.rho_b64[kg]), 0.0f, 0.0f, 0.0f, (float)(E - bx.E_b64[kg])};
            float Wv[5];
            prim_from_deviation(bx.rho_b32[kg], (float)(bx.gamma - 1.0), Dv, Wv);
#pragma unroll
            for (int k = 0; k < 5; ++k) Dn[k * np + i] = Dv[k];
#pragma unroll
            for (int k = 0; k < 5; ++k) Wf[k * np + i] = Wv[k];
        }
    }
};

// On an FP32 stage state held as W (mixed form).  A node's value is T' of T =
// T_b + T', T' = T_b (p'/p_b - rho'/rho_b) / (1 + rho'/rho_b); an extrapolated
// wall temperature is its difference dT from T_b at the wall node, and
// E_w - E_b = cE (rho' T_w + rho_b dT) (E_b = cE rho_b T_b).
struct WallStage {
    using T = float;
    const BoxDev &bx;
    float *W;
    __device__ __forceinline__ float dtemp(float rd, float pd, int kg) const
    {
        const float rr = rd * bx.ir_b32[kg];
        return bx.T_b32[kg] * (pd * bx.ip_b32[kg] - rr) / (1.0f + rr);
    }
    __device__ __forceinline__ float energy(float rd, int kg, float dT) const
    {
        return (float)bx.cE * (rd * (bx.T_b32[kg] + dT) + bx.rho_b32[kg] * dT);
    }
    __device__ __forceinline__ float node(long long i, int kg) const { return dtemp(W[i], W[4 * bx.np + i], kg); }
    __device__ __forceinline__ float extrapolate(int kg, int k1, float t1, int k2, float t2) const
    {
        const float TbP = bx.T_b32[kg];
        const float d1 = (bx.T_b32[k1] - TbP) + t1, d2 = (bx.T_b32[k2] - TbP) + t2;
        return (4.0f * d1 - d2) * (1.0f / 3.0f);
    }
    __device__ __forceinline__ float wall(long long i, int kg, float dT) const
    {
        const float rd = W[i];
        return dtemp(rd, (float)(bx.gamma - 1.0) * energy(rd, kg, dT), kg);
    }
    __device__ __forceinline__ void store(long long i, int kg, float dT) const
    {
        const long long np = bx.np;
        const float Ed = energy(W[i], kg, dT);
        W[np + i] = W[2 * np + i] = W[3 * np + i] = 0.0f;
        W[4 * np + i] = (float)(bx.gamma - 1.0) * Ed;
    }
};

// One step inwards along axis d from a node with coordinate c there: in the
// node index and in the coordinate along gravity.
struct Inward {
    long long s;
    int k;
    __device__ __forceinline__ Inward(const BoxDev &bx, int d, int c)
    {
        const int sg = c == 0 ? 1 : -1;
        s = sg * (d == 0 ? 1LL : (d == 1 ? (long long)bx.n[0] : (long long)bx.n[0] * bx.n[1]));
        k = d == bx.ga ? sg : 0;
    }
};

template <class S>
__device__ __forceinline__ typename S::T along(const S &w, long long i, int kg, const Inward &d)
{
    const auto t1 = w.node(i + d.s, kg + d.k), t2 = w.node(i + 2 * d.s, kg + 2 * d.k);
    return w.extrapolate(kg, kg + d.k, t1, kg + 2 * d.k, t2);
}
template <class S>
__device__ __forceinline__ void face_update(const S &w, long long i, int kg, const Inward &d)
{
    w.store(i, kg, along(w, i, kg, d));
}
// a, b: the edge's two normals, in the order of their axes
template <class S>
__device__ __forceinline__ void edge_update(const S &w, long long i, int kg, const Inward &a, const Inward &b)
{
    using T = typename S::T;
    T t[2][2];  // interior nodes, steps along a and b
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) t[p][q] = w.node(i + (p + 1) * a.s + (q + 1) * b.s, kg + (p + 1) * a.k + (q + 1) * b.k);
    T fa[2], fb[2];  // the face nodes along a (on the wall of b) and along b
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int ka = kg + (p + 1) * a.k, kb = kg + (p + 1) * b.k;
        fa[p] = w.wall(i + (p + 1) * a.s, ka, w.extrapolate(ka, ka + b.k, t[p][0], ka + 2 * b.k, t[p][1]));
        fb[p] = w.wall(i + (p + 1) * b.s, kb, w.extrapolate(kb, kb + a.k, t[0][p], kb + 2 * a.k, t[1][p]));
    }
    w.store(i, kg, (w.extrapolate(kg, kg + a.k, fa[0], kg + 2 * a.k, fa[1]) +
                    w.extrapolate(kg, kg + b.k, fb[0], kg + 2 * b.k, fb[1])) / T(2));
}

// node `run` of edge e = 4 x its axis + the sides of the other two coordinates
template <class S>
__device__ __forceinline__ void edge_node(const BoxDev &bx, unsigned e, int run, const S &w)
{
    const int ax = (int)(e >> 2), a = ax == 0 ? 1 : 0, b = ax == 2 ? 1 : 2;  // a, b: the normals' axes
    const int ca = (e & 1u) ? (a == 0 ? bx.n[0] : bx.n[1]) - 1 : 0, cb = (e & 2u) ? (b == 1 ? bx.n[1] : bx.n[2]) - 1 : 0;
    int c[3];
    c[0] = ax == 0 ? run : ca;
    c[1] = ax == 1 ? run : (ax == 0 ? ca : cb);
    c[2] = ax == 2 ? run : cb;
    const long long i = c[0] + (long long)bx.n[0] * (c[1] + (long long)bx.n[1] * c[2]);
    edge_update(w, i, bx.ga == 0 ? c[0] : (bx.ga == 1 ? c[1] : c[2]), Inward(bx, a, ca), Inward(bx, b, cb));
}

// Wall nodes in order: faces (one wall coordinate), edges (two).
// A box of fewer than 2^31 points has fewer than 2^31 of them.
__host__ __device__ __forceinline__ unsigned face_count(const BoxDev &bx)
{
    const unsigned nx = bx.n[0] - 2, ny = bx.n[1] - 2, nz = bx.n[2] - 2;
    return 2u * (ny * nz + nx * nz + nx * ny);
}
__host__ __device__ __forceinline__ unsigned edge_count(const BoxDev &bx)
{
    return 4u * (unsigned)(bx.n[0] - 2 + bx.n[1] - 2 + bx.n[2] - 2);
}
// faces and edges
__host__ __device__ __forceinline__ unsigned wall_count(const BoxDev &bx)
{
    return face_count(bx) + edge_count(bx);
}
// wall node t (a face or an edge node) of the state seen through w; the edge
// nodes that a corner reads are left to corner_block
template <class S>
__device__ __forceinline__ void wall_update(const BoxDev &bx, unsigned q, const S &w)
{
    const unsigned m[3] = {(unsigned)bx.n[0] - 2u, (unsigned)bx.n[1] - 2u, (unsigned)bx.n[2] - 2u};
    int c[3] = {0, 0, 0};
    const unsigned fx = m[1] * m[2], fy = m[0] * m[2], fz = m[0] * m[1];
    auto at = [&] { return c[0] + (long long)bx.n[0] * (c[1] + (long long)bx.n[1] * c[2]); };
    auto kg = [&] { return bx.ga == 0 ? c[0] : (bx.ga == 1 ? c[1] : c[2]); };
    if (q < 2u * (fx + fy + fz)) {
        int d;
        if (q < 2u * fx) {
            const unsigned side = q >= fx, r = q - side * fx;
            c[0] = side ? bx.n[0] - 1 : 0, c[1] = 1 + (int)(r % m[1]), c[2] = 1 + (int)(r / m[1]);
            d = 0;
        } else if ((q -= 2u * fx) < 2u * fy) {
            const unsigned side = q >= fy, r = q - side * fy;
            c[1] = side ? bx.n[1] - 1 : 0, c[0] = 1 + (int)(r % m[0]), c[2] = 1 + (int)(r / m[0]);
            d = 1;
        } else {
            q -= 2u * fy;
            const unsigned side = q >= fz, r = q - side * fz;
            c[2] = side ? bx.n[2] - 1 : 0, c[0] = 1 + (int)(r % m[0]), c[1] = 1 + (int)(r / m[0]);
            d = 2;
        }
        face_update(w, at(), kg(), Inward(bx, d, d == 0 ? c[0] : (d == 1 ? c[1] : c[2])));
        return;
    }
    q -= 2u * (fx + fy + fz);
    // edges along x, y, z, the other two coordinates at 0 or n - 1 (4 combinations)
    const int e = q < 4u * m[0] ? 0 : (q < 4u * (m[0] + m[1]) ? 1 : 2);
    q -= e == 0 ? 0u : (e == 1 ? 4u * m[0] : 4u * (m[0] + m[1]));
    const unsigned me = e == 0 ? m[0] : (e == 1 ? m[1] : m[2]), combo = q / me;
    const int run = 1 + (int)(q % me), last = (int)me;
    if (run > 2 && run < last - 1) edge_node(bx, 4u * (unsigned)e + combo, run, w);
}

// corner t of 8
template <class S>
__device__ __forceinline__ void corner_update(const BoxDev &bx, unsigned t, const S &w)
{
    int c[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d] = (t >> d) & 1u ? bx.n[d] - 1 : 0;
    const long long i = c[0] + (long long)bx.n[0] * (c[1] + (long long)bx.n[1] * c[2]);
    const int kg = bx.ga == 0 ? c[0] : (bx.ga == 1 ? c[1] : c[2]);
    typename S::T tw = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) tw += along(w, i, kg, Inward(bx, d, c[d]));
    w.store(i, kg, tw / typename S::T(3));
}

// the FP64 state Q (refreshing Dn and Wf when given), or, with Q == nullptr, the
// FP32 stage primitives Ww
__device__ __forceinline__ void wall_node(const BoxDev &bx, unsigned t, double *Q, float *Dn, float *Wf, float *Ww)
{
    if (Q)
        wall_update(bx, t, WallState{bx, Q, Dn, Wf});
    else
        wall_update(bx, t, WallStage{bx, Ww});
}
// The corners and the edge nodes next to them, by all threads of one block (48
// at least).
template <class S>
__device__ __forceinline__ void corner_block_of(const BoxDev &bx, unsigned t, const S &w)
{
    if (t < 48) {
        const unsigned e = t >> 2, k = t & 3;
        const int last = (e < 4 ? bx.n[0] : (e < 8 ? bx.n[1] : bx.n[2])) - 2;  // of the edge's nodes 1 .. last
        const int run = k < 2 ? 1 + (int)k : last - (int)k + 2;
        if (k < 2 || run > 2) edge_node(bx, e, run, w);  // each node once
    }
    __syncthreads();
    if (t < 8) corner_update(bx, t, w);
}
__device__ __forceinline__ void corner_block(const BoxDev &bx, unsigned t, double *Q, float *Dn, float *Wf, float *Ww)
{
    if (Q)
        corner_block_of(bx, t, WallState{bx, Q, Dn, Wf});
    else
        corner_block_of(bx, t, WallStage{bx, Ww});
}

}  // namespace

}  // namespace nopcs
