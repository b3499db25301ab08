// The kernels of a physical step outside the sub-iteration: S refresh (a1), saturation update with
// the move of R to the node pressure (a4, a5), and the output fields; blocks shared by the
// single-lattice launches and the batched ones.
//
// They are bound by memory: at 4096^2 (16.8 M nodes) the saturation update moves 39 planes, 2.6 GB.
// One node per thread with 32-bit loads kept too few bytes in flight (half of the DRAM bandwidth, warps
// waiting on loads), and the move of R was a pass of its own over 19 planes.  At 4096^2, then and
// now: saturation and move of R 565 + 186 and 443 us (5.9 TB/s), refresh 213 and 138 us, P and S or
// u 234 and 129 us (6.3 TB/s).  Here a thread takes four consecutive nodes with 128-bit loads, all issued
// before the first use; the pulls from the neighbouring columns are shuffles.  Walls would make a
// warp run both paths, and a wall quad four nodes one after the other, so wall nodes (and the
// nodes of quads that hold one) are threads of their own, in the first blocks.
#pragma once

#include "lbm2p_device.cuh"
#include "lbm2p_node.cuh"

namespace lbm2p_dev {

constexpr int kStepThreads = 128;

// Interior rows: quads of nodes from column 4 on, none holding column nx - 1; the rest is edge
// nodes.  Blocks [0, eb) take the edge nodes, [eb, eb + qb) the quads.
struct StepMap {
    int nx, ny;
    int fq;                      // quads per interior row
    int er;                      // edge nodes per interior row
    int edges, quads;
    int eb, qb;

    __host__ __device__ StepMap(int nx_, int ny_) : nx(nx_), ny(ny_)
    {
        fq = nx >= 9 && ny > 2 ? (nx - 5) / 4 : 0;
        er = nx - 4 * fq;
        quads = fq * (ny - 2);
        edges = nx * ny - 4 * quads;
        if (fq == 0)
            quads = 0, edges = nx * ny;
        eb = (edges + kStepThreads - 1) / kStepThreads;
        qb = (quads + kStepThreads - 1) / kStepThreads;
    }
    __host__ __device__ int blocks() const { return eb + qb; }
    __host__ __device__ void edge(int e, int &x, int &y) const
    {
        if (fq == 0) {
            y = e / nx;
            x = e - y * nx;
        } else if (e < 2 * nx) {
            y = e < nx ? 0 : ny - 1;
            x = e < nx ? e : e - nx;
        } else {
            e -= 2 * nx;
            y = 1 + e / er;
            x = e - (y - 1) * er;
            x += x < 4 ? 0 : 4 * fq;
        }
    }
};

// A thread's quad; threads past the last one repeat it and store nothing (the warp's shuffles need
// every lane).
struct StepQuad {
    int o;                       // offset of its first node
    int x, y;
    bool first, last;            // the column on its left (right) is not the lane's before (after)
    bool store;

    __device__ __forceinline__ StepQuad(const StepMap &m, int block, int pitch)
    {
        int q = (block - m.eb) * kStepThreads + (int)threadIdx.x;
        store = q < m.quads;
        q = store ? q : m.quads - 1;
        const int r = q / m.fq, c = q - r * m.fq;
        y = r + 1;
        x = 4 + 4 * c;
        o = y * pitch + x;
        const int lane = threadIdx.x & 31;
        first = lane == 0 || c == 0;
        last = lane == 31 || c == m.fq - 1;
    }
};

__device__ __forceinline__ float4 ldq(const float *p, int o)
{
    return *reinterpret_cast<const float4 *>(p + o);
}

__device__ __forceinline__ void stq(float *p, int o, float4 v)
{
    *reinterpret_cast<float4 *>(p + o) = v;
}

// (left neighbour of v.x, v.x, v.y, v.z); where the neighbour is no lane's, it is `edge`
__device__ __forceinline__ float4 from_left(float4 v, float edge, bool first)
{
    const float l = __shfl_up_sync(0xffffffffu, v.w, 1);
    return make_float4(first ? edge : l, v.x, v.y, v.z);
}

// (v.y, v.z, v.w, right neighbour of v.w)
__device__ __forceinline__ float4 from_right(float4 v, float edge, bool last)
{
    const float r = __shfl_down_sync(0xffffffffu, v.x, 1);
    return make_float4(v.y, v.z, v.w, last ? edge : r);
}

__device__ __forceinline__ float4 devq(float4 n, float w, float4 r, float4 r0)
{
    return make_float4(dev1(n.x, w, r.x, r0.x), dev1(n.y, w, r.y, r0.y), dev1(n.z, w, r.z, r0.z),
                       dev1(n.w, w, r.w, r0.w));
}

// what gather_a reads for a quad of interior nodes, in two halves: the loads, then the values
struct PullA {
    float4 n[8], r[3];
    float el[6], er[6];

    __device__ __forceinline__ void load(const float *const *fin, const float *R, const StepQuad &s, int p)
    {
        const int o = s.o;
        n[0] = ldq(fin[0], o);
        n[1] = ldq(fin[1], o - p);
        n[2] = ldq(fin[2], o);
        n[3] = ldq(fin[3], o + p);
        n[4] = ldq(fin[4], o - p);
        n[5] = ldq(fin[5], o - p);
        n[6] = ldq(fin[6], o + p);
        n[7] = ldq(fin[7], o + p);
        r[0] = ldq(R, o - p);
        r[1] = ldq(R, o);
        r[2] = ldq(R, o + p);
#pragma unroll
        for (int k = 0; k < 6; ++k)
            el[k] = er[k] = 0.0f;
        if (s.first) {
            el[0] = fin[0][o - 1];
            el[1] = fin[4][o - p - 1];
            el[2] = fin[7][o + p - 1];
            el[3] = R[o - p - 1];
            el[4] = R[o - 1];
            el[5] = R[o + p - 1];
        }
        if (s.last) {
            er[0] = fin[2][o + 4];
            er[1] = fin[5][o - p + 4];
            er[2] = fin[6][o + p + 4];
            er[3] = R[o - p + 4];
            er[4] = R[o + 4];
            er[5] = R[o + p + 4];
        }
    }
    __device__ __forceinline__ void values(const StepQuad &s, float4 (&f)[8]) const
    {
        const float4 r0 = r[1];
        f[0] = devq(from_left(n[0], el[0], s.first), wgt(1), from_left(r0, el[4], s.first), r0);
        f[1] = devq(n[1], wgt(2), r[0], r0);
        f[2] = devq(from_right(n[2], er[0], s.last), wgt(3), from_right(r0, er[4], s.last), r0);
        f[3] = devq(n[3], wgt(4), r[2], r0);
        f[4] = devq(from_left(n[4], el[1], s.first), wgt(5), from_left(r[0], el[3], s.first), r0);
        f[5] = devq(from_right(n[5], er[1], s.last), wgt(6), from_right(r[0], er[3], s.last), r0);
        f[6] = devq(from_right(n[6], er[2], s.last), wgt(7), from_right(r[2], er[5], s.last), r0);
        f[7] = devq(from_left(n[7], el[2], s.first), wgt(8), from_left(r[2], el[5], s.first), r0);
    }
};

// the same for gather_g
struct PullG {
    float4 n[9];
    float el[3], er[3];

    __device__ __forceinline__ void load(const float *const *gin, int qs, const StepQuad &s, int p)
    {
        const int o = s.o;
        const bool diag = qs == 9;
        n[0] = ldq(gin[0], o);
        n[1] = ldq(gin[1], o);
        n[2] = ldq(gin[2], o - p);
        n[3] = ldq(gin[3], o);
        n[4] = ldq(gin[4], o + p);
        n[5] = n[6] = n[7] = n[8] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (diag) {
            n[5] = ldq(gin[5], o - p);
            n[6] = ldq(gin[6], o - p);
            n[7] = ldq(gin[7], o + p);
            n[8] = ldq(gin[8], o + p);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
            el[k] = er[k] = 0.0f;
        if (s.first) {
            el[0] = gin[1][o - 1];
            if (diag) {
                el[1] = gin[5][o - p - 1];
                el[2] = gin[8][o + p - 1];
            }
        }
        if (s.last) {
            er[0] = gin[3][o + 4];
            if (diag) {
                er[1] = gin[6][o - p + 4];
                er[2] = gin[7][o + p + 4];
            }
        }
    }
    __device__ __forceinline__ void values(const StepQuad &s, float4 (&q)[9]) const
    {
        q[0] = n[0];
        q[1] = from_left(n[1], el[0], s.first);
        q[2] = n[2];
        q[3] = from_right(n[3], er[0], s.last);
        q[4] = n[4];
        q[5] = from_left(n[5], el[1], s.first);
        q[6] = from_right(n[6], er[1], s.last);
        q[7] = from_right(n[7], er[2], s.last);
        q[8] = from_left(n[8], el[2], s.first);
    }
};

__device__ __forceinline__ float &at4(float4 &v, int c) { return (&v.x)[c]; }
__device__ __forceinline__ float at4(const float4 &v, int c) { return (&v.x)[c]; }

// a1 over block `b` of the map: 1/tau_f, and R of the coming solve.  With the warm start the
// equilibrium part of f_i = n_i + w_i R moves with R to the pressure extrapolated in time,
// R' = R + (R - P^{n-1}); n_i (the rest) is kept.
__device__ __forceinline__ void refresh_block(const RefreshArgs &a, int b)
{
    const StepMap m(a.g.nx, a.g.ny);
    if (b < m.eb) {
        const int e = b * kStepThreads + (int)threadIdx.x;
        if (e >= m.edges)
            return;
        int x, y;
        m.edge(e, x, y);
        const int o = y * a.g.pitch + x;
        float q[9];
        gather_g(a.gin, a.g, a.m, a.Sb, x, y, o, q);
        const float K = a.K[o], r = a.Rin[o], pv = a.Pstep_in ? a.Pstep_in[o] : r;
        a.inv_tau[o] = refresh_tau(a, o, q, K);
        a.Rout[o] = a.Pstep_in ? r + (r - pv) : r;
        if (a.Pstep_in)
            a.Pstep_out[o] = r;
        return;
    }
    const StepQuad s(m, b, a.g.pitch);
    PullG g;
    g.load(a.gin, a.m.qs, s, a.g.pitch);
    const float4 K = ldq(a.K, s.o), r = ldq(a.Rin, s.o);
    const float4 pv = a.Pstep_in ? ldq(a.Pstep_in, s.o) : r;
    float4 q[9], it, R;
    g.values(s, q);
    if (!s.store)
        return;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float qc[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            qc[i] = at4(q[i], c);
        at4(it, c) = refresh_tau(a, s.o + c, qc, at4(K, c));
        at4(R, c) = a.Pstep_in ? at4(r, c) + (at4(r, c) - at4(pv, c)) : at4(r, c);
    }
    stq(a.inv_tau, s.o, it);
    stq(a.Rout, s.o, R);
    if (a.Pstep_in)
        stq(a.Pstep_out, s.o, r);
}

// a4 + a5 over block `b` of the map, and the move of R to the node pressure of the pulled state:
// n_i += w_i (R - Rnew) leaves f_i = n_i + w_i R unchanged
__device__ __forceinline__ void saturation_block(const SaturationArgs &a, int b)
{
    const StepMap m(a.g.nx, a.g.ny);
    if (b < m.eb) {
        const int e = b * kStepThreads + (int)threadIdx.x;
        if (e >= m.edges)
            return;
        int x, y;
        m.edge(e, x, y);
        const int o = y * a.g.pitch + x;
        float f[8], q[9], n[8];
        gather_a(a.fin, a.R, a.g, a.Pb, x, y, o, f);
        gather_g(a.gin, a.g, a.m, a.Sb, x, y, o, q);
        const float r0 = a.R[o], it = a.inv_tau[o], K = a.K[o];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            n[i] = a.fin[i][o];
        float mx, my;
        first_moment(f, mx, my);
        const float pn = node_pressure(f, r0);
        const float S = saturation_collide(a, o, mx, my, it, K, q);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            a.nout[i][o] = fmaf(wgt(i + 1), r0 - pn, n[i]);
        a.Rnew[o] = pn;
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (i < a.m.qs)
                a.gout[i][o] = q[i];
        a.S[o] = S;
        return;
    }
    const int p = a.g.pitch;
    const StepQuad s(m, b, p);
    const int o = s.o;
    float4 mx, my, pn, r0;
    PullG g;
    {
        PullA l;
        l.load(a.fin, a.R, s, p);
        g.load(a.gin, a.m.qs, s, p);
        float4 f[8];
        l.values(s, f);
        r0 = l.r[1];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float fc[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                fc[i] = at4(f[i], c);
            first_moment(fc, at4(mx, c), at4(my, c));
            at4(pn, c) = node_pressure(fc, at4(r0, c));
        }
    }
    float4 q[9];
    g.values(s, q);
    if (!s.store)
        return;
    const float4 it = ldq(a.inv_tau, o), K = ldq(a.K, o);
    float4 n[8], S;
#pragma unroll
    for (int i = 0; i < 8; ++i)                       // the node's own: in the cache, other lanes pulled them
        n[i] = ldq(a.fin[i], o);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
            at4(n[i], c) = fmaf(wgt(i + 1), at4(r0, c) - at4(pn, c), at4(n[i], c));
        stq(a.nout[i], o, n[i]);
    }
    stq(a.Rnew, o, pn);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float qc[9];
#pragma unroll
        for (int i = 0; i < 9; ++i)
            qc[i] = at4(q[i], c);
        at4(S, c) = saturation_collide(a, o + c, at4(mx, c), at4(my, c), at4(it, c), at4(K, c), qc);
#pragma unroll
        for (int i = 0; i < 9; ++i)
            at4(q[i], c) = qc[i];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i)
        if (i < a.m.qs)
            stq(a.gout[i], o, q[i]);
    stq(a.S, o, S);
}

}  // namespace lbm2p_dev
