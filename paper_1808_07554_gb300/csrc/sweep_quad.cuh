// One warp's tile of the four-sweep pressure kernel (see sweep_quad.cu), shared by the
// single-lattice launch and the batched one.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "lbm2p_async.cuh"
#include "lbm2p_device.cuh"
#include "lbm2p_node.cuh"

namespace lbm2p_dev {

constexpr int kQuadT = 4;                     // sweeps per launch
constexpr int kQuadCols = 64;                 // columns of a warp: two per lane
constexpr int kQuadHalo = 4;                  // columns on each side that it does not own
constexpr int kQuadOwn = kQuadCols - 2 * kQuadHalo;
constexpr int kQuadThreads = 32;              // a block is one warp with one tile
constexpr int kQuadBlocks = 8;                // blocks per SM: two warps per scheduler, 255 registers
constexpr int kQuadSlots = 7;                 // ring slots: rows in flight = slots - 3

__host__ __device__ constexpr int quad_strips(int nx) { return (nx + kQuadOwn - 1) / kQuadOwn; }

// The tiles of a lattice: strips of 56 columns by H rows, lower where the footprint meets a wall.
// The row of an edge tile took 1.4 times an interior one's, so with one height the edge tiles ended
// last: 1024^2 in one round of resident tiles 27 us of which the interior tiles ran 17.  He rows make
// an edge tile last as long as an interior one (the 8 rows of filling and draining counted in), and
// the edge tiles come first, so that the tail of a launch of several rounds is made of short ones:
// 22 us at 1024^2, 231 -> 218 us at 4096^2 (19.4 and 221 since the edge path sums a node's wells first,
// which made its code shorter).
struct QuadPlan {
    int H, He, Hb;               // rows of interior tiles, of those on x walls, on y walls
    int first;                   // strips 1 .. first - 1 meet no x wall
    int ne, ni;                  // strips on x walls, others
    int nce, nci;                // tiles of a strip on an x wall, of another one
    int ny;

    __host__ __device__ QuadPlan(int H_, int nx, int ny_) : H(H_), ny(ny_)
    {
        const int strips = quad_strips(nx);
        He = 5 * (H + 2 * kQuadT) / 7 - 2 * kQuadT;
        He = He < 2 ? 2 : He;
        He = He < H ? He : H;
        Hb = He > kQuadT ? He : kQuadT;
        // strip s reads column 56 s + 58 in its first sweep
        const int e = kQuadOwn + kQuadT;
        first = nx >= e ? (nx - e) / kQuadOwn + 1 : 1;
        first = first < strips ? first : strips;
        ni = first - 1;
        ne = strips - ni;
        nce = (ny + He - 1) / He;
        const int mid = ny - 2 * Hb;
        nci = ny <= Hb ? 1 : 2 + (mid > 0 ? (mid + H - 1) / H : 0);
    }
    __host__ __device__ long long tiles() const { return (long long)ne * nce + (long long)ni * nci; }
    // strip and rows [y0, y1) of tile t
    __host__ __device__ void at(int t, int &strip, int &y0, int &y1) const
    {
        if (t < ne * nce) {
            const int c = t / ne, s = t - c * ne;
            strip = s ? first - 1 + s : 0;
            y0 = c * He;
            y1 = y0 + He < ny ? y0 + He : ny;
            return;
        }
        t -= ne * nce;
        const int c = t / ni;
        strip = 1 + t - c * ni;
        if (c == 0) {                                 // the low y wall
            y0 = 0;
            y1 = Hb < ny ? Hb : ny;
        } else if (c == 1) {                          // the high y wall
            y0 = ny - Hb > Hb ? ny - Hb : Hb;
            y1 = ny;
        } else {
            y0 = Hb + (c - 2) * H;
            y1 = y0 + H < ny - Hb ? y0 + H : ny - Hb;
        }
    }
};

inline size_t quad_smem_bytes(bool has_fp)
{
    return (size_t)kQuadSlots * (has_fp ? 11 : 10) * kQuadCols * sizeof(float);
}

// 16 bytes global -> shared without a register round trip
__device__ __forceinline__ void cp_async_16(unsigned dst, const float *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int PENDING>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long d, x = *reinterpret_cast<unsigned long long *>(&a),
                          y = *reinterpret_cast<unsigned long long *>(&b);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(x), "l"(y));
    return *reinterpret_cast<float2 *>(&d);
}

__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }

template <int V>
struct Int {
    static constexpr int value = V;
};

// R of one row at a lane's columns x, x + 1 and the columns beside them
struct QuadRow {
    float l;                                  // column x - 1
    float2 v;                                 // columns x, x + 1
    float r;                                  // column x + 2
};

// FQ: there is a source in the tile; GEN: 0 no wall in the tile's footprint, 1 no-flux walls, 2 walls
// of both kinds; UNROLL: rows unrolled by two, the filling rows as straight-line code (GEN 0 only)
template <bool CHECK, bool FQ, int GEN, int S, bool UNROLL>
struct Quad {
    const PressureArgs &a;
    const int lane;
    // planes, kept here: a batched launch has its argument blocks in global memory
    const float *fin, *R, *itau;
    float *fout;
    long long ps;                             // floats from plane to plane
    int pitch;
    // ---- ring ----
    float *ring;
    int slot_floats;
    int off;                                  // this lane's 16 bytes of the next row to copy
    unsigned dst;                             // their place in slot 0 (shared address)
    bool seg;                                 // inside the row
    int nin;                                  // input rows
    int q;                                    // slot of the next row to wait for
    int im, i0, ip;                           // rows t - 2, t - 1, t in the ring (this lane's columns)
    // ---- history ----
    QuadRow rg[6];                            // R, newest row first
    float2 ig[kQuadT + 1];                    // -1/tau_f of the row of sweep s
    float2 fg[kQuadT + 1];                    // F~_p / 8
    float2 c0[kQuadT], c2[kQuadT];            // sweep s's directions 1, 3 at its last row
    float2 d1[kQuadT][2], d4[kQuadT][2], d5[kQuadT][2];   // 2, 5, 6 at its last two rows
    float2 k3[kQuadT], k6[kQuadT], k7[kQuadT];            // 4, 7, 8 at its last row (walls)
    float2 pd;                                // sweep 3's pressure increment at its last row
    // ---- position ----
    int x;                                    // this lane's first column
    int y;                                    // row of sweep 1 in the current iteration
    int o;                                    // offset of the last sweep's node
    bool owner0, owner1;                      // this lane stores column x, x + 1
    bool wl0, wr0, wr1;                       // column x on the low, x or x + 1 on the high x wall
    int wlo, whi;                             // rows of the tile's wells (wlo > whi: none)
    bool in0, in1;                            // column x (x + 1) is in the lattice
    int ylo, yhi;                             // rows that the tile stores
    ResAcc racc;
    float shift, dshift;

    __device__ __forceinline__ Quad(const PressureArgs &a_, int lane_) : a(a_), lane(lane_) {}

    // Copies of the next input row into slot `slot`, 16 bytes per lane and instruction: lanes
    // 0-15 the segment of an even plane, lanes 16-31 that of the next odd one.  The first row
    // feeds only the c_y = +1 pulls of the row above it, the last only the c_y = -1 pulls of the
    // row below; nothing is copied of rows and columns outside the lattice.
    __device__ __forceinline__ void issue(int slot, int k)
    {
        unsigned m = 0x3FFu;
        if (k == 0)
            m = (1u << 1) | (1u << 4) | (1u << 5) | (1u << 8);
        else if (k == nin - 1)
            m = (1u << 3) | (1u << 6) | (1u << 7) | (1u << 8);
        const int r = ylo - kQuadT + k;
        if (seg && k < nin && (!GEN || (r >= 0 && r < a.g.ny))) {
            const bool odd = lane >= 16;
            m >>= odd ? 1 : 0;
            const unsigned d = dst + (unsigned)(slot * slot_floats) * 4u;
            const float *f = fin + (odd ? ps : 0) + off;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (m & (1u << (2 * j)))
                    cp_async_16(d + (unsigned)(2 * j * kQuadCols) * 4u, f + 2 * j * ps);
            if (m & (1u << 8))
                cp_async_16(d + (unsigned)(8 * kQuadCols) * 4u, (odd ? itau : R) + off);
            if (FQ && a.Fp && !odd)
                cp_async_16(d + (unsigned)(10 * kQuadCols) * 4u, a.Fp + off);
        }
        cp_async_commit();
        off += pitch;
    }

    // input row t (the next one) is in place; PENDING: copies of later rows that may be in flight
    template <int PENDING>
    __device__ __forceinline__ void next_row()
    {
        cp_async_wait<PENDING>();
        __syncwarp();
        im = i0;
        i0 = ip;
        ip = q * slot_floats + 2 * lane;
        q = q + 1 == S ? 0 : q + 1;
#pragma unroll
        for (int i = 5; i > 0; --i)
            rg[i] = rg[i - 1];
        const float2 v = *reinterpret_cast<const float2 *>(ring + ip + 8 * kQuadCols);
        rg[0].v = v;
        rg[0].l = __shfl_up_sync(0xffffffffu, v.y, 1);
        rg[0].r = __shfl_down_sync(0xffffffffu, v.x, 1);
    }

    // The wall rules of Sec. 4 at the lane's columns in row yy: a link that crosses a wall takes
    // the node's own value of the opposite direction (bounce-back), or its negative plus
    // 2 w (P_b - R) (anti-bounce-back, where `dir`).  x sides last, since a corner's links use
    // the x-side.  With no-flux walls this is one select per link and column; the wall values of
    // an x side are three per row and lane, loaded together.
    template <int I>
    __device__ __forceinline__ void wall(float &v, bool hit, float own, float r0, bool dir, float pb) const
    {
        if (GEN == 2 && dir)
            own = -own + 2.0f * wgt(I) * (pb - r0);
        v = hit ? own : v;
    }

    // links 2, 5, 6 from below (LOW) or 4, 7, 8 from above of a row on a y wall
    template <bool LOW>
    __device__ __forceinline__ void wall_row(float2 (&f)[8], const float2 (&own)[8], float2 r0) const
    {
        constexpr int I = LOW ? 2 : 4, J = LOW ? 5 : 7, K = LOW ? 6 : 8, sd = LOW ? 2 : 3;
        const bool dir = GEN == 2 && a.g.bc[sd] != BC_NOFLUX;
        float pb[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};     // trace at k0 - 1 .. k0 + 3
        if (dir)
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (k < 3 ? in0 : in1)
                    pb[k] = a.Pb[sd][2 * x + k];
        wall<I>(f[I - 1].x, in0, own[opp(I) - 1].x, r0.x, dir, pb[1]);
        wall<I>(f[I - 1].y, in1, own[opp(I) - 1].y, r0.y, dir, pb[3]);
        wall<J>(f[J - 1].x, in0, own[opp(J) - 1].x, r0.x, dir, pb[1 - cx(J)]);
        wall<J>(f[J - 1].y, in1, own[opp(J) - 1].y, r0.y, dir, pb[3 - cx(J)]);
        wall<K>(f[K - 1].x, in0, own[opp(K) - 1].x, r0.x, dir, pb[1 - cx(K)]);
        wall<K>(f[K - 1].y, in1, own[opp(K) - 1].y, r0.y, dir, pb[3 - cx(K)]);
    }

    __device__ __forceinline__ void walls(float2 (&f)[8], const float2 (&own)[8], float2 r0, int yy) const
    {
        float pb[3] = {0.0f, 0.0f, 0.0f};                 // trace at k - 1, k, k + 1
        const bool dl = GEN == 2 && wl0 && a.g.bc[0] != BC_NOFLUX;
        const bool dr = GEN == 2 && (wr0 || wr1) && a.g.bc[1] != BC_NOFLUX;
        if (GEN == 2 && (dl || dr) && yy >= 0 && yy < a.g.ny) {
            const float *t = (dl ? a.Pb[0] : a.Pb[1]) + 2 * yy;
            pb[0] = t[0];
            pb[1] = t[1];
            pb[2] = t[2];
        }
        if (yy == 0)
            wall_row<true>(f, own, r0);
        if (yy == a.g.ny - 1)
            wall_row<false>(f, own, r0);
        wall<1>(f[0].x, wl0, own[2].x, r0.x, dl, pb[1]);
        wall<5>(f[4].x, wl0, own[6].x, r0.x, dl, pb[0]);
        wall<8>(f[7].x, wl0, own[5].x, r0.x, dl, pb[2]);
        wall<3>(f[2].x, wr0, own[0].x, r0.x, dr, pb[1]);
        wall<6>(f[5].x, wr0, own[7].x, r0.x, dr, pb[0]);
        wall<7>(f[6].x, wr0, own[4].x, r0.x, dr, pb[2]);
        wall<3>(f[2].y, wr1, own[0].y, r0.y, dr, pb[1]);
        wall<6>(f[5].y, wr1, own[7].y, r0.y, dr, pb[0]);
        wall<7>(f[6].y, wr1, own[4].y, r0.y, dr, pb[2]);
    }

    // one sweep at the pair's row from the previous sweep's values n (own columns) in the rows
    // above, at and below, and R of those rows (m, c, p); own: the node's values in all
    // directions (wall rules).  Returns the pressure increment.
    __device__ __forceinline__ float2 sweep(const float2 (&n)[8], const QuadRow &m, const QuadRow &c,
                                            const QuadRow &p, float2 nit, float2 Fq,
                                            const float2 (&own)[8], int yy, float2 (&out)[8])
    {
        // a_i = n_i(x - c_i) + w_i (R(x - c_i) - R(x))
        const float l0 = __shfl_up_sync(0xffffffffu, n[0].y, 1);
        const float r2 = __shfl_down_sync(0xffffffffu, n[2].x, 1);
        const float l4 = __shfl_up_sync(0xffffffffu, n[4].y, 1);
        const float r5 = __shfl_down_sync(0xffffffffu, n[5].x, 1);
        const float r6 = __shfl_down_sync(0xffffffffu, n[6].x, 1);
        const float l7 = __shfl_up_sync(0xffffffffu, n[7].y, 1);
        float2 f[8];
        f[1] = __ffma2_rn(dup2(wgt(2)), sub2(m.v, c.v), n[1]);
        f[3] = __ffma2_rn(dup2(wgt(4)), sub2(p.v, c.v), n[3]);
        const float e = c.v.y - c.v.x;
        f[0] = make_float2(dev1(l0, wgt(1), c.l, c.v.x), fmaf(wgt(1), -e, n[0].x));
        f[2] = make_float2(fmaf(wgt(3), e, n[2].y), dev1(r2, wgt(3), c.r, c.v.y));
        f[4] = make_float2(dev1(l4, wgt(5), m.l, c.v.x), dev1(n[4].x, wgt(5), m.v.x, c.v.y));
        f[5] = make_float2(dev1(n[5].y, wgt(6), m.v.y, c.v.x), dev1(r5, wgt(6), m.r, c.v.y));
        f[6] = make_float2(dev1(n[6].y, wgt(7), p.v.y, c.v.x), dev1(r6, wgt(7), p.r, c.v.y));
        f[7] = make_float2(dev1(l7, wgt(8), p.l, c.v.x), dev1(n[7].x, wgt(8), p.v.x, c.v.y));
        if (GEN)
            walls(f, own, c.v, yy);
        const float2 dP = __fmul2_rn(
            __fadd2_rn(__fadd2_rn(__fadd2_rn(f[0], f[1]), __fadd2_rn(f[2], f[3])),
                       __fadd2_rn(__fadd2_rn(f[4], f[5]), __fadd2_rn(f[6], f[7]))),
            dup2(1.8f));
        // a + (w dP - a) / tau_f + F / 8 with both products negated (exact)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            out[i] = __ffma2_rn(__ffma2_rn(dup2(-wgt(i + 1)), dP, f[i]), nit, f[i]);
            if (FQ)
                out[i] = __fadd2_rn(out[i], Fq);
        }
        return dP;
    }

    // the sources of the tile's wells in row yy, where no source plane is read (rare); those of one
    // node are added up before they are rounded into its populations, as in the single sweep
    __device__ __forceinline__ void add_wells(float2 (&v)[8], int yy) const
    {
        float2 F = make_float2(0.0f, 0.0f);
#pragma unroll 1
        for (int w = 0; w < a.w.n; ++w) {
            const int wo = a.w.idx[w] - (yy * a.g.pitch + x);
            if (wo == 0 && in0)
                F.x += a.w.fp[w];
            else if (wo == 1 && in1)
                F.y += a.w.fp[w];
        }
        F = __fmul2_rn(dup2(0.125f), F);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            v[i] = __fadd2_rn(v[i], F);
    }

    // directions 2, 5, 6 of two rows: in sets indexed by the row's parity P where the row loop is
    // unrolled by two, else moved on from row to row (edge tiles: half the code)
    static constexpr int NP = GEN || !UNROLL ? 1 : 2;

    // what sweep s + 1 will need of sweep s's row
    template <int P>
    __device__ __forceinline__ void keep(int s, const float2 (&v)[8])
    {
        c0[s] = v[0];
        c2[s] = v[2];
        if (NP == 1) {
            d1[s][1] = d1[s][0];
            d4[s][1] = d4[s][0];
            d5[s][1] = d5[s][0];
        }
        constexpr int at = NP == 2 ? P : 0;
        d1[s][at] = v[1];
        d4[s][at] = v[4];
        d5[s][at] = v[5];
        if (GEN) {
            k3[s] = v[3];
            k6[s] = v[6];
            k7[s] = v[7];
        }
    }

    // Iteration t: the next input row arrives, sweep 1 at the row before it, sweep s another s - 1
    // rows back once the rows that it needs are there (t >= 2 (s - 1)); P: the row's parity
    template <int P, int NS>
    __device__ __forceinline__ void row(int t)
    {
        next_row<S - 3>();
        float2 v[8], n[8], own[8];
        auto at = [&](int r, int i) {
            return *reinterpret_cast<const float2 *>(ring + r + i * kQuadCols);
        };
        n[0] = at(i0, 0);
        n[1] = at(im, 1);
        n[2] = at(i0, 2);
        n[3] = at(ip, 3);
        n[4] = at(im, 4);
        n[5] = at(im, 5);
        n[6] = at(ip, 6);
        n[7] = at(ip, 7);
#pragma unroll
        for (int s = kQuadT; s > 1; --s) {
            ig[s] = ig[s - 1];
            if (FQ)
                fg[s] = fg[s - 1];
        }
        const float2 it = at(i0, 9);
        ig[1] = make_float2(-it.x, -it.y);
        if (FQ) {
            float2 F = make_float2(0.0f, 0.0f);
            if (a.Fp)
                F = at(i0, 10);
            if (GEN && y >= wlo && y <= whi)
                for (int w = 0; w < a.w.n; ++w) {
                    const int wo = a.w.idx[w] - (y * a.g.pitch + x);
                    if (wo == 0 && in0)
                        F.x += a.w.fp[w];
                    else if (wo == 1 && in1)
                        F.y += a.w.fp[w];
                }
            fg[1] = make_float2(0.125f * F.x, 0.125f * F.y);   // w_bar_i = 1/8 (Eq. 3-5a)
        }
        if (GEN)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                own[i] = at(i0, i);
        float2 dPp = sweep(n, rg[2], rg[1], rg[0], ig[1], fg[1], own, y, v);
        if (GEN == 1 && y >= wlo && y <= whi)
            add_wells(v, y);
        __syncwarp();
        // every lane is done with row t - 2, whose slot is two before the one just read
        issue(q >= 3 ? q - 3 : q + S - 3, t + S);
        next_sweep<P, NS, 2>(t, v, dPp);
        ++y;
    }

    // sweep s of iteration t from sweep s - 1's row v (pressure increments dPp), then the next
    template <int P, int NS, int s>
    __device__ __forceinline__ void next_sweep(int t, const float2 (&v)[8], float2 dPp)
    {
        if (s > NS || (NP == 1 && t < 2 * (s - 1))) {
            keep<P>(s - 1, v);
            if (CHECK && s == kQuadT)
                pd = dPp;
            return;
        }
        constexpr int older = NP == 2 ? P : 1, newer = NP == 2 ? 1 - P : 0;
        float2 n[8], own[8], w[8];
        n[0] = c0[s - 1];
        n[1] = d1[s - 1][older];
        n[2] = c2[s - 1];
        n[3] = v[3];
        n[4] = d4[s - 1][older];
        n[5] = d5[s - 1][older];
        n[6] = v[6];
        n[7] = v[7];
        if (GEN) {
            own[0] = c0[s - 1];
            own[1] = d1[s - 1][newer];
            own[2] = c2[s - 1];
            own[3] = k3[s - 1];
            own[4] = d4[s - 1][newer];
            own[5] = d5[s - 1][newer];
            own[6] = k6[s - 1];
            own[7] = k7[s - 1];
        }
        const float2 dP = sweep(n, rg[s + 1], rg[s], rg[s - 1], ig[s], fg[s], own, y - s + 1, w);
        keep<P>(s - 1, v);
        if (GEN == 1 && y - s + 1 >= wlo && y - s + 1 <= whi)
            add_wells(w, y - s + 1);
        if constexpr (s < kQuadT) {
            next_sweep<P, NS, s + 1>(t, w, dP);
        } else {
            const int y4 = y - s + 1;
            const bool rowin = !GEN || (y4 >= ylo && y4 < yhi);
            if (!GEN) {
                if (owner0)
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        *reinterpret_cast<float2 *>(fout + i * ps + o) = w[i];
            } else if (rowin) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (owner0)
                        fout[i * ps + o] = w[i].x;
                    if (owner1)
                        fout[i * ps + o + 1] = w[i].y;
                }
            }
            if (CHECK) {
                if (rowin && owner0)
                    racc.add((dP.x - pd.x) - dshift, (rg[s].v.x - shift) + dP.x);
                if (rowin && owner1)
                    racc.add((dP.y - pd.y) - dshift, (rg[s].v.y - shift) + dP.y);
                pd = dPp;
            }
            o += pitch;
        }
    }

    // the tile's columns [x0, x0 + 56) and rows [y0, y1), from input rows y0 - 4 .. y1 + 3
    __device__ __forceinline__ void tile(int x0, int y0, int y1, float *smem, int wlo_, int whi_)
    {
        const Geom &g = a.g;
        fin = a.fin[0];
        fout = a.fout[0];
        ps = a.fin[1] - a.fin[0];
        R = a.R;
        itau = a.inv_tau;
        pitch = g.pitch;
        ring = smem;
        slot_floats = (a.Fp ? 11 : 10) * kQuadCols;
        const int xs = x0 - kQuadHalo;                 // column of lane 0
        const int xc = xs + 4 * (lane & 15);           // this lane's 16 bytes
        seg = xc >= 0 && xc < g.pitch;
        nin = y1 - y0 + 2 * kQuadT;
        off = (y0 - kQuadT) * g.pitch + xc;
        dst = smem_u32(ring + (lane >> 4) * kQuadCols + 4 * (lane & 15));
        q = 0;
        im = i0 = ip = 0;
        x = xs + 2 * lane;
        y = y0 - kQuadT + 1;
        o = y0 * g.pitch + x;
        ylo = y0;
        yhi = y1;
        const bool own = lane >= kQuadHalo / 2 && lane < 32 - kQuadHalo / 2;
        owner0 = own && (!GEN || x < g.nx);
        owner1 = own && (!GEN || x + 1 < g.nx);
        if (GEN) {
            wl0 = x == 0;
            wr0 = x == g.nx - 1;
            wr1 = x + 1 == g.nx - 1;
            wlo = wlo_;
            whi = whi_;
            in0 = x >= 0 && x < g.nx;
            in1 = x + 1 >= 0 && x + 1 < g.nx;
        }
        shift = CHECK ? a.shift[0] : 0.0f;
        dshift = CHECK ? a.shift[1] : 0.0f;
        for (int s = 0; s < S; ++s)
            issue(s, s);
        next_row<S - 1>();
        next_row<S - 2>();
        const int iters = y1 - y0 + 2 * (kQuadT - 1);
        if (NP == 1) {
#pragma unroll 1
            for (int t = 0; t < iters; ++t)
                row<0, kQuadT>(t);
        } else {
            row<0, 1>(0);
            row<1, 1>(1);
            row<0, 2>(2);
            row<1, 2>(3);
            row<0, 3>(4);
            row<1, 3>(5);
            int t = 6;
            for (; t + 1 < iters; t += 2) {
                row<0, 4>(t);
                row<1, 4>(t + 1);
            }
            if (t < iters)
                row<0, 4>(t);
        }
        cp_async_wait<0>();
        __syncwarp();
    }
};

// Tile `tile` of the lattice of `a` (QuadPlan); every lane of the warp calls it with the warp's own
// shared memory.
template <bool CHECK, int S, bool UNROLL>
__device__ __forceinline__ void quad_tile(const PressureArgs &a, int H, int tile, float *smem,
                                          int lane, ResAcc &racc)
{
    const Geom &g = a.g;
    int strip, y0, y1;
    QuadPlan(H, g.nx, g.ny).at(tile, strip, y0, y1);
    const int x0 = strip * kQuadOwn;
    // sweep 1 runs on columns x0 - 3 .. x0 + 58 and rows y0 - 3 .. y1 + 2: no wall node and no
    // well among them?
    constexpr int e = kQuadT - 1;
    const bool inside = x0 - e >= 1 && x0 + kQuadOwn - 1 + e <= g.nx - 2 && y0 - e >= 1 &&
                        y1 - 1 + e <= g.ny - 2;
    int wlo = g.ny, whi = -1;
    for (int w = 0; w < a.w.n; ++w) {
        const int wy = a.w.idx[w] / g.pitch, wx = a.w.idx[w] - wy * g.pitch;
        if (wx >= x0 - e && wx <= x0 + kQuadOwn - 1 + e && wy >= y0 - e && wy <= y1 - 1 + e) {
            wlo = wy < wlo ? wy : wlo;
            whi = wy > whi ? wy : whi;
        }
    }
    const bool well = wlo <= whi;
    bool dir = false;
    for (int sd = 0; sd < 4; ++sd)
        dir = dir || g.bc[sd] != BC_NOFLUX;
    auto go = [&](auto fq, auto gen) {
        Quad<CHECK, decltype(fq)::value, decltype(gen)::value, S, UNROLL> t(a, lane);
        t.tile(x0, y0, y1, smem, wlo, whi);
        racc = t.racc;
    };
    if (inside && !well && !a.Fp)
        go(Int<0>(), Int<0>());
    else if (inside && !well)
        go(Int<1>(), Int<0>());
    else if (!dir && !a.Fp)
        go(Int<0>(), Int<1>());
    else
        go(Int<1>(), Int<2>());
}

}  // namespace lbm2p_dev
