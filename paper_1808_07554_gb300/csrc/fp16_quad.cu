// Four FP16-storage pressure sweeps (fp16.cu) per launch on lattices with walls on every side.
//
// What bounded the sub-iteration was the launch per sweep: 44 B per node and sweep through the staged
// rows, 60 us at 2048^2 where the bytes take 27.  Here, as in the FP32 form (sweep_quad.cu, whose
// tiles, halo and pipeline these are), a warp carries four sweeps of a tile of 56 columns in
// registers: 11 B per node and sweep.  Between sweeps a lane keeps the populations of its two columns
// as they would be stored, two FP16 values in a register, so every sweep rounds as the launch per
// sweep does and the results are the same bit for bit; half the registers of the FP32 form, which
// the rows of R that every sweep changes take up again.  A pull from a neighbouring column is one
// shuffle of a packed register and a byte permute.  Arithmetic is FP32 in packed pairs.
// The row loop is one row with guards for the filling sweeps: 555 instructions, two of which no longer
// fit the instruction cache nearest to the warps (unrolled by two with straight-line filling rows as
// the FP32 form is, warps waited for instructions most, 86 us).
// Four sweeps at 2048^2: 242 us in four launches, 78 us in one.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm2p_async.cuh"
#include "lbm2p_device.cuh"
#include "lbm2p_node.cuh"
#include "sweep_quad.cuh"

namespace lbm2p_dev {
namespace {

constexpr int kHalfRow = 8 * kQuadCols / 2 + 2 * kQuadCols;   // 32-bit words of a ring slot
constexpr int kHalfBlocks = 8;                                // as the FP32 form: 255 registers

__host__ __device__ constexpr size_t quad_h_smem(bool has_fp)
{
    return (size_t)kQuadSlots * (kHalfRow + (has_fp ? kQuadCols : 0)) * sizeof(float);
}

// 8 bytes global -> shared without a register round trip (four FP16 values: x0 - 4 is on 8 bytes)
__device__ __forceinline__ void cp_async_8(unsigned dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ float2 widen(unsigned v)
{
    return __half22float2(*reinterpret_cast<const __half2 *>(&v));
}

__device__ __forceinline__ unsigned narrow(float2 v)
{
    const __half2 h = __floats2half2_rn(v.x, v.y);
    return *reinterpret_cast<const unsigned *>(&h);
}

// columns x - 1, x from the pairs of this lane and the one before; x + 1, x + 2 with the one after
__device__ __forceinline__ unsigned pair_left(unsigned v)
{
    return __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);
}

__device__ __forceinline__ unsigned pair_right(unsigned v)
{
    return __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);
}

// GEN: 0 no wall and no well in the tile's footprint, 1 any; FP: a source plane is read
template <bool CHECK, bool FP, int GEN>
struct QuadH {
    static constexpr int S = kQuadSlots;
    const HalfSweepArgs &a;
    const int lane;
    const float2 s2, inv_s2;
    const __half *nin;                        // plane 0 (lanes 16-31: plane 1)
    long long ps;                             // FP16 values from plane to plane
    const float *Rit, *Fp;                    // R (lanes 16-31: 1/tau_f); F~_p
    // ---- ring ----
    const unsigned *ring;
    int off;                                  // this lane's part of the next row to copy
    unsigned dst;                             // its place in slot 0: populations,
    unsigned dstf;                            // and FP32 planes
    bool seg;
    int nrows;                                // input rows
    int q;
    int im, i0, ip;                           // rows t - 2, t - 1, t in the ring (words)
    // ---- history ----
    QuadRow rw[kQuadT + 1][3];                // R that sweep s reads: rows above, at, below its row
    float2 kp[kQuadT + 1];                    // 1 - 1/tau_f of the row of sweep s
    float2 fg[kQuadT + 1];                    // F~_p of the source plane
    unsigned c0[kQuadT], c2[kQuadT];          // sweep s's directions 1, 3 at its last row
    unsigned d1[kQuadT][2], d4[kQuadT][2], d5[kQuadT][2];   // 2, 5, 6 at its last two rows
    unsigned k3[kQuadT], k6[kQuadT], k7[kQuadT];            // 4, 7, 8 at its last row (walls)
    // ---- position ----
    int x, y, o;
    bool owner0, owner1, wl0, wr0, wr1, in0, in1;
    int wlo, whi, ylo, yhi;
    ResAcc racc;
    float nmax, shift, dshift;

    __device__ __forceinline__ QuadH(const HalfSweepArgs &a_, int lane_, float s, float inv_s)
        : a(a_), lane(lane_), s2(dup2(s)), inv_s2(dup2(inv_s))
    {
    }

    static constexpr int kSlot = kHalfRow + (FP ? kQuadCols : 0);

    __device__ __forceinline__ void issue(int slot, int k)
    {
        unsigned m = 0x3FFu;
        if (k == 0)
            m = (1u << 1) | (1u << 4) | (1u << 5) | (1u << 8);
        else if (k == nrows - 1)
            m = (1u << 3) | (1u << 6) | (1u << 7) | (1u << 8);
        const int r = ylo - kQuadT + k;
        if (seg && k < nrows && (!GEN || (r >= 0 && r < a.g.ny))) {
            const bool odd = lane >= 16;
            m >>= odd ? 1 : 0;
            const unsigned so = (unsigned)(slot * kSlot) * 4u;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (m & (1u << (2 * j)))
                    cp_async_8(dst + so + (unsigned)(2 * j * kQuadCols) * 2u, nin + 2 * j * ps + off);
            if (m & (1u << 8))
                cp_async_16(dstf + so, Rit + off);
            if (FP && !odd)
                cp_async_16(dstf + so + (unsigned)(2 * kQuadCols) * 4u, Fp + off);
        }
        cp_async_commit();
        off += a.g.pitch;
    }

    __device__ __forceinline__ unsigned at(int r, int i) const { return ring[r + i * (kQuadCols / 2)]; }
    __device__ __forceinline__ float2 atf(int r, int i) const
    {
        // r holds the lane once; an FP32 plane has two words per lane
        return *reinterpret_cast<const float2 *>(ring + r + lane + 8 * (kQuadCols / 2) + i * kQuadCols);
    }

    __device__ __forceinline__ void push_R(int s, float2 v)
    {
        rw[s][2] = rw[s][1];
        rw[s][1] = rw[s][0];
        rw[s][0].v = v;
        rw[s][0].l = __shfl_up_sync(0xffffffffu, v.y, 1);
        rw[s][0].r = __shfl_down_sync(0xffffffffu, v.x, 1);
    }

    template <int PENDING>
    __device__ __forceinline__ void next_row()
    {
        cp_async_wait<PENDING>();
        __syncwarp();
        im = i0;
        i0 = ip;
        ip = q * kSlot + lane;
        q = q + 1 == S ? 0 : q + 1;
        push_R(1, atf(ip, 0));
    }

    template <int I>
    __device__ __forceinline__ void wall(float &v, bool hit, float own, float r0, bool dir, float pb) const
    {
        if (dir)
            own = -own + 2.0f * wgt(I) * (pb - r0);
        v = hit ? own : v;
    }

    template <bool LOW>
    __device__ __forceinline__ void wall_row(float2 (&f)[8], const unsigned (&own)[8], float2 r0) const
    {
        constexpr int I = LOW ? 2 : 4, J = LOW ? 5 : 7, K = LOW ? 6 : 8, sd = LOW ? 2 : 3;
        const bool dir = a.g.bc[sd] != BC_NOFLUX;
        float pb[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (dir)
#pragma unroll
            for (int k = 0; k < 5; ++k)
                if (k < 3 ? in0 : in1)
                    pb[k] = a.Pb[sd][2 * x + k];
        const float2 oi = own_of(own, opp(I)), oj = own_of(own, opp(J)), ok = own_of(own, opp(K));
        wall<I>(f[I - 1].x, in0, oi.x, r0.x, dir, pb[1]);
        wall<I>(f[I - 1].y, in1, oi.y, r0.y, dir, pb[3]);
        wall<J>(f[J - 1].x, in0, oj.x, r0.x, dir, pb[1 - cx(J)]);
        wall<J>(f[J - 1].y, in1, oj.y, r0.y, dir, pb[3 - cx(J)]);
        wall<K>(f[K - 1].x, in0, ok.x, r0.x, dir, pb[1 - cx(K)]);
        wall<K>(f[K - 1].y, in1, ok.y, r0.y, dir, pb[3 - cx(K)]);
    }

    __device__ __forceinline__ float2 own_of(const unsigned (&own)[8], int i) const
    {
        return __fmul2_rn(widen(own[i - 1]), inv_s2);
    }

    __device__ __forceinline__ void walls(float2 (&f)[8], const unsigned (&own)[8], float2 r0, int yy) const
    {
        float pb[3] = {0.0f, 0.0f, 0.0f};
        const bool dl = wl0 && a.g.bc[0] != BC_NOFLUX;
        const bool dr = (wr0 || wr1) && a.g.bc[1] != BC_NOFLUX;
        if ((dl || dr) && yy >= 0 && yy < a.g.ny) {
            const float *t = (dl ? a.Pb[0] : a.Pb[1]) + 2 * yy;
            pb[0] = t[0];
            pb[1] = t[1];
            pb[2] = t[2];
        }
        if (yy == 0)
            wall_row<true>(f, own, r0);
        if (yy == a.g.ny - 1)
            wall_row<false>(f, own, r0);
        const float2 o1 = own_of(own, 1), o3 = own_of(own, 3), o5 = own_of(own, 5), o6 = own_of(own, 6),
                     o7 = own_of(own, 7), o8 = own_of(own, 8);
        wall<1>(f[0].x, wl0, o3.x, r0.x, dl, pb[1]);
        wall<5>(f[4].x, wl0, o7.x, r0.x, dl, pb[0]);
        wall<8>(f[7].x, wl0, o6.x, r0.x, dl, pb[2]);
        wall<3>(f[2].x, wr0, o1.x, r0.x, dr, pb[1]);
        wall<6>(f[5].x, wr0, o8.x, r0.x, dr, pb[0]);
        wall<7>(f[6].x, wr0, o5.x, r0.x, dr, pb[2]);
        wall<3>(f[2].y, wr1, o1.y, r0.y, dr, pb[1]);
        wall<6>(f[5].y, wr1, o8.y, r0.y, dr, pb[0]);
        wall<7>(f[6].y, wr1, o5.y, r0.y, dr, pb[2]);
    }

    // F~_p / 8 of sweep s's row yy
    __device__ __forceinline__ float2 source(int s, int yy) const
    {
        float2 F = FP ? fg[s] : make_float2(0.0f, 0.0f);
        if (GEN && yy >= wlo && yy <= whi)
#pragma unroll 1
            for (int w = 0; w < a.w.n; ++w) {
                const int wo = a.w.idx[w] - (yy * a.g.pitch + x);
                if (wo == 0 && in0)
                    F.x += a.w.fp[w];
                else if (wo == 1 && in1)
                    F.y += a.w.fp[w];
            }
        return make_float2(0.125f * F.x, 0.125f * F.y);
    }

    // one sweep at the pair's row from the previous one's stored values n and its R (m, c, p: rows
    // above, at, below); returns the pressure increment
    __device__ __forceinline__ float2 sweep(const unsigned (&n)[8], const QuadRow &m, const QuadRow &c,
                                            const QuadRow &p, float2 keep, float2 Fq,
                                            const unsigned (&own)[8], int yy, unsigned (&out)[8])
    {
        float2 f[8];
        float2 h = __fmul2_rn(widen(pair_left(n[0])), inv_s2);
        f[0] = make_float2(dev1(h.x, wgt(1), c.l, c.v.x), dev1(h.y, wgt(1), c.v.x, c.v.y));
        f[1] = __ffma2_rn(dup2(wgt(2)), sub2(m.v, c.v), __fmul2_rn(widen(n[1]), inv_s2));
        h = __fmul2_rn(widen(pair_right(n[2])), inv_s2);
        f[2] = make_float2(dev1(h.x, wgt(3), c.v.y, c.v.x), dev1(h.y, wgt(3), c.r, c.v.y));
        f[3] = __ffma2_rn(dup2(wgt(4)), sub2(p.v, c.v), __fmul2_rn(widen(n[3]), inv_s2));
        h = __fmul2_rn(widen(pair_left(n[4])), inv_s2);
        f[4] = make_float2(dev1(h.x, wgt(5), m.l, c.v.x), dev1(h.y, wgt(5), m.v.x, c.v.y));
        h = __fmul2_rn(widen(pair_right(n[5])), inv_s2);
        f[5] = make_float2(dev1(h.x, wgt(6), m.v.y, c.v.x), dev1(h.y, wgt(6), m.r, c.v.y));
        h = __fmul2_rn(widen(pair_right(n[6])), inv_s2);
        f[6] = make_float2(dev1(h.x, wgt(7), p.v.y, c.v.x), dev1(h.y, wgt(7), p.r, c.v.y));
        h = __fmul2_rn(widen(pair_left(n[7])), inv_s2);
        f[7] = make_float2(dev1(h.x, wgt(8), p.l, c.v.x), dev1(h.y, wgt(8), p.v.x, c.v.y));
        if (GEN)
            walls(f, own, c.v, yy);
        const float2 dP = __fmul2_rn(
            __fadd2_rn(__fadd2_rn(__fadd2_rn(f[0], f[1]), __fadd2_rn(f[2], f[3])),
                       __fadd2_rn(__fadd2_rn(f[4], f[5]), __fadd2_rn(f[6], f[7]))),
            dup2(1.8f));
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float2 e = __ffma2_rn(dup2(-wgt(i + 1)), dP, f[i]);
            out[i] = narrow(__fmul2_rn(__ffma2_rn(keep, e, Fq), s2));
        }
        return dP;
    }

    __device__ __forceinline__ void keep_row(int s, const unsigned (&v)[8])
    {
        c0[s] = v[0];
        c2[s] = v[2];
        d1[s][1] = d1[s][0];
        d4[s][1] = d4[s][0];
        d5[s][1] = d5[s][0];
        d1[s][0] = v[1];
        d4[s][0] = v[4];
        d5[s][0] = v[5];
        if (GEN) {
            k3[s] = v[3];
            k6[s] = v[6];
            k7[s] = v[7];
        }
    }

    // iteration t: the next input row, sweep 1 at the row before it, sweep s once its rows are there
    __device__ __forceinline__ void row(int t)
    {
        next_row<S - 3>();
        unsigned v[8], n[8], own[8];
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
            kp[s] = kp[s - 1];
            if (FP)
                fg[s] = fg[s - 1];
        }
        const float2 it = atf(i0, 1);
        kp[1] = make_float2(1.0f - it.x, 1.0f - it.y);
        if (FP)
            fg[1] = atf(i0, 2);
        if (GEN)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                own[i] = at(i0, i);
        const float2 dP = sweep(n, rw[1][2], rw[1][1], rw[1][0], kp[1], source(1, y), own, y, v);
        __syncwarp();
        issue(q >= 3 ? q - 3 : q + S - 3, t + S);
        next_sweep<2>(t, v, dP);
        ++y;
    }

    // sweep s of iteration t from sweep s - 1's row v (pressure increment dPp), then the next
    template <int s>
    __device__ __forceinline__ void next_sweep(int t, const unsigned (&v)[8], float2 dPp)
    {
        push_R(s, __fadd2_rn(rw[s - 1][1].v, dPp));
        if (t < 2 * (s - 1)) {
            keep_row(s - 1, v);
            return;
        }
        unsigned n[8], own[8], w[8];
        n[0] = c0[s - 1];
        n[1] = d1[s - 1][1];
        n[2] = c2[s - 1];
        n[3] = v[3];
        n[4] = d4[s - 1][1];
        n[5] = d5[s - 1][1];
        n[6] = v[6];
        n[7] = v[7];
        if (GEN) {
            own[0] = c0[s - 1];
            own[1] = d1[s - 1][0];
            own[2] = c2[s - 1];
            own[3] = k3[s - 1];
            own[4] = d4[s - 1][0];
            own[5] = d5[s - 1][0];
            own[6] = k6[s - 1];
            own[7] = k7[s - 1];
        }
        const int yy = y - s + 1;
        const float2 dP = sweep(n, rw[s][2], rw[s][1], rw[s][0], kp[s], source(s, yy), own, yy, w);
        keep_row(s - 1, v);
        if constexpr (s < kQuadT) {
            next_sweep<s + 1>(t, w, dP);
        } else {
            const bool rowin = !GEN || (yy >= ylo && yy < yhi);
            const float2 Rn = __fadd2_rn(rw[s][1].v, dP);
            if (rowin && owner1) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    *reinterpret_cast<unsigned *>(a.nout[i] + o) = w[i];
                *reinterpret_cast<float2 *>(a.Rout + o) = Rn;
            } else if (GEN && rowin && owner0) {
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    a.nout[i][o] = __ushort_as_half((unsigned short)(w[i] & 0xffffu));
                a.Rout[o] = Rn.x;
            }
            if (CHECK && rowin) {
                if (owner0)
                    racc.add(dP.x - dshift, (rw[s][1].v.x - shift) + dP.x);
                if (owner1)
                    racc.add(dP.y - dshift, (rw[s][1].v.y - shift) + dP.y);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float2 h = widen(w[i]);
                    if (owner0)
                        nmax = fmaxf(nmax, fabsf(h.x));
                    if (owner1)
                        nmax = fmaxf(nmax, fabsf(h.y));
                }
            }
            o += a.g.pitch;
        }
    }

    // the tile's columns [x0, x0 + 56) and rows [y0, y1), from input rows y0 - 4 .. y1 + 3
    __device__ __forceinline__ void tile(int x0, int y0, int y1, unsigned *smem, int wlo_, int whi_)
    {
        const Geom &g = a.g;
        const bool odd = lane >= 16;
        nin = odd ? a.nin[1] : a.nin[0];
        ps = a.nin[1] - a.nin[0];
        Rit = odd ? a.inv_tau : a.Rin;
        Fp = a.Fp;
        ring = smem;
        const int xs = x0 - kQuadHalo;
        const int xc = xs + 4 * (lane & 15);
        seg = xc >= 0 && xc < g.pitch;
        nrows = y1 - y0 + 2 * kQuadT;
        off = (y0 - kQuadT) * g.pitch + xc;
        dst = smem_u32(smem) + (unsigned)(odd ? kQuadCols : 0) * 2u + 8u * (unsigned)(lane & 15);
        dstf = smem_u32(smem) + (unsigned)(8 * (kQuadCols / 2) + (odd ? kQuadCols : 0) + 4 * (lane & 15)) * 4u;
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
        nmax = 0.0f;
        for (int s = 0; s < S; ++s)
            issue(s, s);
        next_row<S - 1>();
        next_row<S - 2>();
        const int iters = y1 - y0 + 2 * (kQuadT - 1);
#pragma unroll 1
        for (int t = 0; t < iters; ++t)
            row(t);
        cp_async_wait<0>();
        __syncwarp();
    }
};

// one tile (QuadPlan) per block of one warp
template <bool CHECK>
__global__ void __launch_bounds__(32, kHalfBlocks)
    k_pressure_quad_h(const __grid_constant__ HalfSweepArgs a, int H)
{
    extern __shared__ __align__(128) unsigned smem_h[];
    const Geom &g = a.g;
    const int lane = threadIdx.x;
    int strip, y0, y1;
    QuadPlan(H, g.nx, g.ny).at(blockIdx.x, strip, y0, y1);
    const int x0 = strip * kQuadOwn;
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
    ResAcc racc;
    float nmax = 0.0f;
    const float s = a.scale[0], inv_s = a.scale[1];
    auto go = [&](auto fp, auto gen) {
        QuadH<CHECK, decltype(fp)::value != 0, decltype(gen)::value> t(a, lane, s, inv_s);
        t.tile(x0, y0, y1, smem_h, wlo, whi);
        racc = t.racc;
        nmax = t.nmax;
    };
    const bool gen = !inside || wlo <= whi;
    if (!gen && !a.Fp)
        go(Int<0>(), Int<0>());
    else if (!gen)
        go(Int<1>(), Int<0>());
    else if (!a.Fp)
        go(Int<0>(), Int<1>());
    else
        go(Int<1>(), Int<1>());
    if (CHECK) {
#pragma unroll
        for (int sh = 16; sh > 0; sh >>= 1)
            nmax = fmaxf(nmax, __shfl_xor_sync(0xffffffffu, nmax, sh));
        double v[4];
        racc.warp_totals(v);
        if (lane == 0) {
            for (int c = 0; c < 4; ++c)
                a.partials[4 * (size_t)blockIdx.x + c] = v[c];
            atomicMax(reinterpret_cast<unsigned int *>(&a.scale_out[3]), __float_as_uint(nmax));
        }
    }
}

void *quad_h_func(bool check)
{
    return check ? (void *)k_pressure_quad_h<true> : (void *)k_pressure_quad_h<false>;
}

}  // namespace
}  // namespace lbm2p_dev

namespace lbm2p_launch {

using namespace lbm2p_dev;

int quad_h_slots(bool has_fp)
{
    int dev = 0, sms = 0, lo = 1 << 30;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    for (bool c : {false, true}) {
        int b = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, quad_h_func(c), 32, quad_h_smem(has_fp)) !=
            cudaSuccess)
            return 0;
        lo = b < lo ? b : lo;
    }
    return lo * sms;
}

void pressure_sweeps_quad_h(const HalfSweepArgs &a, bool check, int H, int grid, void *stream)
{
    void *args[] = {(void *)&a, (void *)&H};
    cudaLaunchKernel(quad_h_func(check), dim3((unsigned)grid), dim3(32), args,
                     quad_h_smem(a.Fp != nullptr), reinterpret_cast<cudaStream_t>(stream));
}

}  // namespace lbm2p_launch
