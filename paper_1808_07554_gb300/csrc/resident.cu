// A whole pressure sub-iteration (Sec. 3: Eq. 3-1 swept until the stopping rule is met) in one
// launch, for lattices small enough to stay on chip: a thread-block cluster holds the populations
// in its shared memory from the first sweep to the last.
//
// A small lattice is bound by launches, not by its nodes: a 64^2 sweep took 4.1 us as a kernel of
// its own, and each residual check another 12 us for the reduction and the conditional graph nodes
// around it.  Here a sweep is one pass over shared memory and one cluster barrier, and the check is
// a reduction across the cluster that every block evaluates for itself.
//
// Block r of the cluster owns rows [r h, (r + 1) h), one to three nodes per thread, in two buffers
// of eight planes with a border of one ghost cell.  Every pull of every node is then the same plain
// read of a neighbouring cell: what differs between an interior node, a wall, a periodic side and a
// row of the next block is put where it is written.  The node that computes an outgoing value also
// stores it into the one ghost cell that is read in its place: in the block that owns the reader
// (through distributed shared memory), or its own on a wall, where the reader is the node itself in
// the opposite direction (bounce-back; with its sign changed for anti-bounce-back).  The targets
// are a table of eight addresses per node on the border of a block's rows.  The term that a pull
// adds, w_i (R(x - c_i) - R(x)), or 2 w_i (P_b - R(x)) at a Dirichlet wall, or nothing, does not
// change between rebases and is kept per direction in registers as the factor of w_i.
//
// Measured, 16 blocks: 64^2 0.7 us per sweep and 1.7 us per check (before 4.1 us per sweep as a
// launch of its own, or 2.9 as a quarter of a four-sweep launch, and 10 to 12 us per check with the
// finalize kernel and the graph's conditional nodes); 128^2 1.2 us per sweep and 2.3 per check.  What
// bounds it now is the cluster barrier with the distributed stores before it (about 0.5 us) and, at
// 128^2, one node per thread on 32 warps.  The check's sums are FP32 inside a warp and FP64 in one warp
// per block, and its test a product instead of a division and a root: with FP64 in every warp it took
// 6.8 us at 64^2 and 10.4 us at 128^2, all of it the few FP64 units.
//
// Per node the arithmetic is that of the single sweep (dev1, pressure_of, collide1; the factor 2 of
// a Dirichlet wall is exact), so a solve equals the same number of single sweeps bit for bit; the
// residual differs from theirs only in the grouping of its sums.  All blocks compute the stopping
// test from the same sums in the same order, so they leave the loop together.
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm2p_async.cuh"
#include "lbm2p_device.cuh"
#include "lbm2p_node.cuh"
#include "residual.cuh"

namespace lbm2p_dev {
namespace {

constexpr int kResMaxThreads = 1024;
constexpr int kResMaxNpt = 3;

struct ResidentShape {
    int C, h, cells, edges, npt, threads;
    size_t smem;
};

__device__ __forceinline__ void cluster_store(unsigned a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

__device__ __forceinline__ double cluster_load(unsigned a)
{
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

__device__ __forceinline__ float flip(float v, bool f)
{
    return __uint_as_float(__float_as_uint(v) ^ (f ? 0x80000000u : 0u));
}

// where the link from (x, y) by (dx, dy) ends: a node (wrapped on periodic sides; returns -1), or
// the wall it crosses (the side; x sides first)
__device__ __forceinline__ int link_end(const Geom &g, int x, int y, int dx, int dy, int &xe, int &ye)
{
    xe = x + dx;
    ye = y + dy;
    int side = -1;
    if (xe < 0 || xe >= g.nx) {
        const int sd = xe < 0 ? 0 : 1;
        if (g.bc[sd] == BC_PERIODIC)
            xe += xe < 0 ? g.nx : -g.nx;
        else
            side = sd;
    }
    if (side < 0 && (ye < 0 || ye >= g.ny)) {
        const int sd = ye < 0 ? 2 : 3;
        if (g.bc[sd] == BC_PERIODIC)
            ye += ye < 0 ? g.ny : -g.ny;
        else
            side = sd;
    }
    return side;
}

template <int NPT>
struct ResNode {
    float D[8];                   // factor of w_i in the pull of direction i + 1
    float it, Fq, r0, dp;         // 1/tau_f, F~_p / 8, R, the last pressure increment
    unsigned cell;                // byte offset of the node's cell in a plane; ~0: no node
    int edge;                     // its row of the target table, or -1
    int go;                       // offset in the global planes
};

template <int NPT>
__global__ void __launch_bounds__(kResMaxThreads, 1)
    k_pressure_resident(const __grid_constant__ PressureArgs a, const __grid_constant__ ResidentArgs s)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ float red[7][kResMaxThreads / 32];     // the warps' residual sums, pivots and nodes
    __shared__ double part[4];            // this block's residual sums, read by the whole cluster
    __shared__ double tot[4];
    __shared__ int sh_stop;
    const Geom &g = a.g;
    const unsigned rank = cluster_rank(), C = cluster_size();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int y0 = (int)rank * s.h;
    const int rows = y0 + s.h < g.ny ? s.h : g.ny - y0;
    const int wc = g.nx + 2;
    const unsigned plane = (unsigned)s.cells * 4u, buffer = 8u * plane;
    const unsigned base = smem_u32(smem_raw);
    uint4 *table = reinterpret_cast<uint4 *>(smem_raw + 2 * (size_t)buffer);
    auto load = [&](unsigned addr) {
        float v;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
        return v;
    };
    auto store = [&](unsigned addr, float v) {
        asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
    };
    // distance in bytes from a node's cell to the source of direction i + 1, in its plane
    int src[8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        src[i] = (int)(i * plane) - 4 * (cx(i + 1) + cy(i + 1) * wc);

    ResNode<NPT> nd[NPT];
    // factors of w_i of node q from the node pressures R (fresh: written by this launch)
    auto factors = [&](ResNode<NPT> &n, int x, int y, bool fresh) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int ex = cx(i + 1), ey = cy(i + 1);
            int xs, ys;
            const int side = link_end(g, x, y, -ex, -ey, xs, ys);
            float d = 0.0f;
            if (side < 0) {
                const float *p = a.R + ys * g.pitch + xs;
                d = (fresh ? __ldcg(p) : *p) - n.r0;
            } else if (g.bc[side] != BC_NOFLUX) {
                const int k = side < 2 ? 2 * y + 1 - ey : 2 * x + 1 - ex;
                d = 2.0f * (a.Pb[side][k] - n.r0);
            }
            n.D[i] = d;
        }
    };
    // a node's new values: its own cell, and the ghost cells that are read in its place
    auto put = [&](const ResNode<NPT> &n, unsigned buf, const float (&v)[8]) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
            store(buf + i * plane + n.cell, v[i]);
        if (n.edge >= 0) {
            const uint4 t0 = table[2 * n.edge], t1 = table[2 * n.edge + 1];
            const unsigned t[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (t[i])
                    cluster_store((t[i] & ~3u) + (buf - base), flip(v[i], (t[i] & 2u) != 0));
        }
    };

    // ---- the nodes of this thread, and the targets of those on the border ------------------
#pragma unroll
    for (int q = 0; q < NPT; ++q) {
        ResNode<NPT> &n = nd[q];
        const int l = tid + q * (int)blockDim.x;
        n.cell = ~0u;
        n.edge = -1;
        n.dp = n.it = n.Fq = n.r0 = 0.0f;
        n.go = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i)
            n.D[i] = 0.0f;
        if (l >= rows * g.nx)
            continue;
        const int ly = l / g.nx, x = l - ly * g.nx, y = y0 + ly;
        n.cell = 4u * (unsigned)((ly + 1) * wc + x + 1);
        n.go = y * g.pitch + x;
        n.r0 = a.R[n.go];
        n.it = a.inv_tau[n.go];
        float F = a.Fp ? a.Fp[n.go] : 0.0f;
        for (int w = 0; w < a.w.n; ++w)
            if (n.go == a.w.idx[w])
                F += a.w.fp[w];
        n.Fq = 0.125f * F;   // w_bar_i = 1/8 (Eq. 3-5a)
        factors(n, x, y, false);
        // border nodes: the first and last row of the block, then the two end columns
        if (ly == 0)
            n.edge = x;
        else if (ly == rows - 1)
            n.edge = g.nx + x;
        else if (x == 0)
            n.edge = 2 * g.nx + ly;
        else if (x == g.nx - 1)
            n.edge = 2 * g.nx + s.h + ly;
        if (n.edge >= 0) {
            unsigned t[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int ex = cx(i + 1), ey = cy(i + 1);
                int xe, ye;
                const int side = link_end(g, x, y, ex, ey, xe, ye);
                t[i] = 0u;
                if (side >= 0) {
                    // the reader is this node, pulling the opposite direction from beyond the wall
                    const int cell = (y + ey - y0 + 1) * wc + x + ex + 1;
                    t[i] = cluster_addr(base + (unsigned)(opp(i + 1) - 1) * plane + 4u * (unsigned)cell,
                                        rank) | 1u | (g.bc[side] != BC_NOFLUX ? 2u : 0u);
                } else {
                    // the reader (xe, ye) pulls direction i + 1 from its cell (xe - ex, ye - ey)
                    const unsigned owner = (unsigned)(ye / s.h);
                    const int row = ye - ey - (int)owner * s.h + 1, col = xe - ex + 1;
                    if (owner != rank || row != ly + 1 || col != x + 1)
                        t[i] = cluster_addr(base + (unsigned)i * plane + 4u * (unsigned)(row * wc + col),
                                            owner) | 1u;
                }
            }
            table[2 * n.edge] = make_uint4(t[0], t[1], t[2], t[3]);
            table[2 * n.edge + 1] = make_uint4(t[4], t[5], t[6], t[7]);
        }
    }
    cluster_sync();                                   // every block has started
#pragma unroll
    for (int q = 0; q < NPT; ++q)
        if (nd[q].cell != ~0u) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = a.fin[i][nd[q].go];
            put(nd[q], base, v);
        }
    const float shift0 = a.shift[0], shift1 = a.shift[1];
    const int m = s.ctl ? s.ctl->m : s.m, cap = s.ctl ? s.ctl->cap : s.cap;
    const int every = s.ctl ? s.ctl->every : s.every;
    const double tol = s.ctl ? s.ctl->tol : s.tol;
    cluster_sync();

    // ---- sweeps ------------------------------------------------------------------------
    unsigned cur = base;
    int k = 0, to_check = m, to_rebase = every > 0 ? every : 0x7fffffff;
    double num = nan(""), den = 0.0;
    const double inv_n = 1.0 / ((double)g.nx * (double)g.ny);
    bool checked = false;
    while (k < cap) {
        ++k;
        const bool check = --to_check == 0, before = to_check == 1;
        const unsigned nxt = cur == base ? base + buffer : base;
        // Sums of d, d^2, u, u^2 over this warp's nodes in FP32, relative to means over the warp, so that
        // their rounding is a few 2^-24 of the spread inside the warp, whatever the values of other
        // nodes.  One node per thread: the means of this sweep.  Several: those of the sweep before a
        // check, since the nodes' d and u, kept until the means are there, would take registers that
        // the sweeps need (160^2: 1.94 us per sweep so, 1.73 now, 1.78 with one node's values as
        // everyone's pivots).
        constexpr bool kOne = NPT == 1;
        float s1 = 0.0f, s2 = 0.0f, t1 = 0.0f, t2 = 0.0f;
        float md = !kOne && check ? red[4][warp] : 0.0f, mu = !kOne && check ? red[5][warp] : 0.0f;
#pragma unroll
        for (int q = 0; q < NPT; ++q) {
            ResNode<NPT> &n = nd[q];
            if (n.cell == ~0u)
                continue;
            float f[8], v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
                f[i] = load(cur + n.cell + src[i]);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                f[i] = fmaf(wgt(i + 1), n.D[i], f[i]);
            const float dP = pressure_of(f);
#pragma unroll
            for (int i = 0; i < 8; ++i)
                v[i] = collide1(f[i], wgt(i + 1), dP, n.it, n.Fq);
            put(n, nxt, v);
            if (check || (!kOne && before)) {
                const float e = ((dP - n.dp) - shift1) - md, u = ((n.r0 - shift0) + dP) - mu;
                s1 += e;
                t1 += u;
                if (!kOne) {
                    s2 = fmaf(e, e, s2);
                    t2 = fmaf(u, u, t2);
                }
            }
            n.dp = dP;
        }
        cur = nxt;
        const bool h16 = lane & 16, h8 = lane & 8;
        if (kOne ? check : before) {
            float n = 0.0f;
#pragma unroll
            for (int q = 0; q < NPT; ++q)
                n += (float)__popc(__ballot_sync(0xffffffffu, nd[q].cell != ~0u));
            float v = (h16 ? t1 : s1) + __shfl_xor_sync(0xffffffffu, h16 ? s1 : t1, 16);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1)
                v += __shfl_xor_sync(0xffffffffu, v, o);
            v = n > 0.0f ? v * (1.0f / n) : 0.0f;
            if ((lane & 15) == 0) {
                red[4 + (lane >> 4)][warp] = v;
                red[6][warp] = n;
            }
            if (kOne) {
                md = __shfl_sync(0xffffffffu, v, 0);
                mu = __shfl_sync(0xffffffffu, v, 16);
                const bool mine = nd[0].cell != ~0u;
                s1 = mine ? s1 - md : 0.0f;
                t1 = mine ? t1 - mu : 0.0f;
                s2 = s1 * s1;
                t2 = t1 * t1;
            }
        }
        if (check) {
            // four sums over 32 lanes by six shuffles: lane 8 c ends with sum c
            s1 = (h16 ? t1 : s1) + __shfl_xor_sync(0xffffffffu, h16 ? s1 : t1, 16);
            s2 = (h16 ? t2 : s2) + __shfl_xor_sync(0xffffffffu, h16 ? s2 : t2, 16);
            s1 = (h8 ? s2 : s1) + __shfl_xor_sync(0xffffffffu, h8 ? s1 : s2, 8);
#pragma unroll
            for (int o = 4; o > 0; o >>= 1)
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            if ((lane & 7) == 0)
                red[lane >> 3][warp] = s1;
            __syncthreads();
            if (warp == 0) {
                // sum x = S1 + n p, sum x^2 = S2 + 2 p S1 + n p^2.  Up to eight warps: a lane per warp
                // and sum, half the FP64 instructions of the other form (64^2, per check: 1.7 us
                // against 2.0; with 32 warps, where it takes four rounds, 2.8 against 2.3 at 128^2).
                const int nw = (int)blockDim.x >> 5, c = lane >> 3;
                double t = 0.0;
                if (nw <= 8) {
                    const int w = lane & 7;
                    if (w < nw && red[6][w] > 0.0f) {
                        const double p = red[4 + (c >> 1)][w], S1 = red[c & 2][w];
                        const double raw = fma((double)red[6][w], p, S1);
                        t = (c & 1) ? fma(p, S1 + raw, (double)red[c][w]) : raw;
                    }
                } else {
                    // a lane per warp, then lanes 8 c .. 8 c + 7 hold sum c
                    double v[4] = {0.0, 0.0, 0.0, 0.0};
                    if (lane < nw && red[6][lane] > 0.0f) {
                        const double nodes = red[6][lane];
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            const double p = red[4 + i][lane], S1 = red[2 * i][lane];
                            v[2 * i] = fma(nodes, p, S1);
                            v[2 * i + 1] = fma(p, S1 + v[2 * i], (double)red[2 * i + 1][lane]);
                        }
                    }
                    v[0] = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
                    v[1] = (h16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
                    t = (h8 ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, h8 ? v[0] : v[1], 8);
                }
#pragma unroll
                for (int o = 4; o > 0; o >>= 1)
                    t += __shfl_xor_sync(0xffffffffu, t, o);
                if ((lane & 7) == 0)
                    part[c] = t;
            }
        }
        cluster_sync();
        if (check) {
            to_check = m;
            checked = true;
            // every block adds the blocks' sums in the same order
            for (int w = warp; w < 2; w += (int)blockDim.x >> 5) {
                const unsigned b = lane & 15, c = 2 * w + (lane >> 4);
                double t = b < C ? cluster_load(cluster_addr(smem_u32(&part[c]), b)) : 0.0;
                for (int o = 8; o > 0; o >>= 1)
                    t += __shfl_xor_sync(0xffffffffu, t, o);
                if (b == 0)
                    tot[c] = t;
            }
            __syncthreads();
            if (tid == 0) {
                // the residual r = sqrt(num / den)
                const double sd = tot[0], sp = tot[2];
                int stop = 0;
                num = tot[1] - sd * sd * inv_n;
                den = tot[3] - sp * sp * inv_n;
                if (!isfinite(num) || !isfinite(den)) {
                    num = nan("");
                    stop = 1;
                } else {
                    num = num > 0.0 ? num : 0.0;
                    den = den > 0.0 ? den : 0.0;
                    // r <= tol without the division and the root
                    stop = tol >= 0.0 && num <= tol * tol * den;
                }
                sh_stop = stop;
            }
            __syncthreads();
            if (sh_stop)
                break;
        }
        if (--to_rebase == 0) {
            to_rebase = every;
            if (k < cap) {
                // R moves to the current P: n_i -= w_i dP, R += dP (rebase_mid_node)
#pragma unroll
                for (int q = 0; q < NPT; ++q) {
                    ResNode<NPT> &n = nd[q];
                    if (n.cell == ~0u)
                        continue;
                    float v[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        v[i] = load(cur + i * plane + n.cell);
                    const float dP = 1.8f * ((((v[0] + v[1]) + (v[2] + v[3])) +
                                              ((v[4] + v[5]) + (v[6] + v[7]))) - 8.0f * n.Fq);
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        v[i] = fmaf(-wgt(i + 1), dP, v[i]);
                    put(n, cur, v);
                    n.r0 = n.r0 + dP;
                    n.dp -= dP;
                    s.Rw[n.go] = n.r0;
                }
                __threadfence();
                cluster_sync();
#pragma unroll
                for (int q = 0; q < NPT; ++q)
                    if (nd[q].cell != ~0u) {
                        const int y = nd[q].go / g.pitch;
                        factors(nd[q], nd[q].go - y * g.pitch, y, true);
                    }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NPT; ++q)
        if (nd[q].cell != ~0u)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                a.fout[i][nd[q].go] = load(cur + i * plane + nd[q].cell);
    if (rank == 0 && tid == 0) {
        double r = nan("");
        if (checked) {
            const double mean0 = (double)shift0 + tot[2] * inv_n;
            const double mean1 = (double)shift1 + tot[0] * inv_n;
            r = isnan(num) ? num : (den > 0.0 ? sqrt(num / den) : (num > 0.0 ? INFINITY : 0.0));
            s.out->r = r;
            s.out->mean_P = mean0;
            for (int c = 0; c < 4; ++c)
                s.out->sums[c] = tot[c];
            if (!isnan(num)) {
                s.shift_out[0] = (float)mean0;
                s.shift_out[1] = (float)mean1;
            }
        }
        if (s.ctl) {
            s.ctl->k = k;
            s.ctl->r = r;
        }
        if (s.set_ok)
            cudaGraphSetConditional(s.ok, isnan(r) ? 0u : 1u);
    }
    cluster_sync();                                   // no block leaves while its memory is read
}

void *resident_func(int npt)
{
    return npt == 1 ? (void *)k_pressure_resident<1>
                    : (npt == 2 ? (void *)k_pressure_resident<2> : (void *)k_pressure_resident<3>);
}

// the shape for clusters of C blocks, or C = 0 when the lattice does not fit
ResidentShape resident_shape(int C, int nx, int ny)
{
    ResidentShape p{};
    const long long h = (ny + C - 1) / C;
    if ((long long)(C - 1) * h >= ny)                 // a block without rows
        return p;
    const long long nodes = h * nx, cells = (h + 2) * (nx + 2LL), edges = 2LL * nx + 2 * h;
    if (nodes > (long long)kResMaxNpt * kResMaxThreads)
        return p;
    const long long bytes = cells * 64 + edges * 32;
    if (bytes > 220 * 1024)
        return p;
    p.C = C;
    p.h = (int)h;
    p.cells = (int)cells;
    p.edges = (int)edges;
    p.npt = (int)((nodes + kResMaxThreads - 1) / kResMaxThreads);
    const long long per = (nodes + p.npt - 1) / p.npt;
    p.threads = (int)((per + 31) / 32 * 32);
    p.smem = (size_t)bytes;
    return p;
}

cudaLaunchConfig_t resident_config(const ResidentShape &p, cudaLaunchAttribute *attr, void *stream)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)p.C);
    c.blockDim = dim3((unsigned)p.threads);
    c.dynamicSmemBytes = p.smem;
    c.stream = reinterpret_cast<cudaStream_t>(stream);
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)p.C;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    c.attrs = attr;
    c.numAttrs = 1;
    return c;
}

}  // namespace
}  // namespace lbm2p_dev

namespace lbm2p_launch {

using namespace lbm2p_dev;

bool resident_fits(int C, int nx, int ny)
{
    const ResidentShape p = resident_shape(C, nx, ny);
    if (p.C == 0)
        return false;
    void *f = resident_func(p.npt);
    cudaLaunchAttribute attr{};
    cudaLaunchConfig_t c = resident_config(p, &attr, nullptr);
    int clusters = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024) != cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, f, &c) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

// what the kernel relies on: a sweep between two checks (`part` is rewritten by the next one), and a
// check at the cap
static bool resident_args_ok(const ResidentShape &p, const ResidentArgs &s)
{
    return p.C > 0 && s.m >= 2 && s.cap >= s.m && s.cap % s.m == 0;
}

cudaError_t pressure_resident(const PressureArgs &a, const ResidentArgs &s_, int C, void *stream)
{
    const ResidentShape p = resident_shape(C, a.g.nx, a.g.ny);
    if (!resident_args_ok(p, s_))
        return cudaErrorInvalidValue;
    ResidentArgs s = s_;
    s.h = p.h;
    s.cells = p.cells;
    cudaLaunchAttribute attr{};
    cudaLaunchConfig_t c = resident_config(p, &attr, stream);
    void *args[] = {(void *)&a, (void *)&s};
    return cudaLaunchKernelExC(&c, resident_func(p.npt), args);
}

cudaError_t node_resident(cudaGraphNode_t *n, cudaGraph_t g, const cudaGraphNode_t *dep,
                          const PressureArgs &a, const ResidentArgs &s_, int C)
{
    const ResidentShape p = resident_shape(C, a.g.nx, a.g.ny);
    if (!resident_args_ok(p, s_))
        return cudaErrorInvalidValue;
    ResidentArgs s = s_;
    s.h = p.h;
    s.cells = p.cells;
    cudaKernelNodeParams prm{};
    prm.func = resident_func(p.npt);
    prm.gridDim = dim3((unsigned)p.C);
    prm.blockDim = dim3((unsigned)p.threads);
    prm.sharedMemBytes = (unsigned)p.smem;
    void *args[] = {(void *)&a, (void *)&s};
    prm.kernelParams = args;
    cudaError_t e = cudaGraphAddKernelNode(n, g, dep, dep ? 1 : 0, &prm);
    if (e != cudaSuccess)
        return e;
    cudaKernelNodeAttrValue v{};
    v.clusterDim.x = (unsigned)p.C;
    v.clusterDim.y = v.clusterDim.z = 1;
    return cudaGraphKernelNodeSetAttribute(*n, cudaKernelNodeAttributeClusterDimension, &v);
}

}  // namespace lbm2p_launch
