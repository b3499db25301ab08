// A small convolutional operator on the fifth-generation tensor cores (tcgen05): the 3x3
// convolutions of a five-layer network that predicts the next step's pressure for the warm
// start of the lattice Boltzmann pressure solve, with the kernels its training needs.
//
// Convolution as an implicit GEMM (forward and input gradient): a CTA computes tiles of
// M = 128 consecutive pixels by N = C_out channels; the reduction runs over K = 9 taps x C_in
// channels in steps of 16 (tcgen05.mma, BF16 inputs, FP32 accumulators in tensor memory, K-major
// core matrices in shared memory).  The weights stay in shared memory for the whole kernel.  The
// epilogue (tcgen05.ld, bias, activation, the ReLU mask of the input-gradient pass) stores BF16
// channels-last rows.
//
// Weight gradient: M = (input row, input channel), N = C_out, K = pixels, the channels-last operands
// read MN-major as they are; each CTA reduces a share of the pixels at one dx in tensor memory and adds
// its partial sums into the FP32 gradient with atomics.
//
// Every wait on an mbarrier is bounded; a CTA that gives up records the failure in *err,
// waits (bounded) for its MMAs in flight, frees its tensor memory and returns.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm2p.h"
#include "lbm2p_async.cuh"
#include "lbm2p_operator.h"

namespace lbm2p_internal {
lbm2p_status set_global_error(lbm2p_status st, const char *fmt, ...);
}

namespace lbm2p_op {
using lbm2p_dev::bar_arrive;
using lbm2p_dev::bar_init;
using lbm2p_dev::bar_try_wait;
using lbm2p_dev::kWaitLimit;
using lbm2p_dev::smem_u32;

typedef __nv_bfloat16 bf16;

// ---- tcgen05 primitives (inline PTX) --------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(slot)),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before()
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after()
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// shared-memory writes of this thread become visible to the tensor core (async proxy)
__device__ __forceinline__ void fence_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// D (tensor memory) = A B^T (+ D when accumulate), A: M x 16, B: N x 16, both K-major
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// the mbarrier receives one arrival when every tcgen05.mma issued so far by this thread is done
__device__ __forceinline__ void umma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

// 32 tensor-memory lanes x 16 consecutive 32-bit columns: thread l of the warp receives lane
// (base lane + l); the wait for the load is part of the same statement
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i)
        v[i] = __uint_as_float(r[i]);
}

// Shared-memory matrix descriptor, no swizzle, K-major core matrices of 8 rows x 16 bytes:
// start address, LBO = bytes between the two core matrices along K, SBO = bytes between
// 8-row groups along M (or N); bits 46..48 hold the descriptor version 0b001.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator (bit 4), BF16 A and B (bits 7, 10),
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
           ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool wait_bounded(uint64_t *bar, unsigned parity)
{
    for (unsigned it = 0; it < kWaitLimit; ++it)
        if (bar_try_wait(bar, parity))
            return true;
    return false;
}

// 0xffff in each half whose BF16 value is positive
__device__ __forceinline__ uint32_t positive2(uint32_t v)
{
    return __hgt2_mask(*reinterpret_cast<const __nv_bfloat162 *>(&v), __float2bfloat162_rn(0.0f));
}

struct ConvArgs {
    const bf16 *x;        // [npix][cin]
    const bf16 *w;        // [9][cout][cin]
    const float *bias;    // [cout] or null
    const bf16 *mask;     // [npix][cout] or null
    bf16 *y;              // [npix][cout] or null
    float *y0;            // [npix] or null
    int nimg, H, W;
    int act;
    int *err;
};

// ---- convolution on staged rows ----------------------------------------------------------
// A tile is 128 consecutive pixels of one image row (x0 .. x0 + 127, the last tile of a row
// ragged).  A CTA works down a strip of 128 columns, so its ring holds input rows, each copied once
// and read by the three tiles that it borders: pixels x0 - 1 .. x0 + 128 of a row as channel-chunk
// planes, chunk c (channels 8 c .. 8 c + 7) an array of 130 pixels x 16 bytes.  In that layout the A
// operand of tap (dy, dx) and K-half j is the K-major core-matrix matrix that starts at row
// dy + 1, chunk 2 j, pixel dx + 1: a shift by one pixel is a shift of the descriptor's start address
// by 16 bytes.  Rows above and below an image are zero: their taps are left out.
//
// The three stages of a tile run in different warps, handed on by mbarriers: eight warps copy (whole
// pixels, a warp 512 contiguous bytes, the next three rows' loads in registers while one is
// stored: cp.async with a chunk plane as its target makes a request of every 16 bytes and kept the
// load/store unit 60 to 80 % busy), one thread issues the MMAs (descriptors by additions), four warps
// read the accumulator, of which there are two, apply bias, activation and mask and store whole pixels
// through a padded row per warp.
// 1024^2 pixels, 32 -> 32 channels: 80 us with all three in turn in one set of warps, 56 us in three
// with every tile's three rows copied anew (the load/store unit's data path 64 % busy), 46 us so.
constexpr int kRowPix = 130;                        // staged pixels per row
constexpr uint32_t kChunkBytes = kRowPix * 16;      // one channel chunk of a staged row
constexpr int kCvCopiers = 8, kCvEpilogue = 4;      // warps 0-7, 8-11; warp 12 issues the MMAs
constexpr int kCvThreads = 32 * (kCvCopiers + kCvEpilogue + 1);
constexpr int kCvRows = 8;                          // input rows in the ring
constexpr int kCvAhead = 4;                         // rows that a copying lane has in registers
constexpr uint32_t kCvTmemCols = 64;                // two accumulators of 32 columns

// 16 bytes of padding per pixel row of the output tile of a warp
template <int COUT>
__host__ __device__ constexpr uint32_t conv_out_row() { return COUT * 2 + 16; }

template <int CIN, int COUT>
__host__ __device__ constexpr size_t conv_rows_smem_bytes()
{
    return (size_t)(9 * CIN / 16) * COUT * 32 + kCvRows * (size_t)(CIN / 8) * kChunkBytes +
           (size_t)kCvEpilogue * 32 * conv_out_row<COUT>() + (2 * kCvRows + 4) * 8 + 16 + 128;
}

// A CTA's tiles: `left` of them from row r of strip `strip` on, down the rows of all images and on
// to the next strip.  A segment is the part in one strip: tiles r .. r + n - 1, which read the input
// rows lo .. hi (the first and last rows of an image beside them included, read or not).
struct ConvWalk {
    long long rows;                                 // of all images
    long long r, lo, hi;
    int strip;
    unsigned n, left;

    __device__ __forceinline__ void open()
    {
        const long long room = rows - r;
        n = (long long)left < room ? left : (unsigned)room;
        left -= n;
        lo = r > 0 ? r - 1 : 0;
        hi = r + n < rows ? r + n : rows - 1;
    }
    __device__ __forceinline__ ConvWalk(long long first, unsigned count, long long rows_)
        : rows(rows_), r(first % rows_), strip((int)(first / rows_)), left(count)
    {
        open();
    }
    __device__ __forceinline__ bool next()
    {
        if (left == 0)
            return false;
        r = 0;
        ++strip;
        open();
        return true;
    }
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(kCvThreads, 2) k_conv3x3_rows(const ConvArgs a)
{
    constexpr int CH = CIN / 8, GH = COUT / 8;
    constexpr int KH = CIN / 16;                      // K-halves of 16 channels per tap
    constexpr int KS = 9 * KH;
    constexpr uint32_t kBBytes = COUT * 16 * 2;
    constexpr uint32_t kRowBytes = CH * kChunkBytes;
    constexpr uint32_t IDESC = idesc_bf16(128, COUT);
    constexpr uint32_t ORow = conv_out_row<COUT>();
    constexpr unsigned R = kCvRows;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    unsigned char *wsm = smem;
    unsigned char *stg = smem + KS * kBBytes;
    unsigned char *osm = stg + R * kRowBytes;
    // full[s] / empty[s]: ring row s copied / read; done[d] / taken[d]: accumulator d ready / read
    uint64_t *full = reinterpret_cast<uint64_t *>(osm + kCvEpilogue * 32 * ORow);
    uint64_t *empty = full + R, *done = empty + R, *taken = done + 2;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(taken + 2);
    __shared__ int failed;
    __shared__ unsigned issued;                       // tiles given to the tensor core
    __shared__ __align__(16) float bsm[COUT];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kMmaWarp = kCvCopiers + kCvEpilogue;

    for (int i = tid; i < KS * COUT * 2; i += kCvThreads) {
        const int s = i / (COUT * 2), rem = i - s * (COUT * 2);
        const int kc = rem / COUT, n = rem - kc * COUT;
        const int t = s / KH, j = s - t * KH;
        const uint4 v = *reinterpret_cast<const uint4 *>(a.w + ((size_t)(t * COUT + n) * CIN + 16 * j + 8 * kc));
        *reinterpret_cast<uint4 *>(wsm + s * kBBytes + kc * (COUT * 16) + n * 16) = v;
    }
    if (a.bias && tid < COUT)
        bsm[tid] = a.bias[tid];
    if (warp == kMmaWarp) {
        tmem_alloc(tslot, kCvTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        failed = 0;
        issued = 0;
        for (unsigned i = 0; i < R; ++i) {
            bar_init(full + i, kCvCopiers);
            bar_init(empty + i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            bar_init(done + i, 1);
            bar_init(taken + i, kCvEpilogue);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const long long rows = (long long)a.nimg * a.H, tiles = rows * ((a.W + 127) / 128);
    const long long first = tiles * blockIdx.x / gridDim.x;
    const unsigned count = (unsigned)(tiles * (blockIdx.x + 1) / gridDim.x - first);
    bool ok = true;
    if (warp == kMmaWarp) {
        if (lane == 0) {
            // descriptors: start addresses count 16 bytes
            const uint64_t ad0 = sdesc(smem_u32(stg), kChunkBytes, 128);
            const uint64_t bd0 = sdesc(smem_u32(wsm), COUT * 16, 128);
            unsigned waited = 0, released = 0, n = 0;  // ring rows, tiles
            auto wait_to = [&](unsigned k) {          // ring rows up to k are there
                for (; ok && waited <= k; ++waited)
                    ok = wait_bounded(full + waited % R, (waited / R) & 1u);
            };
            ConvWalk wk(first, count, rows);
            unsigned k0 = 0;                          // ring row of the segment's first
            do {
                int y = (int)(wk.r % a.H);
                for (unsigned i = 0; i < wk.n && ok; ++i, ++n) {
                    const unsigned kc = k0 + (unsigned)(wk.r - wk.lo) + i;   // ring row of the tile's own
                    const bool up = y > 0, down = y < a.H - 1;
                    wait_to(down ? kc + 1 : kc);
                    ok = ok && (n < 2 || wait_bounded(taken + (n & 1u), ((n >> 1) + 1u) & 1u));
                    if (!ok)
                        break;
                    tc_fence_after();
                    const uint32_t d = tmem + 32u * (n & 1u);
#pragma unroll
                    for (int dy = 0; dy < 3; ++dy) {
                        if (dy == 0 ? !up : (dy == 2 && !down))
                            continue;
                        const uint64_t ad = ad0 + ((kc + dy - 1) % R) * (kRowBytes >> 4);
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                            for (int j = 0; j < KH; ++j)
                                umma_bf16(d, ad + ((2 * j * kChunkBytes + dx * 16) >> 4),
                                          bd0 + ((((dy * 3 + dx) * KH + j) * kBBytes) >> 4), IDESC,
                                          dx + j > 0 || dy == 2 || (dy == 1 && up) ? 1u : 0u);
                    }
                    // rows that no later tile of the segment reads go back
                    const bool end = i + 1 == wk.n;
                    const unsigned done_to = end ? k0 + (unsigned)(wk.hi - wk.lo) + 1u : kc;
                    if (end)
                        wait_to(done_to - 1u);
                    for (; released < done_to; ++released)
                        umma_commit(empty + released % R);
                    umma_commit(done + (n & 1u));
                    issued = n + 1;
                    y = down ? y + 1 : 0;
                }
                k0 += (unsigned)(wk.hi - wk.lo) + 1u;
            } while (ok && wk.next());
        }
        __syncwarp();
    } else if (warp < kCvCopiers) {
        // ---- copies: chunk c of pixels px, px + P, ... of a row; its last two pixels by the first
        // lanes ----
        constexpr int P = 32 * kCvCopiers / CH;       // pixels per pass
        constexpr int NP = 128 / P, NV = NP + 1;
        const int c = tid % CH, px = tid / CH;
        const bool tail = tid < 2 * CH;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        ConvWalk wk(first, count, rows);
        long long row = wk.lo;
        bool more = true;
        auto fetch = [&](uint4 (&v)[NV]) {            // the next row
            if (!more)
                return;
            const int x0 = wk.strip * 128;
            const bf16 *src = a.x + (row * a.W + x0 - 1) * CIN + 8 * c;
            auto get = [&](int p) {
                const int xx = x0 - 1 + p;
                return xx >= 0 && xx < a.W ? __ldg(reinterpret_cast<const uint4 *>(src + (long long)p * CIN)) : zero;
            };
#pragma unroll
            for (int q = 0; q < NP; ++q)
                v[q] = get(px + q * P);
            v[NP] = tail ? get(128 + px) : zero;
            if (row < wk.hi) {
                ++row;
            } else {
                more = wk.next();
                row = wk.lo;
            }
        };
        auto hand_over = [&](unsigned k, const uint4 (&v)[NV]) {
            if (k >= R && !wait_bounded(empty + k % R, (k / R + 1u) & 1u)) {
                ok = false;
                return;
            }
            unsigned char *dst = stg + (k % R) * kRowBytes + c * kChunkBytes;
#pragma unroll
            for (int q = 0; q < NP; ++q)
                *reinterpret_cast<uint4 *>(dst + (px + q * P) * 16) = v[q];
            if (tail)
                *reinterpret_cast<uint4 *>(dst + (128 + px) * 16) = v[NP];
            fence_async_smem();
            __syncwarp();
            if (lane == 0)
                bar_arrive(full + k % R);
        };
        unsigned total = 0;                           // rows of all segments
        {
            ConvWalk t(first, count, rows);
            do
                total += (unsigned)(t.hi - t.lo) + 1u;
            while (t.next());
        }
        uint4 v[kCvAhead][NV];
#pragma unroll
        for (int d = 0; d < kCvAhead; ++d)
            fetch(v[d]);
        for (unsigned k = 0; k < total && ok; k += kCvAhead)
#pragma unroll
            for (int d = 0; d < kCvAhead; ++d)
                if (k + d < total && ok) {
                    hand_over(k + d, v[d]);
                    fetch(v[d]);
                }
    } else {
        // ---- epilogue: a pixel per lane, 32 lanes of tensor memory per warp ----
        const int w = warp - kCvCopiers;              // = warp % 4, the warp's tensor-memory lanes
        unsigned char *out = osm + w * 32 * ORow;
        // stores: whole pixels, GH lanes each; lane's chunk sc of pixels sp, sp + 32 / GH, ...
        const int sc = lane % GH, sp = lane / GH;
        ConvWalk wk(first, count, rows);
        long long row = wk.r - 1;
        unsigned left = wk.n;                         // tiles of the segment
        for (unsigned n = 0; n < count; ++n) {
            ++row;
            if (left == 0) {
                wk.next();
                row = wk.r;
                left = wk.n;
            }
            --left;
            const int xw = wk.strip * 128 + 32 * w;   // the warp's first pixel
            const long long q0 = row * a.W + xw;
            // the mask is on its way while the tensor core works
            uint4 mk[GH];
            if (a.mask)
#pragma unroll
                for (int i = 0; i < GH; ++i) {
                    const int px = i * (32 / GH) + sp;
                    mk[i] = xw + px < a.W ? __ldg(reinterpret_cast<const uint4 *>(
                                                a.mask + (q0 + px) * COUT + 8 * sc))
                                          : make_uint4(0u, 0u, 0u, 0u);
                }
            const bool m0 = a.mask && a.y0 && xw + lane < a.W
                                ? __bfloat162float(a.mask[(q0 + lane) * COUT]) > 0.0f : true;
            ok = wait_bounded(done + (n & 1u), (n >> 1) & 1u);
            if (!ok)
                break;
            tc_fence_after();
            float v[COUT];
#pragma unroll
            for (int h = 0; h < COUT / 16; ++h)
                tmem_ld16(tmem + ((uint32_t)(32 * w) << 16) + 32u * (n & 1u) + 16u * h,
                          *reinterpret_cast<float (*)[16]>(v + 16 * h));
            tc_fence_before();
            __syncwarp();
            if (lane == 0)
                bar_arrive(taken + (n & 1u));
            if (a.bias)
#pragma unroll
                for (int i = 0; i < COUT; i += 4) {
                    const float4 t = *reinterpret_cast<const float4 *>(bsm + i);
                    v[i] += t.x;
                    v[i + 1] += t.y;
                    v[i + 2] += t.z;
                    v[i + 3] += t.w;
                }
            if (a.act == 1)
#pragma unroll
                for (int i = 0; i < COUT; ++i)
                    v[i] = fmaxf(v[i], 0.0f);
            if (a.y0 && xw + lane < a.W)
                a.y0[q0 + lane] = m0 ? v[0] : 0.0f;
            if (!a.y)
                continue;
#pragma unroll
            for (int c = 0; c < GH; ++c) {
                __nv_bfloat162 o[4];
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    o[e] = __floats2bfloat162_rn(v[8 * c + 2 * e], v[8 * c + 2 * e + 1]);
                *reinterpret_cast<uint4 *>(out + lane * ORow + c * 16) = *reinterpret_cast<const uint4 *>(o);
            }
            __syncwarp();
#pragma unroll
            for (int i = 0; i < GH; ++i) {
                const int px = i * (32 / GH) + sp;
                uint4 o = *reinterpret_cast<const uint4 *>(out + px * ORow + sc * 16);
                if (a.mask) {
                    o.x &= positive2(mk[i].x);
                    o.y &= positive2(mk[i].y);
                    o.z &= positive2(mk[i].z);
                    o.w &= positive2(mk[i].w);
                }
                if (xw + px < a.W)
                    *reinterpret_cast<uint4 *>(a.y + (q0 + px) * COUT + 8 * sc) = o;
            }
            __syncwarp();
        }
    }
    if (!ok)
        failed = 1;
    __syncthreads();
    // every MMA issued has ended when the last commits have arrived
    for (unsigned q = issued > 2u ? issued - 2u : 0u; q < issued; ++q)
        if (!wait_bounded(done + (q & 1u), (q >> 1) & 1u))
            ok = false;
    if ((!ok || failed) && lane == 0)
        atomicExch(a.err, 1);
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) {
        tc_fence_after();
        tmem_dealloc(tmem, kCvTmemCols);
    }
}

// ---- weight gradient --------------------------------------------------------------------
// dw[t][co][ci] = sum over pixels p of x[p + d_t][ci] g[p][co]: M = (input row dy, channel), N = C_out,
// K = pixels, a CTA per dx and chain.  The operands have their channels contiguous, i.e. they are
// MN-major, which the tensor core reads as they are (transpose bits of the instruction descriptor):
// a chunk of eight channels by eight pixels is one 128-byte core matrix, so a stage holds, per input
// row and chunk, eight K-steps of 16 pixels x 16 bytes (core matrices 128 bytes apart along K).  The rows of M beyond 3 C_in read whatever follows and are not
// used.  Sixteen (eight) warps load whole pixels (two groups of eight K-steps ahead, in registers: cp.async
// with chunk planes as its target fetched every 16 bytes by a request of its own, 194 us), store them
// into a ring of stages and hand these over by mbarriers to the warp that issues the MMAs; the
// accumulator stays in tensor memory over all of a CTA's K-steps and is added to the gradient
// with FP32 atomics at the end.  In the CTAs of dx = 0 every copying lane also
// adds up what it copied of g: the bias gradient.
//
// The pixels are reduced in gridDim.y chains, chain s taking K-steps s, s + chains, ...: a third
// (half) of the SMs, i.e. one chain per SM and 128 rows of the 9 C_in.  The tensor core truncates when
// it accumulates, so a result depends on the length of its chain: 50 chains are 2e-5 from the exact
// sums where 456 shorter ones were 2e-6 (and took a fifth less of a training step), but results are
// kept as they have been.
// 16 images of 256^2, 32 -> 32 channels: 1551 us before (one K-step at a time, transposed by 2-byte
// stores into K-major matrices) and 22 us for the bias on its own.
// warps that copy (16 bytes of three rows of x per lane and group), beside the one that issues the
// MMAs: sixteen at 32 input channels, eight at 16, where two CTAs share an SM
__host__ __device__ constexpr int wgrad_copiers(int cin) { return cin == 32 ? 16 : 8; }
__host__ __device__ constexpr int wgrad_threads(int cin) { return 32 * (wgrad_copiers(cin) + 1); }
constexpr int kWgSteps = 8;                          // K-steps of a stage
constexpr uint32_t kWgTmemCols = 32;
template <int CIN>
__host__ __device__ constexpr int wgrad_stages() { return 3; }
// bytes from chunk plane to chunk plane in a stage: the lanes of a warp copy whole pixels, chunk by
// chunk, and the distance keeps their 16-byte writes in different banks
__host__ __device__ constexpr uint32_t wgrad_plane(int channels)
{
    return kWgSteps * 256 + (channels == 32 ? 32 : 64);
}

struct WgradArgs {
    const bf16 *x;        // [npix][cin]
    const bf16 *g;        // [npix][cout]
    float *dw;            // [9][cout][cin]
    float *db;            // [cout] or null
    int nimg, H, W;
    int *err;
};

template <int CIN, int COUT>
__host__ __device__ constexpr uint32_t wgrad_stage_bytes()
{
    return (uint32_t)(3 * (CIN / 8)) * wgrad_plane(CIN) + (uint32_t)(COUT / 8) * wgrad_plane(COUT);
}

// the 16 planes that an MMA's 128 rows span reach past the last stage
template <int CIN, int COUT>
__host__ __device__ constexpr size_t wgrad_smem_bytes()
{
    const size_t st = wgrad_stage_bytes<CIN, COUT>(), reach = 16 * (size_t)wgrad_plane(CIN);
    return (wgrad_stages<CIN>() - 1) * st + (st > reach ? st : reach) + wgrad_stages<CIN>() * 16 + 16 + 128;
}

template <int CIN, int COUT>
__global__ void __launch_bounds__(wgrad_threads(CIN), CIN == 32 ? 1 : 2) k_conv3x3_wgrad(const WgradArgs a)
{
    constexpr int CH = CIN / 8, GH = COUT / 8;
    constexpr int kCopiers = wgrad_copiers(CIN);
    // 16-byte pieces of g per lane and group
    constexpr int GI = kWgSteps * GH * 16 > 32 * kCopiers ? kWgSteps * GH / (2 * kCopiers) : 1;
    constexpr uint32_t IDESC = idesc_bf16(128, COUT) | (1u << 15) | (1u << 16);
    constexpr uint32_t kXP = wgrad_plane(CIN), kGP = wgrad_plane(COUT);
    constexpr uint32_t kG = 3 * CH * kXP;                     // the output gradients in a stage
    constexpr uint32_t kStage = wgrad_stage_bytes<CIN, COUT>();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    constexpr int R = wgrad_stages<CIN>();
    // full[s]: every copying warp's share of stage s is in place; empty[s]: its MMAs are done
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + wgrad_smem_bytes<CIN, COUT>() - 128 - 16 - R * 16);
    uint64_t *empty = full + R;
    uint32_t *tslot = reinterpret_cast<uint32_t *>(empty + R);
    __shared__ int failed;
    __shared__ unsigned issued;                               // groups given to the tensor core
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int dx = (int)blockIdx.x - 1;
    const long long chains = gridDim.y;

    if (warp == kCopiers) {
        tmem_alloc(tslot, kWgTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        failed = 0;
        issued = 0;
        for (int i = 0; i < R; ++i) {
            bar_init(full + i, kCopiers);
            bar_init(empty + i, 1);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const long long npix = (long long)a.nimg * a.H * a.W;
    const long long ksteps = (npix + 15) / 16;
    // this chain's K-steps, in groups of kWgSteps
    const long long mine = ksteps > (long long)blockIdx.y ? (ksteps - blockIdx.y + chains - 1) / chains : 0;
    const unsigned groups = (unsigned)((mine + kWgSteps - 1) / kWgSteps);
    bool ok = true;
    if (warp == kCopiers) {
        // ---- MMAs: one thread ----
        if (lane == 0) {
            // descriptors: start addresses count 16 bytes
            const uint64_t xd0 = sdesc(smem_u32(smem), 128, kXP), gd0 = sdesc(smem_u32(smem) + kG, 128, kGP);
            for (unsigned n = 0; n < groups && ok; ++n) {
                ok = wait_bounded(full + n % R, (n / R) & 1u);
                if (!ok)
                    break;
                tc_fence_after();
                const uint64_t at = (n % R) * (kStage >> 4);
                const long long left = mine - (long long)n * kWgSteps;
#pragma unroll
                for (int ks = 0; ks < kWgSteps; ++ks)
                    if (ks < left)
                        umma_bf16(tmem, xd0 + at + ks * 16, gd0 + at + ks * 16, IDESC,
                                  (n > 0 || ks > 0) ? 1u : 0u);
                umma_commit(empty + n % R);
                issued = n + 1;
            }
        }
        __syncwarp();
    } else {
        // ---- copies ----
        // pixel k of K-step ks, one chunk of x (in three rows) and one of g of every group.  From
        // group to group the pixel moves on by 16 kWgSteps chains; image row and column move with
        // it (no division inside the loop).
        const int k = (tid / CH) & 15, xc = tid % CH, xks = tid / (16 * CH);
        const int gk = (tid / GH) & 15, gc = tid % GH, gks = tid / (16 * GH);
        const long long step = 16 * kWgSteps * chains;
        const int step_y = (int)((step / a.W) % a.H), step_x = (int)(step % a.W);
        long long xp = ((long long)blockIdx.y + xks * chains) * 16 + k;
        long long gp = ((long long)blockIdx.y + gks * chains) * 16 + gk;
        int y = (int)((xp / a.W) % a.H), x = (int)(xp % a.W);
        const long long wrow = (long long)a.W * CIN;
        const bool bias = dx == 0 && a.db && gks < kWgSteps;
        float bsum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        const unsigned xoff = xc * kXP + xks * 256 + k * 16, goff = kG + gc * kGP + gks * 256 + gk * 16;
        const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
        // this lane's loads of group grp (zeros outside the image), then on to the next group
        auto fetch = [&](unsigned grp, uint4 (&v)[3 + GI]) {
            const bool in = xks < kWgSteps && xp < npix && (long long)grp * kWgSteps + xks < mine &&
                            x + dx >= 0 && x + dx < a.W;
            const bf16 *src = a.x + (xp + dx) * CIN + 8 * xc;
            v[0] = in && y > 0 ? __ldg(reinterpret_cast<const uint4 *>(src - wrow)) : zero;
            v[1] = in ? __ldg(reinterpret_cast<const uint4 *>(src)) : zero;
            v[2] = in && y < a.H - 1 ? __ldg(reinterpret_cast<const uint4 *>(src + wrow)) : zero;
#pragma unroll
            for (int q = 0; q < GI; ++q) {
                const int ks = gks + q * (kWgSteps / GI);
                const long long p = gp + q * (kWgSteps / GI) * 16 * chains;
                v[3 + q] = ks < kWgSteps && p < npix && (long long)grp * kWgSteps + ks < mine
                               ? __ldg(reinterpret_cast<const uint4 *>(a.g + p * COUT + 8 * gc)) : zero;
            }
            xp += step;
            gp += step;
            x += step_x;
            y += step_y;
            if (x >= a.W) {
                x -= a.W;
                ++y;
            }
            if (y >= a.H)
                y -= a.H;
        };
        auto hand_over = [&](unsigned grp, const uint4 (&v)[3 + GI]) {
            if (grp >= (unsigned)R && !wait_bounded(empty + grp % R, (grp / R + 1u) & 1u)) {
                ok = false;
                return;
            }
            unsigned char *buf = smem + (grp % R) * kStage;
            if (xks < kWgSteps)
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    *reinterpret_cast<uint4 *>(buf + r * CH * kXP + xoff) = v[r];
            if (gks < kWgSteps)
#pragma unroll
                for (int q = 0; q < GI; ++q)
                    *reinterpret_cast<uint4 *>(buf + goff + q * (kWgSteps / GI) * 256) = v[3 + q];
            fence_async_smem();
            __syncwarp();
            if (lane == 0)
                bar_arrive(full + grp % R);
            if (bias)
#pragma unroll
                for (int q = 0; q < GI; ++q) {
                    const uint32_t w[4] = {v[3 + q].x, v[3 + q].y, v[3 + q].z, v[3 + q].w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        bsum[2 * e] += __uint_as_float(w[e] << 16);
                        bsum[2 * e + 1] += __uint_as_float(w[e] & 0xFFFF0000u);
                    }
                }
        };
        // D - 1 groups of loads in flight while another is stored
        constexpr int D = 3;
        uint4 v[D][3 + GI];
#pragma unroll
        for (int u = 0; u < D - 1; ++u)
            if ((unsigned)u < groups)
                fetch(u, v[u]);
        for (unsigned n = 0; n < groups && ok; n += D)
#pragma unroll
            for (int u = 0; u < D; ++u) {
                if (n + u + D - 1 < groups)
                    fetch(n + u + D - 1, v[(u + D - 1) % D]);
                if (n + u < groups && ok)
                    hand_over(n + u, v[u]);
            }
        if (bias && ok) {
            // lanes of the same chunk are GH apart
#pragma unroll
            for (int e = 0; e < 8; ++e) {
#pragma unroll
                for (int o = 16; o >= GH; o >>= 1)
                    bsum[e] += __shfl_xor_sync(0xffffffffu, bsum[e], o);
                if (lane < GH)
                    atomicAdd(a.db + 8 * gc + e, bsum[e]);
            }
        }
    }
    if (!ok)
        failed = 1;
    __syncthreads();
    // every MMA issued has ended when the last commits have arrived
    for (unsigned q = issued > (unsigned)R ? issued - R : 0; q < issued; ++q)
        if (!wait_bounded(empty + q % R, (q / R) & 1u))
            ok = false;
    ok = ok && !failed;
    if (ok && groups > 0) {
        tc_fence_after();
        const int cb = 16 * (warp >> 2), row = 32 * (warp & 3) + lane;
        if (cb < COUT) {
            float v[16];
            tmem_ld16(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)cb, v);
            if (row < 3 * CIN) {
                const int r = row / CIN, ci = row - r * CIN;
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    atomicAdd(a.dw + ((size_t)(3 * r + dx + 1) * COUT + cb + i) * CIN + ci, v[i]);
            }
        }
    }
    if (!ok && lane == 0)
        atomicExch(a.err, 1);
    tc_fence_before();
    __syncthreads();
    if (warp == kCopiers) {
        tc_fence_after();
        tmem_dealloc(tmem, kWgTmemCols);
    }
}

// ---- CUDA-core helpers -------------------------------------------------------------------
__global__ void k_flip(const bf16 *w, bf16 *wt, int cin, int cout)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;   // over wt[t][ci][co]
    if (i >= 9 * cin * cout)
        return;
    const int t = i / (cin * cout), r = i - t * cin * cout;
    const int ci = r / cout, co = r - ci * cout;
    wt[i] = w[((size_t)(8 - t) * cout + co) * cin + ci];
}

__global__ void k_adam(float *p, const float *g, float *m, float *v, bf16 *pb, long long n,
                       float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pi;
        if (pb)
            pb[i] = __float2bfloat16_rn(pi);
    }
}

__device__ __forceinline__ float sd_of(const double *st, long long n)
{
    const double m = st[0] / (double)n;
    const double v = st[1] / (double)n - m * m;
    return v > 1e-60 ? (float)sqrt(v) : 1.0f;
}

// a + b = s + e exactly (Knuth's two-sum); returns s
__device__ __forceinline__ float two_sum(float a, float b, float &e)
{
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// A running sum as x + y + z: what x rounds off goes into y exactly, what y rounds off into z, so the
// whole is good to about 2^-70 where an FP64 sum is good to 2^-53.
struct Sum3 {
    float x = 0.0f, y = 0.0f, z = 0.0f;

    __device__ __forceinline__ void mid(float m)              // m some 2^-24 of the sum
    {
        float e;
        y = two_sum(y, m, e);
        z += e;
    }
    __device__ __forceinline__ void add(float h, float m)     // h + m, m at most 2^-24 of h
    {
        float e;
        x = two_sum(x, h, e);
        mid(e);
        mid(m);
    }
    __device__ __forceinline__ void scale(float f)            // f^2, a power of two
    {
        x = x * f * f;
        y = y * f * f;
        z = z * f * f;
    }
    __device__ __forceinline__ void add_lane(int o)           // the same sum of the lane o away
    {
        const float h = __shfl_xor_sync(0xffffffffu, x, o), m = __shfl_xor_sync(0xffffffffu, y, o);
        z += __shfl_xor_sync(0xffffffffu, z, o);
        add(h, m);
    }
    __device__ __forceinline__ double value() const { return (double)x + ((double)y + (double)z); }
};

// a power of two that brings |v| near 1 (1 for zero, infinities and NaN)
__device__ __forceinline__ float unit_scale(float v)
{
    const int e = (int)((__float_as_uint(v) >> 23) & 255u);
    return e == 255 || v == 0.0f ? 1.0f : __uint_as_float((unsigned)(e < 253 ? 254 - e : 1) << 23);
}

// Sums of a - b and (a - b)^2.  The difference of two floats is a pair of floats exactly, its square
// one of four: each thread adds these in FP32 sums that lose less than FP64 ones (Sum3), the squares
// scaled by a power of two that follows its largest difference (so they cover the range that FP64
// would); a warp adds its lanes' sums at the scale of the largest, and one lane turns them into FP64,
// which the block and the grid add.  FP64 per element took 27 us for a 1024^2 plane, FP64 per thread
// 32 us (an FP64 instruction holds its SM for 16 cycles, and every warp ran forty), this 8 us.  VEC:
// 128-bit loads (both planes aligned).
struct DiffSums {
    static constexpr float kFar = 0x1p95f;                    // room for 2^32 of them in an FP32 sum
    Sum3 s1, s2;
    float sc = 0.0f;                                          // scale of s2's terms (0: none yet)
    float lim = 0.0f;                                         // largest difference at that scale
    bool far = false;                                         // left something to add_far

    template <int N>
    __device__ __forceinline__ static float largest(const float (&x)[N], const float (&y)[N])
    {
        float big = 0.0f;
#pragma unroll
        for (int i = 0; i < N; ++i)
            big = fmaxf(big, fabsf(__fsub_rn(x[i], y[i])));
        return big;
    }

    // N differences at a time: their sums are independent but for one addition each
    template <int N>
    __device__ __forceinline__ void add(const float (&x)[N], const float (&y)[N])
    {
        float h[N], l[N];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            h[i] = __fsub_rn(x[i], y[i]);
            const float yy = __fsub_rn(x[i], h[i]);
            l[i] = __fsub_rn(__fsub_rn(x[i], __fadd_rn(h[i], yy)), __fsub_rn(y[i], yy));
        }
        const float big = largest(x, y);
        if (big > lim) {
            if (big >= kFar) {
                far = true;
#pragma unroll
                for (int i = 0; i < N; ++i)
                    h[i] = l[i] = 0.0f;
            } else {
                const float ns = unit_scale(big);
                s2.scale(sc == 0.0f ? 0.0f : ns / sc);        // both powers of two
                sc = ns;
                lim = fminf(1073741824.0f / ns, 0x1.fffffep94f);
            }
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            s1.add(h[i], l[i]);
            // (u + v)^2 = u u + 2 u v + v v
            const float u = h[i] * sc, v = l[i] * sc, q = __fmul_rn(u, u), p = __fmul_rn(2.0f * u, v);
            s2.add(q, fmaf(u, u, -q));
            s2.mid(p);
            s2.z += fmaf(v, v, fmaf(2.0f * u, v, -p));
        }
    }

    // What add left out, in FP64: where a difference is beyond what FP32 sums hold, or infinite, its
    // parts are of no use, but two finite floats have a finite FP64 difference with a finite square.
    // (A NaN has made the FP32 sums NaN by itself.)
    template <int N>
    __device__ __forceinline__ static void add_far(const float (&x)[N], const float (&y)[N], double &f1,
                                                   double &f2)
    {
        if (largest(x, y) >= kFar)
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const double d = (double)x[i] - (double)y[i];
                f1 += d;
                f2 += d * d;
            }
    }

    // the sums of the warp in every lane
    __device__ __forceinline__ void warp_sum()
    {
        float low = sc > 0.0f ? sc : __int_as_float(0x7f800000);
        for (int o = 16; o > 0; o >>= 1)
            low = fminf(low, __shfl_xor_sync(0xffffffffu, low, o));
        s2.scale(sc > 0.0f ? low / sc : 0.0f);                // at most 1, a power of two
        sc = isinf(low) ? 0.0f : low;
        for (int o = 16; o > 0; o >>= 1) {
            s1.add_lane(o);
            s2.add_lane(o);
        }
    }
};

// f of every four (one at the end, one by one where the planes are not aligned) of this thread's values
template <bool VEC, class F>
__device__ __forceinline__ void each_pair(const float *a, const float *b, long long n, F f)
{
    const long long t0 = blockIdx.x * 256LL + threadIdx.x, step = gridDim.x * 256LL;
    auto one = [&](long long i) {
        const float x[1] = {a[i]}, y[1] = {b[i]};
        f(x, y);
    };
    if (VEC) {
        const long long nq = n / 4;
#pragma unroll 2
        for (long long i = t0; i < nq; i += step) {
            const float4 p = reinterpret_cast<const float4 *>(a)[i], q = reinterpret_cast<const float4 *>(b)[i];
            const float x[4] = {p.x, p.y, p.z, p.w}, y[4] = {q.x, q.y, q.z, q.w};
            f(x, y);
        }
        if (t0 < n - 4 * nq)
            one(4 * nq + t0);
    } else {
        for (long long i = t0; i < n; i += step)
            one(i);
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256) k_diff_stats(const float *a, const float *b, long long n, double *st)
{
    __shared__ double red[2][8];
    DiffSums d;
    each_pair<VEC>(a, b, n, [&](const auto &x, const auto &y) { d.add(x, y); });
    double f1 = 0.0, f2 = 0.0;
    if (__any_sync(0xffffffffu, d.far)) {
        each_pair<VEC>(a, b, n, [&](const auto &x, const auto &y) { DiffSums::add_far(x, y, f1, f2); });
        for (int o = 16; o > 0; o >>= 1) {
            f1 += __shfl_xor_sync(0xffffffffu, f1, o);
            f2 += __shfl_xor_sync(0xffffffffu, f2, o);
        }
        d.far = true;
    }
    d.warp_sum();
    if ((threadIdx.x & 31) == 0) {
        const double is = d.sc > 0.0f ? 1.0f / d.sc : 0.0f;   // exact: a power of two
        double v1 = d.s1.value(), v2 = d.s2.value() * is * is;
        if (d.far) {
            v1 += f1;
            v2 += f2;
        }
        red[0][threadIdx.x >> 5] = v1;
        red[1][threadIdx.x >> 5] = v2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w)
            t += red[threadIdx.x][w];
        atomicAdd(st + threadIdx.x, t);
    }
}

__global__ void k_features(const float *lnK, const float *S, const float *Sp, const float *P,
                           const float *Pp, const double *dss, const double *dps, bf16 *feat,
                           long long n, float sm, float ss)
{
    // the standard deviations once per block: an FP64 root and divisions in every thread took 55 of
    // the 63 us of a 1024^2 plane
    __shared__ float sd[2];
    if (threadIdx.x < 2)
        sd[threadIdx.x] = 1.0f / sd_of(threadIdx.x ? dps : dss, n);
    __syncthreads();
    const float inv_ds = sd[0], inv_dp = sd[1];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        __align__(16) bf16 o[16];
#pragma unroll
        for (int c = 0; c < 16; ++c)
            o[c] = __float2bfloat16_rn(0.0f);
        o[0] = __float2bfloat16_rn(lnK[i]);
        o[1] = __float2bfloat16_rn((S[i] - sm) / ss);
        o[2] = __float2bfloat16_rn((S[i] - Sp[i]) * inv_ds);
        o[3] = __float2bfloat16_rn((P[i] - Pp[i]) * inv_dp);
        uint4 *dst = reinterpret_cast<uint4 *>(feat + i * 16);
        dst[0] = reinterpret_cast<const uint4 *>(o)[0];
        dst[1] = reinterpret_cast<const uint4 *>(o)[1];
    }
}

__global__ void k_target(const float *Pn, const float *P, const float *Pp, const double *dps,
                         float *out, long long n)
{
    __shared__ float sd;
    if (threadIdx.x == 0)
        sd = 1.0f / sd_of(dps, n);
    __syncthreads();
    const float inv_dp = sd;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = (Pn[i] - (2.0f * P[i] - Pp[i])) * inv_dp;
}

__global__ void k_predict(const float *P, const float *Pp, const float *d, const double *dps,
                          float *out, long long n)
{
    __shared__ float sh;
    if (threadIdx.x == 0)
        sh = sd_of(dps, n);
    __syncthreads();
    const float sd = sh;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = (2.0f * P[i] - Pp[i]) + sd * d[i];
}

// VEC: g is 16-byte aligned (else 2-byte stores)
template <bool VEC>
__global__ void k_mse_grad(const float *y0, const float *t, bf16 *g, double *loss, long long n,
                           int cout)
{
    __shared__ double red[8];
    double s = 0.0;
    const float sc = 2.0f / (float)n;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const float e = y0[i] - t[i];
        s += (double)e * e;
        if (VEC) {
            // 2-byte stores took 89 us where the bytes need 6 (2^20 pixels, 16 channels)
            uint4 *dst = reinterpret_cast<uint4 *>(g + i * cout);
            dst[0] = make_uint4((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(sc * e)), 0u, 0u, 0u);
            for (int c = 1; c < cout / 8; ++c)
                dst[c] = make_uint4(0u, 0u, 0u, 0u);
        } else {
            g[i * cout] = __float2bfloat16_rn(sc * e);
            for (int c = 1; c < cout; ++c)
                g[i * cout + c] = __float2bfloat16_rn(0.0f);
        }
    }
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
            tot += red[w];
        atomicAdd(loss, tot / (double)n);
    }
}

// ---- launch helpers -----------------------------------------------------------------------
int g_sms = 0;

int sm_count()
{
    if (g_sms <= 0) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            g_sms = 1;
    }
    return g_sms;
}

// CTAs of `func` that fit on one SM by its registers, threads and `smem` bytes of dynamic
// shared memory (the occupancy rule written out from the device attributes), and by the tensor
// memory (tmem_cols of the 512 columns per CTA)
int resident_per_sm(const void *func, size_t smem, int threads, uint32_t tmem_cols)
{
    int dev = 0, smem_sm = 0, reserved = 0, regs_sm = 0, thr_sm = 0;
    cudaFuncAttributes fa{};
    if (cudaGetDevice(&dev) != cudaSuccess || cudaFuncGetAttributes(&fa, func) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) != cudaSuccess)
        return 1;
    const long long per_smem = (long long)smem_sm / ((long long)smem + fa.sharedSizeBytes + reserved);
    const int regs_cta = ((fa.numRegs * 32 + 255) / 256) * 256 * (threads / 32);
    const long long per_regs = regs_cta > 0 ? regs_sm / regs_cta : 1;
    long long per = per_smem < per_regs ? per_smem : per_regs;
    per = per < thr_sm / threads ? per : thr_sm / threads;
    per = per < 512 / (long long)tmem_cols ? per : 512 / (long long)tmem_cols;
    return per < 1 ? 1 : (int)per;
}

template <int CIN, int COUT>
cudaError_t launch_conv(const ConvArgs &a, cudaStream_t s)
{
    const size_t smem = conv_rows_smem_bytes<CIN, COUT>();
    cudaError_t e = cudaFuncSetAttribute(k_conv3x3_rows<CIN, COUT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    // all of the unified L1/shared storage as shared memory, so that two CTAs (95 KB each at 32 input
    // and output channels) fit on an SM
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_conv3x3_rows<CIN, COUT>,
                                 cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess)
        return e;
    // the runtime's occupancy query answered one CTA per SM for a kernel of this kind where ncu's
    // limits gave what its registers and shared memory allow, so they are computed here
    const int per_sm = resident_per_sm((const void *)k_conv3x3_rows<CIN, COUT>, smem, kCvThreads,
                                       kCvTmemCols);
    const long long tiles = (long long)a.nimg * a.H * ((a.W + 127) / 128);
    long long grid = (long long)sm_count() * per_sm;
    if (grid > tiles)
        grid = tiles;
    k_conv3x3_rows<CIN, COUT><<<(unsigned)grid, kCvThreads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int CIN, int COUT>
cudaError_t launch_wgrad(const WgradArgs &a, cudaStream_t s)
{
    const size_t smem = wgrad_smem_bytes<CIN, COUT>();
    cudaError_t e = cudaFuncSetAttribute(k_conv3x3_wgrad<CIN, COUT>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_conv3x3_wgrad<CIN, COUT>,
                                 cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess)
        return e;
    const long long ksteps = ((long long)a.nimg * a.H * a.W + 15) / 16;
    long long chains = sm_count() / ((9 * CIN + 127) / 128);
    if (chains < 1)
        chains = 1;
    if (chains > ksteps)
        chains = ksteps;
    k_conv3x3_wgrad<CIN, COUT><<<dim3(3, (unsigned)chains), wgrad_threads(CIN), smem, s>>>(a);
    return cudaGetLastError();
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool shape_ok(int n_img, int H, int W, int c_in, int c_out)
{
    return n_img >= 1 && H >= 1 && W >= 1 && (c_in == 16 || c_in == 32) &&
           (c_out == 16 || c_out == 32) && (long long)n_img * H * W < (1LL << 40);
}

unsigned grid_for(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    const long long cap = (long long)sm_count() * 16;
    if (b > cap)
        b = cap;
    return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace lbm2p_op

using namespace lbm2p_op;
using lbm2p_internal::set_global_error;

extern "C" {

lbm2p_status lbm2p_op_conv3x3(const void *x, const void *w, const float *bias, const void *mask,
                              void *y, float *y0, int n_img, int H, int W, int c_in, int c_out,
                              int act, int *err, void *stream)
{
    if (!shape_ok(n_img, H, W, c_in, c_out))
        return set_global_error(LBM2P_EINVAL, "conv3x3: need n_img, H, W >= 1 and C_in, C_out in {16, 32}");
    if (!x || !w || !err || (!y && !y0) || act < 0 || act > 1)
        return set_global_error(LBM2P_EINVAL, "conv3x3: x, w, err and one of y, y0 are required; act 0 or 1");
    if (!aligned16(x) || !aligned16(w) || (y && !aligned16(y)) || (mask && !aligned16(mask)))
        return set_global_error(LBM2P_EINVAL, "conv3x3: x, w, y and mask must be 16-byte aligned");
    if (y && (y == x || y == mask))
        return set_global_error(LBM2P_EINVAL, "conv3x3: y must not alias x or mask");
    ConvArgs a{};
    a.x = static_cast<const bf16 *>(x);
    a.w = static_cast<const bf16 *>(w);
    a.bias = bias;
    a.mask = static_cast<const bf16 *>(mask);
    a.y = static_cast<bf16 *>(y);
    a.y0 = y0;
    a.nimg = n_img;
    a.H = H;
    a.W = W;
    a.act = act;
    a.err = err;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e;
    if (c_in == 16)
        e = c_out == 16 ? launch_conv<16, 16>(a, s) : launch_conv<16, 32>(a, s);
    else
        e = c_out == 16 ? launch_conv<32, 16>(a, s) : launch_conv<32, 32>(a, s);
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "conv3x3 launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_conv3x3_wgrad(const void *x, const void *g, float *dw, float *dbias,
                                    int n_img, int H, int W, int c_in, int c_out, int accumulate,
                                    int *err, void *stream)
{
    if (!shape_ok(n_img, H, W, c_in, c_out))
        return set_global_error(LBM2P_EINVAL, "conv3x3_wgrad: need n_img, H, W >= 1 and C_in, C_out in {16, 32}");
    if (!x || !g || !dw || !err || !aligned16(x) || !aligned16(g))
        return set_global_error(LBM2P_EINVAL, "conv3x3_wgrad: x, g (16-byte aligned), dw and err are required");
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaSuccess;
    if (!accumulate) {
        e = cudaMemsetAsync(dw, 0, (size_t)9 * c_in * c_out * sizeof(float), s);
        if (e == cudaSuccess && dbias)
            e = cudaMemsetAsync(dbias, 0, (size_t)c_out * sizeof(float), s);
        if (e != cudaSuccess)
            return set_global_error(LBM2P_ECUDA, "conv3x3_wgrad: clearing failed: %s", cudaGetErrorString(e));
    }
    WgradArgs a{};
    a.x = static_cast<const bf16 *>(x);
    a.g = static_cast<const bf16 *>(g);
    a.dw = dw;
    a.db = dbias;
    a.nimg = n_img;
    a.H = H;
    a.W = W;
    a.err = err;
    if (c_in == 16)
        e = c_out == 16 ? launch_wgrad<16, 16>(a, s) : launch_wgrad<16, 32>(a, s);
    else
        e = c_out == 16 ? launch_wgrad<32, 16>(a, s) : launch_wgrad<32, 32>(a, s);
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "conv3x3_wgrad launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_flip_weights(const void *w, void *wt, int c_in, int c_out, void *stream)
{
    if (!w || !wt || w == wt || !shape_ok(1, 1, 1, c_in, c_out))
        return set_global_error(LBM2P_EINVAL, "flip_weights: distinct w, wt and C_in, C_out in {16, 32}");
    const int n = 9 * c_in * c_out;
    k_flip<<<(n + 255) / 256, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        static_cast<const bf16 *>(w), static_cast<bf16 *>(wt), c_in, c_out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "flip_weights launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_adam(float *p, const float *g, float *m, float *v, void *pb, long long n,
                           float lr, float beta1, float beta2, float eps, int t, void *stream)
{
    if (!p || !g || !m || !v || n < 1 || t < 1 || !(lr > 0.0f) || !(eps > 0.0f) ||
        !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f))
        return set_global_error(LBM2P_EINVAL, "adam: bad arguments");
    const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
    k_adam<<<grid_for(n, 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        p, g, m, v, static_cast<bf16 *>(pb), n, lr, beta1, beta2, eps, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "adam launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_diff_stats(const float *a, const float *b, long long n, double *stats,
                                 void *stream)
{
    if (!a || !b || !stats || n < 1)
        return set_global_error(LBM2P_EINVAL, "diff_stats: bad arguments");
    // a block adds 4096 differences at least (its FP64 end costs as much as some 2000), and the grid
    // fills the SMs four times at most
    long long blocks = (n + 4095) / 4096;
    blocks = blocks < 4LL * sm_count() ? blocks : 4LL * sm_count();
    if (aligned16(a) && aligned16(b))
        k_diff_stats<true><<<(unsigned)blocks, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(a, b, n, stats);
    else
        k_diff_stats<false><<<(unsigned)blocks, 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(a, b, n, stats);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "diff_stats launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_features(const float *lnK, const float *S, const float *S_prev,
                               const float *P, const float *P_prev, const double *ds_stats,
                               const double *dp_stats, void *feat, int H, int W, float s_mean,
                               float s_scale, void *stream)
{
    if (!lnK || !S || !S_prev || !P || !P_prev || !ds_stats || !dp_stats || !feat || H < 1 ||
        W < 1 || !aligned16(feat) || !(s_scale > 0.0f))
        return set_global_error(LBM2P_EINVAL, "features: bad arguments");
    const long long n = (long long)H * W;
    k_features<<<grid_for(n, 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        lnK, S, S_prev, P, P_prev, ds_stats, dp_stats, static_cast<bf16 *>(feat), n, s_mean,
        s_scale);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "features launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_target(const float *P_next, const float *P, const float *P_prev,
                             const double *dp_stats, float *tgt, int H, int W, void *stream)
{
    if (!P_next || !P || !P_prev || !dp_stats || !tgt || H < 1 || W < 1)
        return set_global_error(LBM2P_EINVAL, "target: bad arguments");
    const long long n = (long long)H * W;
    k_target<<<grid_for(n, 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        P_next, P, P_prev, dp_stats, tgt, n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "target launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_predict(const float *P, const float *P_prev, const float *d,
                              const double *dp_stats, float *P_pred, int H, int W, void *stream)
{
    if (!P || !P_prev || !d || !dp_stats || !P_pred || H < 1 || W < 1)
        return set_global_error(LBM2P_EINVAL, "predict: bad arguments");
    const long long n = (long long)H * W;
    k_predict<<<grid_for(n, 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        P, P_prev, d, dp_stats, P_pred, n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "predict launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

lbm2p_status lbm2p_op_mse_grad(const float *y0, const float *tgt, void *g, double *loss,
                               long long npix, int c_out, void *stream)
{
    if (!y0 || !tgt || !g || !loss || npix < 1 || (c_out != 16 && c_out != 32))
        return set_global_error(LBM2P_EINVAL, "mse_grad: bad arguments");
    const auto kernel = aligned16(g) ? k_mse_grad<true> : k_mse_grad<false>;
    kernel<<<grid_for(npix, 256), 256, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        y0, tgt, static_cast<bf16 *>(g), loss, npix, c_out);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess)
        return set_global_error(LBM2P_ECUDA, "mse_grad launch failed: %s", cudaGetErrorString(e));
    return LBM2P_OK;
}

}  // extern "C"
