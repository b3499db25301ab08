// Four pressure sweeps (Eq. 3-1, pull stream + BGK collide) per launch on lattices with walls on
// every side.
//
// What bounded the sub-iteration was the launches that carry two sweeps (k_pressure_rows2,
// k_pressure_pair_direct): 154 thread instructions per node and sweep and 36 B per node and sweep.
// Here a warp owns a tile of 56 columns by H rows and carries four sweeps in registers, about 55
// thread instructions and 18 B per node and sweep:
//   - each lane holds two neighbouring columns, so the collision, the sum of Eq. 3-9a and the
//     unshifted pulls are packed FP32 pairs (add / mul / fma .rn.f32x2, the same IEEE roundings
//     as the scalar operations), half the issue slots of one column per lane;
//   - a pull from a neighbouring column needs one warp shuffle per pair of columns;
//   - the 64 columns of a warp are the 56 it owns and four on each side (one per sweep, and the
//     segment starts on a 16-byte boundary), so warps exchange nothing: no block barrier;
//   - input rows are copied by cp.async (16 bytes per lane) into the warp's own ring of 7 slots,
//     four rows ahead, and waited for by the warp's own copy groups (one cp.async.bulk per plane
//     and row took 115 us per sweep at 4096^2 where these take 88: 256-byte bulk copies cost about
//     40 cycles each).
// Sweep s runs s - 1 rows behind sweep 1.  Of a sweep's values a lane keeps what the next sweep
// still needs: directions 1 and 3 of the last row, 2, 5, 6 (pulled from below) of the last two,
// R of six rows, 1/tau_f of four.  Two warps per scheduler with up to 255 registers: three with 168
// spill inside the row loop (381 against 231 us per launch at 4096^2, whose memory system the
// spills share).  A tile whose footprint holds no wall node takes the interior path; the others
// apply the wall rules of Sec. 4 as selects and keep the planes that the rules read.  The edge
// path is one row body with guards for the filling sweeps, not unrolled: few tiles run it, so its
// instruction fetches are cold (unrolled, the tile at a corner took 500k cycles at 4096^2 where an
// interior tile took 60k).  The interior path exists in both forms: unrolled by two with straight-line
// filling rows it has fewer instructions, as one guarded row it leaves the instruction cache to the
// edge tiles beside it.  Create times both: the first is ahead at 1024^2 (19.4 against 22.2 us per
// launch), the second at 2048^2 (61.9 against 65.6) and, by little, at 512^2 and 4096^2; for batches it
// is the only one.
// The per-node operations and their order are those of the single sweep (dev1, pressure_of,
// collide1), so four sweeps equal four launches of one bit for bit.
// Per sweep, two-sweep launches before and this kernel now: 4096^2 129.5 and 55.2 us (221 us per
// launch, 1.24 times the time that its 1208 MB take at the copy bandwidth), 1024^2 14.0 and
// 4.9 us, 512^2 7.5 and 3.1 us.
#include <cuda_runtime.h>

#include <cstdint>

#include "lbm2p_async.cuh"
#include "lbm2p_device.cuh"
#include "lbm2p_node.cuh"
#include "sweep_quad.cuh"

namespace lbm2p_dev {
namespace {

template <bool CHECK, int S, bool UNROLL>
__global__ void __launch_bounds__(kQuadThreads, kQuadBlocks)
    k_pressure_quad(const __grid_constant__ PressureArgs a, int H)
{
    extern __shared__ __align__(128) float smem_raw[];
    const int lane = threadIdx.x;
    ResAcc racc;
    if (blockIdx.x < QuadPlan(H, a.g.nx, a.g.ny).tiles())
        quad_tile<CHECK, S, UNROLL>(a, H, blockIdx.x, smem_raw, lane, racc);
    if (CHECK) {
        double v[4];
        racc.warp_totals(v);
        if (lane == 0)
            for (int c = 0; c < 4; ++c)
                a.partials[4 * (size_t)blockIdx.x + c] = v[c];
    }
}

// Four sweeps over several lattices in one launch (members of a batch): block t runs the tile
// items[t] = (member m, tile of H[m] rows) with the argument block pa[2 m + parity]; CHECK: its
// residual sums go to parts[4 (pb0[m] + tile) ..].  The grid covers the items of every member and
// the blocks beyond *nitems leave at once, so the hardware balances tiles of different cost.  The
// argument block is read from shared memory: from global memory the compiler keeps it in registers
// and the tile spills.
template <bool CHECK, int S>
__global__ void __launch_bounds__(kQuadThreads, kQuadBlocks)
    k_quad_batch(const PressureArgs *__restrict__ pa, const int *__restrict__ H,
                 const int *__restrict__ pb0, const int2 *__restrict__ items,
                 const int *__restrict__ nitems, int parity, double *__restrict__ parts)
{
    extern __shared__ __align__(128) float smem_raw[];
    __shared__ PressureArgs a;
    if ((int)blockIdx.x >= *nitems)
        return;
    const int lane = threadIdx.x;
    const int2 e = items[blockIdx.x];
    const unsigned *src = reinterpret_cast<const unsigned *>(pa + 2 * e.x + parity);
    for (int i = lane; i < (int)(sizeof(PressureArgs) / 4); i += 32)
        reinterpret_cast<unsigned *>(&a)[i] = src[i];
    __syncwarp();
    ResAcc racc;
    quad_tile<CHECK, S, false>(a, H[e.x], e.y, smem_raw, lane, racc);
    if (CHECK) {
        double v[4];
        racc.warp_totals(v);
        if (lane == 0)
            for (int c = 0; c < 4; ++c)
                parts[4 * ((size_t)pb0[e.x] + e.y) + c] = v[c];
    }
}

void *quad_batch_func(bool check)
{
    return check ? (void *)k_quad_batch<true, kQuadSlots> : (void *)k_quad_batch<false, kQuadSlots>;
}

void *quad_func(bool check, bool unroll)
{
    if (unroll)
        return check ? (void *)k_pressure_quad<true, kQuadSlots, true>
                     : (void *)k_pressure_quad<false, kQuadSlots, true>;
    return check ? (void *)k_pressure_quad<true, kQuadSlots, false>
                 : (void *)k_pressure_quad<false, kQuadSlots, false>;
}

}  // namespace
}  // namespace lbm2p_dev

namespace lbm2p_launch {

using lbm2p_dev::PressureArgs;
using namespace lbm2p_dev;

long long quad_grid(int H, int nx, int ny)
{
    return QuadPlan(H, nx, ny).tiles();
}

int quad_tile_slots(bool has_fp)
{
    int dev = 0, sms = 0, lo = 1 << 30;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    for (bool c : {false, true}) {
        int b = 0;
        for (bool u : {false, true}) {
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, quad_func(c, u), kQuadThreads,
                                                              quad_smem_bytes(has_fp)) != cudaSuccess)
                return 0;
            lo = b < lo ? b : lo;
        }
    }
    return sms * lo;
}

cudaError_t quad_prepare()
{
    for (bool c : {false, true})
        for (void *f : {quad_func(c, false), quad_func(c, true), quad_batch_func(c)}) {
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)quad_smem_bytes(true));
            if (e != cudaSuccess)
                return e;
        }
    return cudaSuccess;
}

void pressure_sweeps_quad(const PressureArgs &a, bool check, int H, bool unroll, int grid, void *stream)
{
    void *args[] = {(void *)&a, (void *)&H};
    cudaLaunchKernel(quad_func(check, unroll), dim3(grid), dim3(kQuadThreads), args,
                     quad_smem_bytes(a.Fp != nullptr), reinterpret_cast<cudaStream_t>(stream));
}

cudaError_t node_pressure_quad(cudaGraphNode_t *n, cudaGraph_t g, const cudaGraphNode_t *dep,
                               const PressureArgs &a, bool check, int H, bool unroll, int grid)
{
    cudaKernelNodeParams prm{};
    prm.func = quad_func(check, unroll);
    prm.gridDim = dim3((unsigned)grid);
    prm.blockDim = dim3(kQuadThreads);
    prm.sharedMemBytes = (unsigned)quad_smem_bytes(a.Fp != nullptr);
    void *args[] = {(void *)&a, (void *)&H};
    prm.kernelParams = args;
    prm.extra = nullptr;
    return cudaGraphAddKernelNode(n, g, dep, dep ? 1 : 0, &prm);
}

int quad_batch_slots()
{
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return kQuadBlocks;
    return sms * kQuadBlocks;
}

int quad_tiles(int H, int nx, int ny)
{
    return (int)QuadPlan(H, nx, ny).tiles();
}

cudaError_t node_quad_batch(cudaGraphNode_t *n, cudaGraph_t g, const cudaGraphNode_t *dep,
                            const PressureArgs *pa, const int *H, const int *pb0,
                            const int2 *items, const int *nitems, int parity, bool check,
                            double *parts, int grid, bool has_fp)
{
    cudaKernelNodeParams prm{};
    prm.func = quad_batch_func(check);
    prm.gridDim = dim3((unsigned)grid);
    prm.blockDim = dim3(kQuadThreads);
    prm.sharedMemBytes = (unsigned)quad_smem_bytes(has_fp);
    void *args[] = {(void *)&pa, (void *)&H, (void *)&pb0, (void *)&items, (void *)&nitems,
                    (void *)&parity, (void *)&parts};
    prm.kernelParams = args;
    prm.extra = nullptr;
    return cudaGraphAddKernelNode(n, g, dep, dep ? 1 : 0, &prm);
}

}  // namespace lbm2p_launch
