// The residual of a checking sweep (Sec. 3's stopping test) from its partial sums, and the cluster
// operations that it and the on-chip solve use.
#pragma once

#include <cuda_runtime.h>

#include "lbm2p_device.cuh"

namespace lbm2p_dev {

__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ unsigned cluster_size()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_arrive()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_wait()
{
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void cluster_sync()
{
    cluster_arrive();
    cluster_wait();
}

// the address of this block's shared address `a` in block `rank` of the cluster
__device__ __forceinline__ unsigned cluster_addr(unsigned a, unsigned rank)
{
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

// What bounds this: it runs alone between two launches of the loop, so its latency counts, and an
// FP64 instruction occupies its SM for 16 cycles.  One block that added every partial (a tree per
// component, five divisions in one thread) took 8.2 us at 1024^2 and 18.4 us at 4096^2.
// Now a cluster of kFinBlocks blocks divides the additions, a thread adds one component (four loads
// in flight), the trees are shuffles, and the two variances are formed in two lanes.
constexpr int kFinBlocks = 8;
constexpr int kFinThreads = 256;

// r = ||dP - mean dP|| / ||P - mean P|| from nparts partials of four sums each (FP64, in an order
// fixed by nparts).  CL blocks of kFinThreads threads; true in the lanes of warp 0 of block 0, where
// lane 0 holds r.  Updates shift (the constants that this check subtracted and the next
// will; nullptr: none) and, when given, out.
template <int CL>
__device__ __forceinline__ bool finalize_residual(const double *__restrict__ partials, int nparts,
                                                  long long nnodes, float *shift, ResidualOut *out,
                                                  double &r)
{
    __shared__ double red[kFinThreads / 32][4];
    __shared__ double all[8][4];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = tid & 3;
    const unsigned rank = CL > 1 ? cluster_rank() : 0u;
    if (CL > 1)
        cluster_arrive();                             // block 0 runs: its shared memory is there
    const int step = CL * (kFinThreads / 4);
    double s = 0.0;
    for (int i = (int)rank * (kFinThreads / 4) + (tid >> 2); i < nparts; i += 4 * step) {
        double v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
            v[j] = i + j * step < nparts ? partials[4 * (size_t)(i + j * step) + c] : 0.0;
        s += (v[0] + v[1]) + (v[2] + v[3]);
    }
    auto tree = [](double v) {                        // over the lanes of one component
#pragma unroll
        for (int h = 4; h < 32; h <<= 1)
            v += __shfl_xor_sync(0xffffffffu, v, h);
        return v;
    };
    s = tree(s);
    if (lane < 4)
        red[warp][lane] = s;
    __syncthreads();
    double v = 0.0;
    if (warp == 0)
        v = tree(red[lane >> 2][c]);
    if (CL > 1) {
        cluster_wait();
        if (warp == 0 && lane < 4) {
            const unsigned a = cluster_addr((unsigned)__cvta_generic_to_shared(&all[rank][lane]), 0);
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
        }
        cluster_sync();
        if (warp == 0 && rank == 0)
            v = tree((lane >> 2) < CL ? all[lane >> 2][c] : 0.0);
    }
    if (warp != 0 || rank != 0)
        return false;
    // sums of (dP - dP_prev - shift[1]) and (P - shift[0]): variances are shift invariant.  Even
    // lanes form that of the first, odd lanes that of the second.
    const bool finite = __all_sync(0xffffffffu, isfinite(v));
    const int odd = lane & 1;
    const double s1 = __shfl_sync(0xffffffffu, v, 2 * odd);
    const double s2 = __shfl_sync(0xffffffffu, v, 2 * odd + 1);
    const double mean = s1 / (double)nnodes;
    double var = s2 - s1 * mean;
    var = var > 0.0 ? var : 0.0;
    const double num = __shfl_sync(0xffffffffu, var, 0);
    const double den = __shfl_sync(0xffffffffu, var, 1);
    r = !finite ? nan("") : (den > 0.0 ? sqrt(num / den) : (num > 0.0 ? INFINITY : 0.0));
    if (lane < 2) {
        const double base = (shift ? (double)shift[1 - lane] : 0.0) + mean;
        if (out && lane == 1)
            out->mean_P = base;
        if (finite && shift)
            shift[1 - lane] = (float)base;
    }
    if (out) {
        if (lane == 0)
            out->r = r;
        if (lane < 4)
            out->sums[lane] = v;
    }
    return true;
}

}  // namespace lbm2p_dev
