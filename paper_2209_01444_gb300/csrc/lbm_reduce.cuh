// Node pass of the metrics reduction, shared by the handle's reduction
// (lbm_aux.cu) and its allocation-free variant (lbm_noalloc.cu), which
// therefore give the same partials bit for bit.
//
// Block b folds the nodes [b * kRedNodesPerBlock, (b + 1) * kRedNodesPerBlock)
// (row-major over the nx x ny grid, pitch skipped), thread t the nodes
// t, t + kRedThreadsPerBlock, ... of that chunk (16 of them).  A thread sums
// its nodes' small deviations in FP32 (phi + 1, C - 1, H - H_ref, the nine
// flow deviations, max |u|, non-finite count) and adds the constant
// reference terms once, in FP64, with its exact node count; warps and the
// block then combine FP64 values in a fixed order.  GB300 issues FP64 at a
// small fraction of its FP32 rate, so per-node FP64 arithmetic would bound
// this pass well below the memory bandwidth.
//
// Partials per block (kRedValues doubles): sum (1 + phi)/2, sum C, sum H,
// sum of the flow populations, max |u|, non-finite count, sum phi.
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr int kRedValues = 7;
constexpr int kRedThreadsPerBlock = 256;
constexpr int kRedNodesPerBlock = 4096;  // 16 nodes per thread

// Blocks of the node pass for an nx x ny grid.
__host__ __device__ inline long long reduce_chunk_blocks(long long nodes)
{
    return (nodes + kRedNodesPerBlock - 1) / kRedNodesPerBlock;
}

__device__ __forceinline__ double red_warp_sum(double v)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    return v;
}
__device__ __forceinline__ double red_warp_max(double v)
{
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, d));
    return v;
}

template <class Store>
__device__ __forceinline__ void reduce_chunk(const StepParams& P, const void* __restrict__ sc,
                                             const void* __restrict__ fl, double* __restrict__ partials)
{
    // (grids hold at most 2^31 nodes: 32-bit division, once per thread)
    const unsigned N = (unsigned)P.nx * (unsigned)P.ny;
    const unsigned first = blockIdx.x * (unsigned)kRedNodesPerBlock;
    const unsigned nodes = min((unsigned)kRedNodesPerBlock, N - first);
    unsigned y = (first + threadIdx.x) / (unsigned)P.nx, x = (first + threadIdx.x) - y * (unsigned)P.nx;
    float sp1 = 0.0f, sdC = 0.0f, sdH = 0.0f, sh = 0.0f, umax = 0.0f;
    int bad = 0, count = 0;
    // the next node's 24 loads are in flight while a node is added
    float v[24], w[24];
    auto load = [&](float (&d)[24]) {
        const long long o = (long long)y * P.pitch + x;
#pragma unroll
        for (int i = 0; i < 24; ++i) d[i] = Store::load(sc, fl, i, o, P);
        x += kRedThreadsPerBlock;
        while (x >= (unsigned)P.nx) {
            x -= (unsigned)P.nx;
            ++y;
        }
    };
    if (threadIdx.x < nodes) load(w);
    for (unsigned t = threadIdx.x; t < nodes; t += kRedThreadsPerBlock) {
#pragma unroll
        for (int i = 0; i < 24; ++i) v[i] = w[i];
        if (t + kRedThreadsPerBlock < nodes) load(w);
        const float *f = v + kF, *n = v + kN, *g = v + kG, *h = v + kH;
        const Macro m = node_macros(f, n, g, h, P);
        float s9 = 0.0f;
#pragma unroll
        for (int i = 0; i < 9; ++i) s9 += h[i];
        const float u = sqrtf(m.ux * m.ux + m.uy * m.uy);
        sp1 += m.p1;
        sdC += m.dC;
        sdH += m.dH;
        sh += s9;
        umax = fmaxf(umax, u);
        bad += (isfinite(m.p1) && isfinite(m.dC) && isfinite(m.dth) && isfinite(u)) ? 0 : 1;
        ++count;
    }
    const double c = (double)count;
    double acc[kRedValues];
    acc[0] = 0.5 * (double)sp1;
    acc[1] = c + (double)sdC;
    acc[2] = c * ((double)P.theta_ref + (double)P.latent) + (double)sdH;
    acc[3] = c * (double)P.rho0 + (double)sh;
    acc[4] = (double)umax;
    acc[5] = (double)bad;
    acc[6] = (double)sp1 - c;
    __shared__ double sm[kRedValues][kRedThreadsPerBlock / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kRedValues; ++k) {
        const double v = k == 4 ? red_warp_max(acc[k]) : red_warp_sum(acc[k]);
        if (lane == 0) sm[k][wid] = v;
    }
    __syncthreads();
    if (threadIdx.x < kRedValues) {
        const int k = threadIdx.x;
        double v = sm[k][0];
        for (int w = 1; w < kRedThreadsPerBlock / 32; ++w) v = (k == 4) ? fmax(v, sm[k][w]) : v + sm[k][w];
        partials[(long long)blockIdx.x * kRedValues + k] = v;
    }
}

}  // namespace lbm
