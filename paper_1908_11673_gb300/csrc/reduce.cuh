// Deterministic grid reductions shared by the vector kernels (blas.cu) and the
// hopping kernel with fused inner products (hop_dots.cu).  Every block writes its
// FP64 partial sums; the last block to finish (a ticket counter) adds all partials
// in block order, so the result is the same on every run for a given grid.
#pragma once

#include <map>
#include <mutex>

#include "blas.h"
#include "qxd_internal.h"

namespace qxd {

constexpr int kRedThreads = 256;

// Grid of a grid-stride kernel: at most one full wave of resident blocks (the
// occupancy of this kernel on this device, looked up once), and no more blocks
// than the work needs.  A fixed grid for a given device and size keeps the
// order of the reduction, and so its result, the same on every run.
template <typename K>
static int wave_blocks(qxd_ctx* ctx, K kernel, int threads, size_t work_per_block, size_t nch) {
    static std::map<const void*, int> per_sm;  // per kernel instantiation
    static std::mutex mu;
    int b_sm;
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = per_sm.find((const void*)kernel);
        if (it == per_sm.end()) {
            int n = 0;
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, 0) != cudaSuccess || n < 1) {
                cudaGetLastError();
                n = 1;
            }
            it = per_sm.emplace((const void*)kernel, n).first;
        }
        b_sm = it->second;
    }
    size_t cap = (size_t)b_sm * ctx->nsm;
    if (cap > (size_t)kMaxRedBlocks) cap = kMaxRedBlocks;
    size_t need = (nch + work_per_block - 1) / work_per_block;
    return (int)(need < cap ? (need > 0 ? need : 1) : cap);
}

struct RedOut {
    double* partials;
    unsigned* ticket;
    double* result;
};

static RedOut red_out(qxd_ctx* ctx, int slot) { return RedOut{ctx->red_partials, ctx->red_ticket, ctx->red_result + slot}; }

// Sums of NC numbers over the grid from the T threads' values in shared memory vs[c][thread].
// A warp's FP64 addition holds its scheduler for 64 cycles, so each number is summed by one
// group of warps (32 lanes x a few values, five shuffles) instead of by every warp, and the
// last block sums the numbers' partials side by side: with 20 numbers on 42 blocks the whole
// launch took 35 us when every warp shuffled every number and the last block went through them
// one after the other, 22 us so (k_hop_dots on 8 x 28 x 12 x 8; k_multi_dot with eight fields
// 18 -> 10 us).
template <int NC, int T>
__device__ void smem_reduce_finish(double (*vs)[T], const RedOut& o) {
    constexpr int NW = T / 32;
    constexpr int WP = NC >= NW ? 1 : NC > NW / 2 ? 1 : NC > NW / 4 ? 2 : NC > NW / 8 ? 4 : 8;  // warps of a number
    __shared__ double sub[NC][WP];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = warp % WP;
    __syncthreads();
    for (int c = warp / WP; c < NC; c += NW / WP) {
        double x = 0.0;
#pragma unroll
        for (int k = 0; k < NW / WP; ++k) x += vs[c][lane + 32 * (s + WP * k)];
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) x += __shfl_down_sync(0xffffffffu, x, m);
        if (lane == 0) sub[c][s] = x;
    }
    __syncthreads();
    if (threadIdx.x < NC) {
        double x = sub[threadIdx.x][0];
        for (int k = 1; k < WP; ++k) x += sub[threadIdx.x][k];
        o.partials[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = x;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(o.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int nb = gridDim.x;
    for (int c = warp / WP; c < NC; c += NW / WP) {
        const double* part = o.partials + (size_t)c * nb;
        double x = 0.0;
        for (int b = lane + 32 * s; b < nb; b += 4 * 32 * WP) {
            double y[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) y[k] = b + k * 32 * WP < nb ? __ldcg(part + b + k * 32 * WP) : 0.0;
            x += (y[0] + y[1]) + (y[2] + y[3]);
        }
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) x += __shfl_down_sync(0xffffffffu, x, m);
        if (lane == 0) sub[c][s] = x;
    }
    __syncthreads();
    if (threadIdx.x < NC) {
        double x = sub[threadIdx.x][0];
        for (int k = 1; k < WP; ++k) x += sub[threadIdx.x][k];
        o.result[threadIdx.x] = x;
    }
    if (threadIdx.x == 0) *o.ticket = 0u;
}

template <int NC>
__device__ void block_reduce_finish(double v[NC], const RedOut& o) {
    __shared__ double vs[NC][kRedThreads];
#pragma unroll
    for (int c = 0; c < NC; ++c) vs[c][threadIdx.x] = v[c];
    smem_reduce_finish<NC, kRedThreads>(vs, o);
}

}  // namespace qxd
