// lbm_reduce.cuh -- FP64 block reduction used by the per-physics reduction
// kernels (mass, momentum, residual norms and a bad-node count).
#pragma once

#include "lbm_internal.h"

namespace lbm {

// Accumulator of one thread; reduced across the block through shared memory (one
// warp per value) and written as one partial per block (no atomics: the result
// is deterministic).
struct RedAcc {
    double v[RED_WIDTH];
    __device__ void zero() {
#pragma unroll
        for (int k = 0; k < RED_WIDTH; ++k) v[k] = 0.0;
    }
};

// One warp sums one value's 256 entries: 96 warp-wide FP64 additions per block,
// where shuffling every value in every warp takes 320 (the reductions are bound
// by the FP64 pipe).
__device__ __forceinline__ void block_reduce_store(RedAcc& a, double* __restrict__ partials) {
    static_assert(RED_THREADS == 32 * RED_WIDTH, "one warp per value");
    __shared__ double sh[RED_WIDTH][RED_THREADS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < RED_WIDTH; ++k) sh[k][threadIdx.x] = a.v[k];
    __syncthreads();
    double x = 0.0;
#pragma unroll
    for (int j = 0; j < RED_THREADS / 32; ++j) x += sh[warp][32 * j + lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if (lane == 0) partials[(size_t)blockIdx.x * RED_WIDTH + warp] = x;
}

// The reduction kernels walk the nodes with a grid stride over their index, all
// threads busy whatever nx is, and find a node's coordinates with 32-bit
// multiplications (x-rows cut into 256-node chunks, 64-bit divisions per chunk and
// idle threads past the row's end: 114 us per lbm_reduce at 100^3, now 78 us).
// They are bound by the FP64 pipe (84 % busy): 9 fused multiply-adds, 7 additions
// and 7 conversions a node, 16 cycles per warp instruction, 77 us of the 124 us of
// an lbm_reduce at 128^3; the sums stay in FP64.  (lbm_reduce_state_noalloc keeps the
// chunks of a row.)
struct NodeDiv {
    FastDiv nx, ny;
};
inline NodeDiv node_div(const Box& b) { return {make_fast_div((uint32_t)b.nx), make_fast_div((uint32_t)b.ny)}; }
__device__ __forceinline__ void node_of(uint32_t k, const Box& b, NodeDiv d, int& x, int& y, int& z) {
    const uint32_t row = fast_div(k, d.nx);
    x = (int)(k - row * (uint32_t)b.nx);
    z = (int)fast_div(row, d.ny);
    y = (int)(row - (uint32_t)z * (uint32_t)b.ny);
}

// The previous check's velocity of a node, loaded ahead of the populations so that
// all of a node's loads are in flight together (loaded after them, where it is
// used, they are a second round trip to memory that 24 warps per SM do not hide:
// 128^3, us per lbm_reduce: fluid 282, MHD 354, colour gradient 286; now 123, 127,
// 128; FP64 fluid 437, now 313).  It is read once: past the L1.
template <typename C>
__device__ __forceinline__ void load_prev(const C* uprev, size_t n, uint32_t cell, bool have_prev, C up[3]) {
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = have_prev ? __ldcg(uprev + k * n + cell) : (C)0;
}

// Accumulate one node, with the previous check's velocity up (if have_prev).
// Records u.
template <typename C>
__device__ __forceinline__ void reduce_node(RedAcc& a, C rho, C ux, C uy, C uz, const C up[3], C* uprev, size_t n,
                                            uint32_t cell, bool have_prev, bool record) {
    const bool bad = !(rho > (C)0) || !isfinite(rho) || !isfinite(ux) || !isfinite(uy) || !isfinite(uz);
    if (bad) {
        a.v[6] += 1.0;
        return;
    }
    const double r = (double)rho, x = (double)ux, y = (double)uy, z = (double)uz;
    a.v[0] += r;
    a.v[1] += r * x;
    a.v[2] += r * y;
    a.v[3] += r * z;
    a.v[5] = fma(x, x, fma(y, y, fma(z, z, a.v[5])));
    if (have_prev) {
        const double dx = x - (double)up[0], dy = y - (double)up[1], dz = z - (double)up[2];
        a.v[4] = fma(dx, dx, fma(dy, dy, fma(dz, dz, a.v[4])));
    }
    if (record) {
        __stcg(uprev + cell, ux);
        __stcg(uprev + n + cell, uy);
        __stcg(uprev + 2 * n + cell, uz);
    }
}

}  // namespace lbm
