// qmcrt_support.cuh -- the support of a padded grid, with which walks end where a ray has left
// the medium (support_batches): found anew on the device by every run that uses it.
#pragma once

#include "qmcrt_device.cuh"

namespace qmcrt {

constexpr float SUPPORT_ALL = 3e38f;  // radii beyond every box: no cut

// scale^2 of a medium's support (see support_batches), to a few float roundings.
template <class T>
static float support_scale2(const MediumP<T> &G)
{
    const double s = 0.5 * G.n[0] * (double)G.h[0] * (double)G.inv_half[0];
    return (float)(s * s);
}

// Support of a padded grid: the largest squared distance, in half edges of the box, of a nonzero
// cell's farthest corner from the box centre (ball) and from the line along z through it
// (cylinder), times scale2.  `support`: two words, cleared by the caller.  One read of the grid a run.
template <class T>
static __global__ void __launch_bounds__(256) k_support(const __grid_constant__ MediumP<T> G, float scale2,
                                                       uint32_t *support)
{
    // already the whole box: nothing to find (set by the caller, or by a block that met a corner cell,
    // which sets both; read through L1: 1216 blocks at one word of L2 take 2 us, and an old value will do)
    if (*support == __float_as_uint(SUPPORT_ALL)) return;
    const int lane = threadIdx.x & 31, rows = G.n[1] * G.n[2], warps = gridDim.x * 8;
    const float per[3] = {2.0f / G.n[0], 2.0f / G.n[1], 2.0f / G.n[2]};  // cell edges in half edges of the box
    auto far2 = [&](int first, int last, int axis) {  // squared distance of the farther end of a run of cells
        const float a = first * per[axis] - 1.0f, b = (last + 1) * per[axis] - 1.0f;
        return fmaxf(a * a, b * b);
    };
    float ball = 0.0f, cyl = 0.0f;
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += warps) {
        const int z = r / G.n[1], y = r - z * G.n[1];
        const float *row = G.k + ((size_t)(z + G.pad) * G.stride[2] + (size_t)(y + G.pad) * G.stride[1] + G.pad);
        int x0 = G.n[0], x1 = -1;  // this lane's first and last nonzero cell of the row
        for (int x = lane; x < G.n[0]; x += 32)
            if (__ldg(row + x) > 0.0f) {
                x0 = min(x0, x);
                x1 = x;
            }
        if (x1 >= 0) {
            const float r2 = far2(x0, x1, 0) + far2(y, y, 1);
            cyl = fmaxf(cyl, r2);
            ball = fmaxf(ball, r2 + far2(z, z, 2));
        }
    }
    // positive floats order as integers; a block's largest first, and to memory only if it exceeds
    // what is there (two atomics a warp and a division a cell: 19 us for a 128^3 grid, 7 now, 17 for 256^3)
    __shared__ uint32_t s_max[2];
    if (threadIdx.x < 2) s_max[threadIdx.x] = 0u;
    __syncthreads();
    const uint32_t b = __reduce_max_sync(FULL_MASK, __float_as_uint(ball)), c = __reduce_max_sync(FULL_MASK, __float_as_uint(cyl));
    if (lane == 0 && b) {
        atomicMax(&s_max[0], b);
        atomicMax(&s_max[1], c);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_max[threadIdx.x]) {
        // no cut where it takes in the whole box (a corner, a column at an edge); 2e-5 for the
        // float rounding of the radii, of positions and of directions
        const float r2 = __uint_as_float(s_max[threadIdx.x]) + 2e-5f;
        const uint32_t bits = __float_as_uint(r2 < (threadIdx.x ? 2.0f : 3.0f) ? r2 * scale2 : SUPPORT_ALL);
        if (bits > *(volatile uint32_t *)(support + threadIdx.x)) atomicMax(support + threadIdx.x, bits);
    }
}

}  // namespace qmcrt
