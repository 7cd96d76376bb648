// qmcrt_support.cuh -- the support of a padded grid, with which walks end where a ray has left
// the medium (support_batches): found anew on the device by every run that uses it.
#pragma once

#include "qmcrt_device.cuh"

namespace qmcrt {

// Support of a padded grid: the largest squared distance, in half edges of the box, of a nonzero
// cell's farthest corner from the box centre (ball) and from the line along z through it
// (cylinder).  `support`: two words, cleared by the caller.  One read of the grid a run.
template <class T>
static __global__ void __launch_bounds__(256) k_support(const __grid_constant__ MediumP<T> G, uint32_t *support)
{
    const int lane = threadIdx.x & 31, rows = G.n[1] * G.n[2], warps = gridDim.x * 8;
    auto far2 = [](int c, int n) {
        const float a = 2.0f * c / n - 1.0f, b = 2.0f * (c + 1) / n - 1.0f;
        return fmaxf(a * a, b * b);
    };
    float ball = 0.0f, cyl = 0.0f;
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += warps) {
        const int z = r / G.n[1], y = r - z * G.n[1];
        const float *row = G.k + ((size_t)(z + G.pad) * G.stride[2] + (size_t)(y + G.pad) * G.stride[1] + G.pad);
        float x2 = -1.0f;
        for (int x = lane; x < G.n[0]; x += 32)
            if (__ldg(row + x) > 0.0f) x2 = fmaxf(x2, far2(x, G.n[0]));
        if (x2 >= 0.0f) {
            const float y2 = far2(y, G.n[1]);
            cyl = fmaxf(cyl, x2 + y2);
            ball = fmaxf(ball, x2 + y2 + far2(z, G.n[2]));
        }
    }
    // positive floats order as integers
    const uint32_t b = __reduce_max_sync(FULL_MASK, __float_as_uint(ball)), c = __reduce_max_sync(FULL_MASK, __float_as_uint(cyl));
    if (lane == 0 && b) {
        atomicMax(support, b);
        atomicMax(support + 1, c);
    }
}

}  // namespace qmcrt
