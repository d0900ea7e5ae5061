// Index helpers of the multigrid levels, shared by the E_0 and E_c kernels.
#pragma once

#include <cuda_runtime.h>

#include "mg.h"

namespace rte {

constexpr float kOmega = 0.7f;          // Jacobi damping

__device__ __forceinline__ int nbr(int i, int dir, int m, int n) {
    const int off[7] = {0, 1, -1, m + 1, -(m + 1), m + 2, -(m + 2)};
    const int j = i + off[dir];
    return j < 0 ? 0 : (j >= n ? n - 1 : j);
}

// restriction P^T: fine node q of coarse node I's list (the fine nodes that
// interpolate from I, with their weights; width Cv.rwid, zero-weight padding)
__device__ __forceinline__ int restrict_src(const MGDeviceLevel& Cv, int I, int q, float& w) {
    const size_t k = (size_t)I * Cv.rwid + q;
    w = __ldg(Cv.rw + k);
    return __ldg(Cv.ridx + k);
}

// prolongation: coarse nodes (and weights) interpolating fine node i; the
// coarse mesh is the floor(mf/2)-mesh, and for odd mf the last fine column
// and row take the values of the ones before them
__device__ __forceinline__ void prolong_src(int i, int mf, int& c0, int& c1, float& w0,
                                            float& w1) {
    const int mc = mf / 2;
    const int x = min(i % (mf + 1), 2 * mc), y = min(i / (mf + 1), 2 * mc);
    if (!(x & 1) && !(y & 1)) {
        c0 = c1 = (y / 2) * (mc + 1) + x / 2;
        w0 = 1.f;
        w1 = 0.f;
    } else if ((x & 1) && !(y & 1)) {
        c0 = (y / 2) * (mc + 1) + (x - 1) / 2;
        c1 = c0 + 1;
        w0 = w1 = 0.5f;
    } else if (!(x & 1)) {
        c0 = ((y - 1) / 2) * (mc + 1) + x / 2;
        c1 = c0 + (mc + 1);
        w0 = w1 = 0.5f;
    } else {
        c0 = ((y - 1) / 2) * (mc + 1) + (x - 1) / 2;
        c1 = c0 + (mc + 2);
        w0 = w1 = 0.5f;
    }
}

}  // namespace rte
