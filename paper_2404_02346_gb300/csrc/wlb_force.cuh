// King's surface integral, Eq. (14), in FP64 (the single-lattice and batched
// force kernels).
#pragma once
#include "wlb_internal.cuh"

namespace wlb {

constexpr int kForceThreads = 256;

// Eq. (14) on the surface elements by one block of kForceThreads, fixed
// reduction order.  Writes 4 doubles; sets *err if a component is not finite.
__device__ __forceinline__ void surface_force_block(const Geometry &g, const double *__restrict__ pts,
                                                    const double *__restrict__ acc64, double inv_nw, double *force,
                                                    int *err) {
    __shared__ double red[3][kForceThreads];
    const int t = threadIdx.x;
    double F[3] = {0.0, 0.0, 0.0};
    const double rho0 = g.rho0;
    const double inv_2rc2 = 1.0 / (2.0 * rho0 * g.c0 * g.c0);
    for (int k = t; k < g.n_surface; k += blockDim.x) {
        const double *row = pts + 7 * (long long)k;
        const double *a = acc64 + 5 * (long long)k;
        const double iso = a[0] * inv_nw * inv_2rc2 - 0.5 * rho0 * (a[1] * inv_nw);
        for (int i = 0; i < 3; ++i) F[i] -= row[6] * (iso * row[3 + i] + rho0 * (a[2 + i] * inv_nw));
    }
    for (int i = 0; i < 3; ++i) red[i][t] = F[i];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (t < s)
            for (int i = 0; i < 3; ++i) red[i][t] += red[i][t + s];
        __syncthreads();
    }
    if (t == 0) {
        for (int i = 0; i < 3; ++i) {
            const double v = i < g.dim ? red[i][0] : 0.0;
            force[i] = v;
            if (!isfinite(v)) atomicExch(err, 1);
        }
        force[3] = 0.0;
    }
}

}  // namespace wlb
