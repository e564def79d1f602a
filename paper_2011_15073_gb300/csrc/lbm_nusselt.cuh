// lbm_nusselt.cuh -- the wall Nusselt numbers of one cavity by one block of 256
// threads (device code of the single-cavity and the batched kernel).
#pragma once

#include "lbm_device.cuh"

namespace lbm {

// FP64 block sum of one value (blockDim.x a multiple of 32, <= 1024); the
// reduction tree is fixed, so results are reproducible run to run.
__device__ inline double block_sum(double v, double *sh)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (wid == 0) {
        t = lane < nw ? sh[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    }
    return t;  // valid in thread 0
}

// Streamed temperature of node (x, y) in FP64 (thermal part of the pull).
template <int PREC, bool REV>
__device__ double streamed_T(const typename Store<PREC>::S *__restrict__ src,
                             const Phys<typename Store<PREC>::R> &p, int x, int y)
{
    using R = typename Store<PREC>::R;
    R f[9], g[5];
    pull<PREC, R, REV>(src, p, x, y, f, g);
    return (double)g[0] + (double)g[1] + (double)g[2] + (double)g[3] + (double)g[4];
}

// Wall Nusselt numbers by one block; row j of the hot wall gets
// Nu_j = -L (9 theta_0 - theta_1 - 8) / 3, the cold wall the outward
// L (9 theta_{nx-1} - theta_{nx-2}) / 3, theta = (T - T_c) / (T_h - T_c).
// Rows [row_lo, row_hi) (all rows of a whole cavity, the interior rows of a
// slab); sums[0..1] the sums over them, in thread 0.  nuloc may be null.
template <int PREC, bool REV>
__device__ __forceinline__ void nusselt_rows(const typename Store<PREC>::S *__restrict__ src,
                                             const Phys<typename Store<PREC>::R> &p, double T_hot, double T_cold, double Lw,
                                             double *__restrict__ nuloc, int row_lo, int row_hi, double sums[2])
{
    __shared__ double sh[32];
    const double dT = T_hot - T_cold;
    double sh_hot = 0.0, sh_cold = 0.0;
    for (int j = row_lo + threadIdx.x; j < row_hi; j += blockDim.x) {
        const double t0 = (streamed_T<PREC, REV>(src, p, 0, j) - T_cold) / dT;
        const double t1 = (streamed_T<PREC, REV>(src, p, 1, j) - T_cold) / dT;
        const double ta = (streamed_T<PREC, REV>(src, p, p.nx - 1, j) - T_cold) / dT;
        const double tb = (streamed_T<PREC, REV>(src, p, p.nx - 2, j) - T_cold) / dT;
        const double nh = -Lw * (9.0 * t0 - t1 - 8.0) / 3.0;
        const double nc = Lw * (9.0 * ta - tb) / 3.0;
        if (nuloc) nuloc[j] = nh;
        sh_hot += nh;
        sh_cold += nc;
    }
    sums[0] = block_sum(sh_hot, sh);
    sums[1] = block_sum(sh_cold, sh);
}

}  // namespace lbm
