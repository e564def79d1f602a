// lbm_strip.cu -- launches of the two-steps-in-one kernel (lbm_strip.cuh) on one
// cavity.
#include "lbm_strip.cuh"

#include "lbm_internal.h"

namespace lbm {

namespace {

template <int PREC, int FIELD, int TAU>
__global__ void __launch_bounds__(32, strip_blocks<TAU>())
strip_kernel(const typename Store<PREC>::S *__restrict__ src, typename Store<PREC>::S *__restrict__ dst,
             const float *__restrict__ tsrc, float *__restrict__ tdst, Phys<F2> p, StripPlan plan)
{
    __shared__ typename Store<PREC>::S ring[3][14][64];
    __shared__ float tring[3][64];
    strip_unit<PREC, FIELD, TAU>(src, dst, tsrc, tdst, p, plan, blockIdx.x, ring, tring);
}

template <int PREC, int TAU>
cudaError_t strip_tau(lbm_ctx *c)
{
    using S = typename Store<PREC>::S;
    const int s = c->cur, d = 1 - s;
    // as many units as warps fit on the chip at once (twice as many with the
    // implicit tau)
    const int slots = c->sms * strip_blocks<TAU>() * (TAU == 1 ? 2 : 1);
    StripPlan plan = strip_plan(c->nx);
    plan.cut(c->ny, slots / plan.nstrips);
    const int blocks = plan.units();
    auto *kern = c->d_da ? strip_kernel<PREC, 1, TAU> : strip_kernel<PREC, 0, TAU>;
    kern<<<blocks, 32, 0, c->stream>>>((const S *)c->buf.dist[s], (S *)c->buf.dist[d], (const float *)c->buf.tau[s],
                                       (float *)c->buf.tau[d], make_params<F2>(c), plan);
    c->cur = d;
    return cudaGetLastError();
}
template <int PREC>
cudaError_t strip_t(lbm_ctx *c)
{
    return c->opts.tau_iters > 0 ? strip_tau<PREC, 1>(c) : strip_tau<PREC, 0>(c);
}

}  // namespace

// Measured on the FP32 storages, one step per launch / two (us per step, lagged
// tau): 701 x 499 6.2 / 8.2, 1024 x 640 about 9.0 / 9.4, 1024^2 20.5 / 13.8, 2048^2
// 77 / 46, 4096^2 290 / 174; implicit tau: 2048^2 86 / 74.  Smaller grids stay in
// L2 and have too few rows per warp:
// a segment of four rows takes six rows' first steps, one after the other.
// The 16-bit storages are bound by instruction issue, not by HBM, and keep
// their four-node kernel.
bool two_steps(int nx, int ny, const lbm_opts &o)
{
    if (o.layout != 0 || o.staging != 0 || nx < 128 || ny < 64) return false;
    if (o.prec != LBM_F32 && o.prec != LBM_F32D) return false;
    return (int64_t)nx * ny >= (o.tau_iters > 0 ? 2000000 : 600000);
}

cudaError_t launch_two_steps(lbm_ctx *c)
{
    switch (c->opts.prec) {
    case LBM_F32: return strip_t<LBM_F32>(c);
    case LBM_F32D: return strip_t<LBM_F32D>(c);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
