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

// Up to about 700,000 nodes both buffers stay in L2, and the strips have few rows
// per warp: a segment of four rows takes six rows' first steps, one after the
// other.  The one-step kernel's work goes with the rows' tiles of 64 columns, the
// strips' with their 60, so the line is drawn on the nodes in tiles times the
// ratio of the two.  Measured on the FP32 deviations, lagged tau, one step per
// launch / two (us per step, from replayed graphs as lbm_step launches up to
// 2,000,000 nodes; in brackets that count, in thousands): 256 x 2600 [568] 9.0 / 10.6,
// 1024 x 640 [621] 9.0 / 9.7, 900 x 640 [655] 8.3 / 8.5, 780 x 760 [674] 8.7 / 8.5,
// 1024 x 700 [680] 9.7 / 9.7, 900 x 700 [717] 9.0 / 8.6, 840^2 [803] 10.2 / 9.4,
// 160 x 4096 [839] 10.8 / 9.9, 900^2 [922] 14.3 / 10.7; 1024^2 18.8 / 13.7, 2048^2
// 77 / 46, 4096^2 290 / 174.  From 657 to 700 the two are within 6 % either way, with
// a Darcy field (read once for two steps) the strips up to 9 % ahead (800^2 [659]
// 10.0 / 9.5, 780 x 760 9.5 / 8.7).
// Implicit tau, by the nodes themselves: 2048^2 86 / 74.
// The 16-bit storages are bound by instruction issue, not by HBM, and keep
// their four-node kernel.
bool two_steps(int nx, int ny, const lbm_opts &o)
{
    if (o.layout != 0 || o.staging != 0 || nx < 128 || ny < 64) return false;
    if (o.prec != LBM_F32 && o.prec != LBM_F32D) return false;
    if (o.tau_iters > 0) return (int64_t)nx * ny >= 2000000;
    const int64_t tiles = (nx + 63) / 64 * 64, strips = (int64_t)strip_plan(nx).nstrips * kStripCols;
    return tiles * ny >= 657000 * strips / tiles;
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
