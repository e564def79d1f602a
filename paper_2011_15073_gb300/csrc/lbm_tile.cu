// lbm_tile.cu -- two or four time steps of the two-buffer layout in one launch
// for small grids (FP32 arithmetic).
//
// What bounds the one-step kernel there is latency: a step of a 256^2 grid is
// one wave of warps that wait once for their loads, run one chain of dependent
// instructions and store, plus the launch (2.4 us a step from a replayed
// graph, of which the SMs compute a quarter).  Here a block keeps a window of
// 64 columns x kTileRows rows on the SM and takes several steps on it: each warp
// holds one row, a pair of nodes per lane, in registers; populations that stay in
// the row cross columns by shuffles, those that leave it go through shared
// memory, one barrier per step.  Neighbouring windows overlap: the first step
// reads its sources from global memory, after each further step one more row
// (and column) on every side of the window is out of date, so that 16 - 2 (T - 1)
// rows and 64 - 2 T columns of it are brought to step T.
//
// Measured (us per step, replayed graphs, one step per launch / this): FP32
// deviations 64^2 1.90 / 1.70, 128^2 1.93 / 1.74, 256^2 2.54 / 1.83, 300^2 (two
// steps) 3.1 / 2.7; 256^2 with the implicit tau 3.85 / 2.85.  A launch of four
// steps takes 3 us plus 0.96 a step; that is instruction issue, 16 warps'
// collisions on each SM.
//
// Every node gets the arithmetic, and so the bits, of the one-step kernel
// (SingleLanes: its wall tiles' nodes).
#include "lbm_device.cuh"
#include "lbm_internal.h"

namespace lbm {

namespace {

constexpr int kTileRows = 16;   // rows, and warps, of a window

// A deviation as it comes back from storage.
template <int PREC>
__device__ __forceinline__ F2 stored(F2 d, double rest)
{
    if constexpr (PREC == LBM_F32)
        return Store<PREC>::of_raw((d + F2(float(rest))).v, float(rest));
    else
        return d;
}

template <int PREC, int FIELD, int TAU>
__global__ void __launch_bounds__(32 * kTileRows, 1)
tile_kernel(const typename Store<PREC>::S *__restrict__ src, typename Store<PREC>::S *__restrict__ dst,
            const float *__restrict__ tsrc, float *__restrict__ tdst, Phys<F2> p, int steps, int lo, int hi)
{
    using St = Store<PREC>;
    using S = typename St::S;
    // the populations that leave a row, of the step before: [parity][row]
    // up: f2, f5, f6, g2 (for the row above), down: f4, f7, f8, g4 (below)
    extern __shared__ float2 exchange[];
    using Rows = float2[kTileRows][4][32];
    Rows *up = reinterpret_cast<Rows *>(exchange), *down = up + 2;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int nx = p.nx, ny = p.ny;
    const int xw = blockIdx.x * (64 - 2 * steps) - steps;
    const int x = xw + 2 * lane, y = (int)blockIdx.y * (kTileRows - 2 * (steps - 1)) - (steps - 1) + row;
    const bool inside = y >= 0 && y < ny, below = y > 0, above = y < ny - 1;
    // lanes beyond the walls repeat the nearest pair inside (their values are not used)
    const int xc = x < 0 ? 0 : (x < nx ? x : (nx - 1) & ~1);
    const bool left = x == 0, right_x = x == nx - 1, right_y = x + 1 == nx - 1;
    const bool one = xc < lo || xc >= hi || !below || !above;
    const SingleLanes z{one, one};
    const int64_t P = p.plane, W = p.pitch, k = (int64_t)y * W + xc;

    F2 f[9], g[5], t, da;
    // own diagonals that come back to a side wall's node
    float h0 = 0.f, h1 = 0.f;
    // the pairs' sources before the shift along x -> f, g
    auto arrive = [&](F2 b1, F2 b3, F2 c1, F2 c3) {
        f[1] = from_left(b1, 0.f, lane);
        f[3] = from_right(b3, 0.f, lane);
        g[1] = from_left(c1, 0.f, lane);
        g[3] = from_right(c3, 0.f, lane);
        const F2 l5 = from_left(f[5], 0.f, lane), r6 = from_right(f[6], 0.f, lane);
        const F2 r7 = from_right(f[7], 0.f, lane), l8 = from_left(f[8], 0.f, lane);
        if (below) {
            f[5] = l5;
            f[6] = r6;
        }
        if (above) {
            f[7] = r7;
            f[8] = l8;
        }
        if (left) {
            f[1].v.x = b3.v.x;
            f[5].v.x = h0;
            f[8].v.x = h1;
            g[1].v.x = p.abbd_hot.v.x - c3.v.x;
        }
        if (right_x) {
            f[3].v.x = b1.v.x;
            f[6].v.x = h0;
            f[7].v.x = h1;
            g[3].v.x = p.abbd_cold.v.x - c1.v.x;
        }
        if (right_y) {
            f[3].v.y = b1.v.y;
            f[6].v.y = h0;
            f[7].v.y = h1;
            g[3].v.y = p.abbd_cold.v.x - c1.v.y;
        }
    };
#pragma unroll 1
    for (int s = 0; s < steps; s++) {
        // rows that the window's last step still depends on
        const bool work = inside && row >= s && row < kTileRows - s;
        if (work) {
            if (s == 0) {
                const S *k0 = src + k;
                auto at_f = [&](int i, int64_t off) { return St::ldd2(k0 + off, 0, float(rest_f(i))); };
                auto at_g = [&](int i, int64_t off) { return St::ldd2(k0 + off, 0, float(rest_g(i))); };
                if constexpr (TAU == 0) t = F2(*reinterpret_cast<const float2 *>(tsrc + k));
                if constexpr (FIELD == 1) da = load_da(p, k);
                f[0] = at_f(0, 0);
                f[2] = at_f(2, below ? 2 * P - W : 4 * P);
                f[4] = at_f(4, above ? 4 * P + W : 2 * P);
                f[5] = at_f(5, below ? 5 * P - W : 7 * P);
                f[6] = at_f(6, below ? 6 * P - W : 8 * P);
                f[7] = at_f(7, above ? 7 * P + W : 5 * P);
                f[8] = at_f(8, above ? 8 * P + W : 6 * P);
                g[0] = at_g(0, 9 * P);
                g[2] = at_g(2, below ? 11 * P - W : 13 * P);
                g[4] = at_g(4, above ? 13 * P + W : 11 * P);
                if (left) {
                    h0 = St::ldd(k0 + 7 * P, 0, float(rest_f(7)));
                    h1 = St::ldd(k0 + 6 * P, 0, float(rest_f(6)));
                }
                if (right_x || right_y) {
                    h0 = St::ldd(k0 + 8 * P, right_y, float(rest_f(8)));
                    h1 = St::ldd(k0 + 5 * P, right_y, float(rest_f(5)));
                }
                arrive(at_f(1, P), at_f(3, 3 * P), at_g(1, 10 * P), at_g(3, 12 * P));
            } else {
                // own diagonals, then what the rows below and above sent (a
                // row outside the window is never needed: work)
                h0 = left ? f[7].v.x : (right_y ? f[8].v.y : f[8].v.x);
                h1 = left ? f[6].v.x : (right_y ? f[5].v.y : f[5].v.x);
                const F2 o2 = f[2], o5 = f[5], o6 = f[6], o4 = f[4], o7 = f[7], o8 = f[8], q2 = g[2], q4 = g[4];
                const int b = (s - 1) & 1;
                if (below) {
                    f[2] = F2(up[b][row - 1][0][lane]);
                    f[5] = F2(up[b][row - 1][1][lane]);
                    f[6] = F2(up[b][row - 1][2][lane]);
                    g[2] = F2(up[b][row - 1][3][lane]);
                } else {
                    f[2] = o4;
                    f[5] = o7;
                    f[6] = o8;
                    g[2] = q4;
                }
                if (above) {
                    f[4] = F2(down[b][row + 1][0][lane]);
                    f[7] = F2(down[b][row + 1][1][lane]);
                    f[8] = F2(down[b][row + 1][2][lane]);
                    g[4] = F2(down[b][row + 1][3][lane]);
                } else {
                    f[4] = o2;
                    f[7] = o5;
                    f[8] = o6;
                    g[4] = q2;
                }
                arrive(f[1], f[3], g[1], g[3]);
            }
            Macro<F2> m;
            if constexpr (FIELD == 1) {
                const Darcy<F2> d{da};
                t = collide<F2, 1, 1>(p, f, g, tau_start<TAU, F2, 1, 1>(p, f, g, d, [&] { return t; }, z), m, d, z);
            } else {
                t = collide<F2, 0, 1>(p, f, g, tau_start<TAU, F2, 0, 1>(p, f, g, (int64_t)0, [&] { return t; }, z), m,
                                      (int64_t)0, z);
            }
            if (s < steps - 1) {
#pragma unroll
                for (int i = 0; i < 9; i++) f[i] = stored<PREC>(f[i], rest_f(i));
#pragma unroll
                for (int i = 0; i < 5; i++) g[i] = stored<PREC>(g[i], rest_g(i));
                const int b = s & 1;
                up[b][row][0][lane] = f[2].v;
                up[b][row][1][lane] = f[5].v;
                up[b][row][2][lane] = f[6].v;
                up[b][row][3][lane] = g[2].v;
                down[b][row][0][lane] = f[4].v;
                down[b][row][1][lane] = f[7].v;
                down[b][row][2][lane] = f[8].v;
                down[b][row][3][lane] = g[4].v;
            }
        }
        if (s < steps - 1) __syncthreads();
    }
    const bool out = inside && row >= steps - 1 && row <= kTileRows - steps && 2 * lane >= steps && 2 * lane < 64 - steps && x < nx;
    if (!out) return;
    uint32_t rng = 0;
    if (!right_x) {
#pragma unroll
        for (int i = 0; i < 9; i++) St::sdv2(dst + i * P, k, f[i], float(rest_f(i)), rng);
#pragma unroll
        for (int i = 0; i < 5; i++) St::sdv2(dst + (9 + i) * P, k, g[i], float(rest_g(i)), rng);
        if constexpr (TAU == 0) *reinterpret_cast<float2 *>(tdst + k) = t.v;
    } else {   // an odd row's last node
#pragma unroll
        for (int i = 0; i < 9; i++) St::sdv(dst + i * P, k, f[i].v.x, float(rest_f(i)), rng);
#pragma unroll
        for (int i = 0; i < 5; i++) St::sdv(dst + (9 + i) * P, k, g[i].v.x, float(rest_g(i)), rng);
        if constexpr (TAU == 0) tdst[k] = t.v.x;
    }
}

dim3 tile_grid(int nx, int ny, int steps)
{
    const int cols = 64 - 2 * steps, rows = kTileRows - 2 * (steps - 1);
    return dim3((nx + cols - 1) / cols, (ny + rows - 1) / rows);
}

template <int PREC, int TAU>
cudaError_t tile_tau(lbm_ctx *c, int steps)
{
    using S = typename Store<PREC>::S;
    const int s = c->cur, d = 1 - s;
    const dim3 grid = tile_grid(c->nx, c->ny, steps);
    auto *kern = c->d_da ? tile_kernel<PREC, 1, TAU> : tile_kernel<PREC, 0, TAU>;
    const int smem = 4 * kTileRows * 4 * 32 * (int)sizeof(float2);
    if (const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) return e;
    kern<<<grid, 32 * kTileRows, smem, c->stream>>>((const S *)c->buf.dist[s], (S *)c->buf.dist[d],
                                                    (const float *)c->buf.tau[s], (float *)c->buf.tau[d],
                                                    make_params<F2>(c), steps, 64, (c->nx - 1) / 64 * 64);
    c->cur = d;
    return cudaGetLastError();
}
template <int PREC>
cudaError_t tile_t(lbm_ctx *c, int steps)
{
    return c->opts.tau_iters > 0 ? tile_tau<PREC, 1>(c, steps) : tile_tau<PREC, 0>(c, steps);
}

}  // namespace

// As many steps as leave one block on each of the `sms` SMs: a second wave of blocks costs more
// than the launches saved (384^2: 3.4 us a step in two waves of four steps, 3.7
// one by one; 512^2: 6.4 and 4.9).
int tile_steps(int nx, int ny, const lbm_opts &o, int sms)
{
    if (o.layout != 0 || o.staging != 0 || nx < 64) return 0;
    if (o.prec != LBM_F32 && o.prec != LBM_F32D) return 0;
    for (int steps : {4, 2}) {
        const dim3 g = tile_grid(nx, ny, steps);
        if ((int64_t)g.x * g.y <= sms) return steps;
    }
    return 0;
}

cudaError_t launch_tile(lbm_ctx *c, int steps)
{
    switch (c->opts.prec) {
    case LBM_F32: return tile_t<LBM_F32>(c, steps);
    case LBM_F32D: return tile_t<LBM_F32D>(c, steps);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbm
