// lbm_strip.cuh -- two time steps of the two-buffer layout in one launch
// (FP32 arithmetic).
//
// What bounds the one-step kernel on large grids is HBM: it reads and writes
// every value once per step, at the copy bandwidth.  Two steps in one pass
// move half of that per step.  Each warp marches up a strip of 60 columns (a
// window of 64, one pair of nodes per lane): it updates row y to the first
// step from global memory, keeps it in a ring of three rows in shared memory,
// and updates row y - 1 to the second step from the ring.  The outer pair on
// either side of the window is only good for the first step; the strips of
// neighbouring warps overlap by it (64/60 of the arithmetic, no more DRAM
// traffic: the overlap is read from L2).  A warp needs nobody else's values, so
// there is no barrier in the kernel: lanes exchange the populations that cross
// columns by shuffles, and each lane reads back only the ring columns that it
// wrote.  The loads of row y + 1 are issued before row y is collided.
//
// Measured (4096^2, FP32 deviations): 290 -> 174 us per step, 96 G node
// updates/s, 5.8 TB/s of DRAM traffic; instruction issue and the latency of
// the collision with 12 warps per SM bound it now.
//
// Every node gets the arithmetic, and so the bits, of the one-step kernel: the
// nodes which that one updates one at a time in its wall tiles are rounded as
// single nodes here too (SingleLanes).
#pragma once

#include "lbm_device.cuh"

namespace lbm {

constexpr int kStripCols = 60;   // columns a warp brings to the second step

// One-warp blocks per SM.  Lagged tau: 12, at up to 168 registers (4096^2
// FP32 deviations 178 us per step when compared; 13, 14 and 16, whose fewer
// registers leave less room for the loads ahead, 211, 199 and 196).  The implicit tau waits
// for its special functions rather than for memory: 16, at up to 128 registers
// (4096^2 FP32 281 against 323 us).
template <int TAU>
constexpr int strip_blocks()
{
    return TAU == 1 ? 16 : 12;
}

// The strips, the row segments each is cut into, and the columns [0, lo) and
// [hi, nx) which the one-step kernel updates one node at a time; strips
// [0, first) and [end, nstrips) hold such columns or a side wall.
struct StripPlan {
    int nstrips, first, end, nseg, lo, hi;
    __host__ __device__ int units() const { return nstrips * nseg; }
    __host__ __device__ void cut(int ny, long long segments)
    {
        const int most = ny / 4 > 1 ? ny / 4 : 1;   // a segment also takes the first step of two rows beyond it
        nseg = segments < 1 ? 1 : (segments < most ? (int)segments : most);
    }
};
__host__ __device__ inline StripPlan strip_plan(int nx)
{
    StripPlan s;
    s.lo = 64;
    s.hi = (nx - 1) / 64 * 64;
    s.nstrips = (nx + kStripCols - 1) / kStripCols;
    // windows are [60 i - 2, 60 i + 62)
    s.first = (s.lo + 1) / kStripCols + 1;
    s.end = s.hi < 62 ? 0 : (s.hi - 62) / kStripCols + 1;
    if (s.end < s.first) s.end = s.first = s.nstrips;
    s.nseg = 1;
    return s;
}

// One value of a row of the ring or of a plane, as pairs (x, x + 1).
template <int PREC>
__device__ __forceinline__ F2 pair_at(const typename Store<PREC>::S *p, int64_t k, double rest)
{
    return Store<PREC>::ldd2(p, k, float(rest));
}

// Rows [ya, yb) of a strip brought to the second step by one warp.  SIDE: the
// window holds a side wall or single-rounded columns; ROWS: the rows the
// bottom or top wall.  Without them the loop has no wall rules at all; in no
// form is there a branch around its loads, which would make the compiler wait
// for them there.
template <int PREC, int FIELD, int TAU, bool SIDE, bool ROWS>
__device__ __forceinline__ void
strip_rows(const typename Store<PREC>::S *__restrict__ src, typename Store<PREC>::S *__restrict__ dst,
           const float *__restrict__ tsrc, float *__restrict__ tdst, const Phys<F2> &p, int strip, int ya, int yb,
           int lo, int hi, typename Store<PREC>::S (&ring)[3][14][64], float (&tring)[3][64])
{
    using St = Store<PREC>;
    using S = typename St::S;
    using Raw = typename St::Raw;
    const int lane = threadIdx.x;
    const int nx = p.nx, ny = p.ny;
    const int x = strip * kStripCols - 2 + 2 * lane;
    const bool out = lane > 0 && lane < 31 && x < nx;
    // lanes beyond the walls repeat the last pair inside (their values are not used)
    const int xc = x < 0 ? 0 : (x < nx ? x : (nx - 1) & ~1);
    const bool left = x == 0, right_x = x == nx - 1, right_y = x + 1 == nx - 1;
    const bool single = xc < lo || xc >= hi;
    const int64_t P = p.plane, W = p.pitch;

    // the stored pairs of row y's sources, before the shift along x; across the
    // top and bottom wall the populations that come back from the row itself
    Raw raw[14];
    F2 rawt, da;
    // what comes back to a side wall's node from its own diagonals
    S e0, e1;
    const int64_t own0 = left ? 7 * P : 8 * P + right_y, own1 = left ? 6 * P : 5 * P + right_y;
    auto load = [&](int y) {
        const int64_t k = (int64_t)y * W + xc;
        const S *k0 = src + k;
        auto get = [&](int q, int64_t off) { raw[q] = *reinterpret_cast<const Raw *>(k0 + off); };
        get(0, 0);
        get(1, P);
        get(3, 3 * P);
        get(9, 9 * P);
        get(10, 10 * P);
        get(12, 12 * P);
        const bool below = !ROWS || y > 0, above = !ROWS || y < ny - 1;
        get(2, below ? 2 * P - W : 4 * P);
        get(4, above ? 4 * P + W : 2 * P);
        get(5, below ? 5 * P - W : 7 * P);
        get(6, below ? 6 * P - W : 8 * P);
        get(7, above ? 7 * P + W : 5 * P);
        get(8, above ? 8 * P + W : 6 * P);
        get(11, below ? 11 * P - W : 13 * P);
        get(13, above ? 13 * P + W : 11 * P);
        if constexpr (TAU == 0) rawt = F2(*reinterpret_cast<const float2 *>(tsrc + k));
        if constexpr (FIELD == 1) da = load_da(p, k);
        if constexpr (SIDE) {   // every lane loads, the wall's lanes use it
            e0 = k0[own0];
            e1 = k0[own1];
        }
    };
    // the side walls' nodes: populations that come back from the node itself
    // (b1, b3 and c1, c3: its own f1, f3, g1, g3; h0, h1: its diagonals)
    auto side_walls = [&](F2 f[9], F2 g[5], F2 b1, F2 b3, F2 c1, F2 c3, float h0, float h1) {
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
    auto update_as = [&](F2 f[9], F2 g[5], F2 t, F2 d, auto z) {
        Macro<F2> m;
        if constexpr (FIELD == 1) {
            const Darcy<F2> k{d};
            return collide<F2, 1, 1>(p, f, g, tau_start<TAU, F2, 1, 1>(p, f, g, k, [&] { return t; }, z), m, k, z);
        } else {
            return collide<F2, 0, 1>(p, f, g, tau_start<TAU, F2, 0, 1>(p, f, g, (int64_t)0, [&] { return t; }, z), m,
                                     (int64_t)0, z);
        }
    };
    auto update = [&](F2 f[9], F2 g[5], F2 t, F2 d, int y) {
        if constexpr (SIDE || ROWS) {
            const bool one = single || (ROWS && (y == 0 || y == ny - 1));
            return update_as(f, g, t, d, SingleLanes{one, one});
        } else {
            return update_as(f, g, t, d, AsUsual{});
        }
    };

    const int y0 = ya > 0 ? ya - 1 : 0;
    const int last = yb < ny ? yb : ny - 1;   // last row brought to the first step
    load(y0);
    S *rc = &ring[0][0][2 * lane], *ra = &ring[1][0][2 * lane], *rb = &ring[2][0][2 * lane];
    float *tc = &tring[0][2 * lane], *ta = &tring[1][2 * lane], *tb = &tring[2][2 * lane];
    uint32_t rng = 0;
    F2 dprev;   // Darcy numbers of row y - 1
#pragma unroll 1
    for (int y = y0; y <= yb; y++) {   // at y = ny (the top segment) only the second step of row ny - 1
        F2 d;
        // one copy of the collision for both steps: two overflow the
        // instruction cache with the implicit tau
#pragma unroll 1
        for (int step = 0; step < 2; step++) {
            if (step == 0 ? ROWS && y > last : y <= ya) continue;
            const int Y = y - step;   // the row this step is taken on
            F2 f[9], g[5], t;
            if (step == 0) {
                auto r_f = [&](int i) { return St::of_raw(raw[i], float(rest_f(i))); };
                auto r_g = [&](int i) { return St::of_raw(raw[9 + i], float(rest_g(i))); };
                f[0] = r_f(0);
                f[1] = from_left(r_f(1), 0.f, lane);
                f[2] = r_f(2);
                f[3] = from_right(r_f(3), 0.f, lane);
                f[4] = r_f(4);
                f[5] = from_left(r_f(5), 0.f, lane);
                f[6] = from_right(r_f(6), 0.f, lane);
                f[7] = from_right(r_f(7), 0.f, lane);
                f[8] = from_left(r_f(8), 0.f, lane);
                g[0] = r_g(0);
                g[1] = from_left(r_g(1), 0.f, lane);
                g[2] = r_g(2);
                g[3] = from_right(r_g(3), 0.f, lane);
                g[4] = r_g(4);
                if (ROWS && y == 0) {
                    f[5] = r_f(5);
                    f[6] = r_f(6);
                }
                if (ROWS && y == ny - 1) {
                    f[7] = r_f(7);
                    f[8] = r_f(8);
                }
                    if (SIDE) {
                    float h0, h1;
                    h0 = St::ldd(&e0, 0, float(rest_f(5)));   // the diagonals' rest values are equal
                    h1 = St::ldd(&e1, 0, float(rest_f(5)));
                    side_walls(f, g, r_f(1), r_f(3), r_g(1), r_g(3), h0, h1);
                }
                t = rawt;
                d = da;
                if (y < last) load(y + 1);
            } else {
                const F2 a1 = pair_at<PREC>(ra, 64, rest_f(1)), a3 = pair_at<PREC>(ra, 3 * 64, rest_f(3));
                const F2 c1 = pair_at<PREC>(ra, 10 * 64, rest_g(1)), c3 = pair_at<PREC>(ra, 12 * 64, rest_g(3));
                f[0] = pair_at<PREC>(ra, 0, rest_f(0));
                f[1] = from_left(a1, 0.f, lane);
                f[3] = from_right(a3, 0.f, lane);
                g[0] = pair_at<PREC>(ra, 9 * 64, rest_g(0));
                g[1] = from_left(c1, 0.f, lane);
                g[3] = from_right(c3, 0.f, lane);
                if (!ROWS || Y > 0) {
                    f[2] = pair_at<PREC>(rb, 2 * 64, rest_f(2));
                    f[5] = from_left(pair_at<PREC>(rb, 5 * 64, rest_f(5)), 0.f, lane);
                    f[6] = from_right(pair_at<PREC>(rb, 6 * 64, rest_f(6)), 0.f, lane);
                    g[2] = pair_at<PREC>(rb, 11 * 64, rest_g(2));
                } else {
                    f[2] = pair_at<PREC>(ra, 4 * 64, rest_f(4));
                    f[5] = pair_at<PREC>(ra, 7 * 64, rest_f(7));
                    f[6] = pair_at<PREC>(ra, 8 * 64, rest_f(8));
                    g[2] = pair_at<PREC>(ra, 13 * 64, rest_g(4));
                }
                if (!ROWS || Y < ny - 1) {
                    f[4] = pair_at<PREC>(rc, 4 * 64, rest_f(4));
                    f[7] = from_right(pair_at<PREC>(rc, 7 * 64, rest_f(7)), 0.f, lane);
                    f[8] = from_left(pair_at<PREC>(rc, 8 * 64, rest_f(8)), 0.f, lane);
                    g[4] = pair_at<PREC>(rc, 13 * 64, rest_g(4));
                } else {
                    f[4] = pair_at<PREC>(ra, 2 * 64, rest_f(2));
                    f[7] = pair_at<PREC>(ra, 5 * 64, rest_f(5));
                    f[8] = pair_at<PREC>(ra, 6 * 64, rest_f(6));
                    g[4] = pair_at<PREC>(ra, 11 * 64, rest_g(2));
                }
                if (SIDE) {
                    const int j = right_y;
                    side_walls(f, g, a1, a3, c1, c3, St::ldd(ra, (left ? 7 : 8) * 64 + j, float(rest_f(8))),
                               St::ldd(ra, (left ? 6 : 5) * 64 + j, float(rest_f(5))));
                }
                if constexpr (TAU == 0) t = F2(*reinterpret_cast<const float2 *>(ta));
            }
            t = update(f, g, t, step == 0 ? d : dprev, Y);
            if (step == 0) {
#pragma unroll
                for (int i = 0; i < 9; i++) St::sdv2(rc, i * 64, f[i], float(rest_f(i)), rng);
#pragma unroll
                for (int i = 0; i < 5; i++) St::sdv2(rc, (9 + i) * 64, g[i], float(rest_g(i)), rng);
                if constexpr (TAU == 0) *reinterpret_cast<float2 *>(tc) = t.v;
            } else {
                if (out) {
                    const int64_t k = (int64_t)Y * W + x;
                    if (!SIDE || !right_x) {
#pragma unroll
                        for (int i = 0; i < 9; i++) St::sdv2(dst + i * P, k, f[i], float(rest_f(i)), rng);
#pragma unroll
                        for (int i = 0; i < 5; i++) St::sdv2(dst + (9 + i) * P, k, g[i], float(rest_g(i)), rng);
                        if constexpr (TAU == 0) *reinterpret_cast<float2 *>(tdst + k) = t.v;
                    } else {   // an odd row's last node
                        for (int i = 0; i < 9; i++) St::sdv(dst + i * P, k, f[i].v.x, float(rest_f(i)), rng);
                        for (int i = 0; i < 5; i++) St::sdv(dst + (9 + i) * P, k, g[i].v.x, float(rest_g(i)), rng);
                        if constexpr (TAU == 0) tdst[k] = t.v.x;
                    }
                }
            }
        }
        S *const r = rb;
        rb = ra;
        ra = rc;
        rc = r;
        float *const q = tb;
        tb = ta;
        ta = tc;
        tc = q;
        dprev = d;
    }
}

// Unit `unit` of a grid's plan, by one warp.
template <int PREC, int FIELD, int TAU>
__device__ __forceinline__ void
strip_unit(const typename Store<PREC>::S *__restrict__ src, typename Store<PREC>::S *__restrict__ dst,
           const float *__restrict__ tsrc, float *__restrict__ tdst, const Phys<F2> &p, const StripPlan &plan, int unit,
           typename Store<PREC>::S (&ring)[3][14][64], float (&tring)[3][64])
{
    const int strip = unit % plan.nstrips, seg = unit / plan.nstrips, ny = p.ny;
    // the first and last segments, which hold the bottom and top wall, get 5/8
    // of the others' rows: they take longer, and all units should end together
    const int total = 8 * plan.nseg - 6;
    const int ya = seg == 0 ? 0 : (int)((int64_t)ny * (8 * seg - 3) / total);
    const int yb = seg == plan.nseg - 1 ? ny : (int)((int64_t)ny * (8 * seg + 5) / total);
    const bool side = strip < plan.first || strip >= plan.end;
    if (ya == 0 || yb == ny)
        strip_rows<PREC, FIELD, TAU, true, true>(src, dst, tsrc, tdst, p, strip, ya, yb, plan.lo, plan.hi, ring, tring);
    else if (side)
        strip_rows<PREC, FIELD, TAU, true, false>(src, dst, tsrc, tdst, p, strip, ya, yb, plan.lo, plan.hi, ring, tring);
    else
        strip_rows<PREC, FIELD, TAU, false, false>(src, dst, tsrc, tdst, p, strip, ya, yb, plan.lo, plan.hi, ring, tring);
}

}  // namespace lbm
