// dugks_host.h -- host helpers shared by the context API (dugks_api.cu) and the
// batch API (dugks_batch.cu): face-stencil coefficients of the fast kernel, TMA
// tensor maps of the ghost-bordered plane layout, and ghosted uploads.
#pragma once

#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "../../include/dugks.h"
#include "dugks_internal.h"

namespace dugks {
namespace host {

// ---- face stencils of the fast path ------------------------------------------
// The face value bar f_k(x_b) is a fixed linear combination of bar f^+_k at the
// cells around the face: the Taylor expansion of Eq. (26) about the upwind cell
// (value + d.grad + d d : H / 2, + d d d : T / 6 at order 4), or the central form
// of Eq. (25). Below: the weights at offset (a, b) from the expansion cell of the
// stencils the generic kernel applies (orders 2 and 3: 9-point lattice moments;
// order 4: the 21-point gradient, the Richardson Hessian (4 H_1 - H_2) / 3 and
// second-order central third derivatives).
inline double G9x(int a, int b) {
    if (a < -1 || a > 1 || b < -1 || b > 1) return 0.0;
    return a * (b == 0 ? 1.0 / 3.0 : 1.0 / 12.0);
}
inline double G9y(int a, int b) { return G9x(b, a); }
inline double G21x(int a, int b) {   // weights 13/30, 2/15, -1/60 at (1, +-2), -1/60 at (2, 0), -1/30 at (2, +-1)
    const int aa = a < 0 ? -a : a, bb = b < 0 ? -b : b, s = a < 0 ? -1 : 1;
    if (aa == 0 || aa > 2 || bb > 2) return 0.0;
    if (aa == 1) return s * (bb == 0 ? 13.0 / 30.0 : bb == 1 ? 2.0 / 15.0 : -1.0 / 60.0);
    return s * (bb == 0 ? -1.0 / 60.0 : bb == 1 ? -1.0 / 30.0 : 0.0);
}
inline double G21y(int a, int b) { return G21x(b, a); }
// 9-point lattice-moment Hessian with spacing S (points at S times the 3 x 3 block)
inline double H9s(int i, int j, int a, int b, int S) {   // i, j in {0: x, 1: y}
    if (a % S != 0 || b % S != 0) return 0.0;
    a /= S;
    b /= S;
    if (a < -1 || a > 1 || b < -1 || b > 1) return 0.0;
    const double inv = 1.0 / (S * S);
    if (i != j) return (a != 0 && b != 0) ? 0.25 * a * b * inv : 0.0;
    const int along = i == 0 ? a : b, across = i == 0 ? b : a;
    if (along == 0 && across == 0) return -4.0 / 3.0 * inv;
    if (across == 0) return 2.0 / 3.0 * inv;
    if (along == 0) return -1.0 / 3.0 * inv;
    return 1.0 / 6.0 * inv;
}
inline double Hp(int order, int i, int j, int a, int b) {
    return order == 4 ? 4.0 / 3.0 * H9s(i, j, a, b, 1) - 1.0 / 3.0 * H9s(i, j, a, b, 2) : H9s(i, j, a, b, 1);
}
// third derivatives: txxx = (F(2,0) - F(-2,0)) / 2 - (F(1,0) - F(-1,0)); txxy = ((F(1,1) - F(1,-1))
// + (F(-1,1) - F(-1,-1))) / 2 - (F(0,1) - F(0,-1)); tyyy, txyy by symmetry
inline double Txxx(int a, int b) {
    if (b != 0) return 0.0;
    return a == 2 ? 0.5 : a == -2 ? -0.5 : a == 1 ? -1.0 : a == -1 ? 1.0 : 0.0;
}
inline double Txxy(int a, int b) {
    if ((a == 1 || a == -1) && (b == 1 || b == -1)) return 0.5 * b;
    if (a == 0 && (b == 1 || b == -1)) return -1.0 * b;
    return 0.0;
}
inline double taylor_w(int order, double dx, double dy, int a, int b) {
    double w = (a == 0 && b == 0) ? 1.0 : 0.0;
    if (order == 4) w += dx * G21x(a, b) + dy * G21y(a, b);
    else w += dx * G9x(a, b) + dy * G9y(a, b);
    if (order >= 3)
        w += 0.5 * dx * dx * Hp(order, 0, 0, a, b) + dx * dy * Hp(order, 0, 1, a, b) +
             0.5 * dy * dy * Hp(order, 1, 1, a, b);
    if (order == 4)
        w += (dx * dx * dx * Txxx(a, b) + 3.0 * dx * dx * dy * Txxy(a, b) + 3.0 * dx * dy * dy * Txxy(b, a) +
              dy * dy * dy * Txxx(b, a)) / 6.0;
    return w;
}

// Face-stencil tables for stencil radius R (1: orders 2-3, 2: orders 4 and 5).
template <typename T, int R>
inline FaceCoefs<T, R> make_face_coefs_r(int order, int flux, double h) {
    constexpr int NE = 2 * R + 1, NA = 2 * R + 2;
    double e[9][NE][NA] = {}, n[9][NA][NA] = {};
    auto gx = [&](int a, int b) { return order == 4 ? G21x(a, b) : G9x(a, b); };
    auto gy = [&](int a, int b) { return order == 4 ? G21y(a, b) : G9y(a, b); };
    for (int k = 0; k < 9; k++) {
        const int kx = ex(k), ky = ey(k);
        // east face: taps (b, a) -> e[k][b + R][a + R], b in -R..R, a in -R..R+1
        auto addE = [&](int cx, double wgt, double dx, double dy) {   // expansion about cell (cx, 0)
            for (int b = -R; b <= R; b++)
                for (int a = -R; a <= R; a++) e[k][b + R][cx + a + R] += wgt * taylor_w(order, dx, dy, a, b);
        };
        auto addN = [&](int cy, double wgt, double dx, double dy) {   // expansion about cell (0, cy)
            for (int b = -R; b <= R; b++)
                for (int a = -R; a <= R; a++) n[k][cy + b + R][a + R] += wgt * taylor_w(order, dx, dy, a, b);
        };
        if (order == 5) {
            // DUGKS-T2S5: the degree-4 tensor-product Lagrange interpolant on the 5 x 5
            // cells centred at the cell nearest to x_b - xi h (ties averaged); it needs
            // R = 2 (a radius-1 table is never built for order 5)
            if constexpr (R >= 2) {
            auto L5 = [](int a, double sd) {
                double w = 1.0;
                for (int b = -2; b <= 2; b++)
                    if (b != a) w *= (sd - b) / (double)(a - b);
                return w;
            };
            auto lagE = [&](int cx, double wgt, double sx, double sy) {   // centred at cell (cx, 0)
                for (int b = -2; b <= 2; b++)
                    for (int a = -2; a <= 2; a++) e[k][b + R][cx + a + R] += wgt * L5(a, sx) * L5(b, sy);
            };
            auto lagN = [&](int cy, double wgt, double sx, double sy) {   // centred at cell (0, cy)
                for (int b = -2; b <= 2; b++)
                    for (int a = -2; a <= 2; a++) n[k][cy + b + R][a + R] += wgt * L5(a, sx) * L5(b, sy);
            };
            if (kx > 0) lagE(0, 1.0, 0.5 - h, -ky * h);
            else if (kx < 0) lagE(1, 1.0, h - 0.5, -ky * h);
            else { lagE(0, 0.5, 0.5, -ky * h); lagE(1, 0.5, -0.5, -ky * h); }
            if (ky > 0) lagN(0, 1.0, -kx * h, 0.5 - h);
            else if (ky < 0) lagN(1, 1.0, -kx * h, h - 0.5);
            else { lagN(0, 0.5, -kx * h, 0.5); lagN(1, 0.5, -kx * h, -0.5); }
            }
        } else if (flux == DUGKS_UPWIND) {
            if (kx > 0) addE(0, 1.0, 0.5 - h, -ky * h);
            else if (kx < 0) addE(1, 1.0, h - 0.5, -ky * h);
            else { addE(0, 0.5, 0.5, -ky * h); addE(1, 0.5, -0.5, -ky * h); }
            if (ky > 0) addN(0, 1.0, -kx * h, 0.5 - h);
            else if (ky < 0) addN(1, 1.0, -kx * h, h - 0.5);
            else { addN(0, 0.5, -kx * h, 0.5); addN(1, 0.5, -kx * h, -0.5); }
        } else {
            // east: (F_c + F_E)/2 - h [xi_x (F_E - F_c) + xi_y (dF/dy(c) + dF/dy(E))/2]
            e[k][R][R] += 0.5 + h * kx;
            e[k][R][R + 1] += 0.5 - h * kx;
            n[k][R][R] += 0.5 + h * ky;
            n[k][R + 1][R] += 0.5 - h * ky;
            for (int b = -R; b <= R; b++)
                for (int a = -R; a <= R; a++) {
                    e[k][b + R][a + R] += -0.5 * h * ky * gy(a, b);
                    e[k][b + R][a + R + 1] += -0.5 * h * ky * gy(a, b);
                    n[k][b + R][a + R] += -0.5 * h * kx * gx(a, b);
                    n[k][b + R + 1][a + R] += -0.5 * h * kx * gx(a, b);
                }
        }
    }
    FaceCoefs<T, R> cf;
    for (int k = 0; k < 9; k++) {
        for (int b = 0; b < NE; b++)
            for (int a = 0; a < NA; a++) cf.e[k][b][a] = (T)e[k][b][a];
        for (int b = 0; b < NA; b++)
            for (int a = 0; a < NA; a++) cf.n[k][b][a] = (T)n[k][b][a];
    }
    return cf;
}

template <typename T>
inline FaceCoefs<T> make_face_coefs(int order, int flux, double h) {
    return make_face_coefs_r<T, 1>(order, flux, h);
}

// Expansion coefficients of the row march (orders 2 and 3; the fields are described at
// MarchCoefs). The terms of order 2 and above in the displacement are those of order 3.
template <typename T>
inline MarchCoefs<T> make_march_coefs(int order, double h) {
    MarchCoefs<T> m;
    const double c = 0.5 - h, q = order >= 3 ? 1.0 : 0.0;
    auto row = [&](double x, double y, int b, T *w) {   // C, R + L, R - L; FP64: C, L, R
        const double l = taylor_w(order, x, y, -1, b), r = taylor_w(order, x, y, 1, b);
        w[0] = (T)taylor_w(order, x, y, 0, b);
        w[1] = (T)(sizeof(T) == 8 ? l : 0.5 * (r + l));
        w[2] = (T)(sizeof(T) == 8 ? r : 0.5 * (r - l));
    };
    for (int b = -1; b <= 1; b++) {
        row(c, -h, b, m.dx[b + 1]);
        row(-h, c, b, m.dy[b + 1]);
    }
    m.px = (T)(c / 12.0);
    m.pe = (T)(q * c * c / 12.0);
    m.nu = (T)((0.5 * c + q * 0.5 * c * c) / 6.0);
    m.nd = (T)((-0.5 * c + q * 0.5 * c * c) / 6.0);
    m.nm = (T)(-q * c * c / 6.0);
    m.ge = (T)(q / 96.0);
    m.gp = (T)(q * h * h / 24.0);
    m.gd = (T)(h / 24.0);
    m.b2 = (T)(q * h / 16.0);
    m.h = (T)h;
    m.cu = (T)(0.5 + h);
    m.cd = (T)(0.5 - h);
    m.hk = (T)(h / 24.0);
    return m;
}

// Lane width (columns a lane), segment rows and launch mode of the row march.
// A segment of s rows reads s + 4 (the DVM s + 6), so long segments do less work, and short ones give
// more warps. The costs below are fits to measured steps: FP32 and FP16 storage, 69 sizes from 48^2 to 4096^2
// and 64 x 256 to 3000 x 300, rows from 1 to 64, both widths, dugks_step(n) and step-and-mass loops. In one wave
// of warps a row takes longer with every warp that an SM holds, in several waves it takes `unit` and part of
// a wave is lost at the end. The plan that the costs choose against the best one measured, mean and largest: two-stage
// upwind 1.008 and 1.07, central 1.006 and 1.07, three-stage 1.006 and 1.10, central 1.002 and 1.04, DVM 1.016
// and 1.11, below dt = 1/2 1.013 and 1.11, LBM 1.025 and 1.24. (One set of constants for all DUGKS steps
// and one for all DVM steps had given 1.010 and 1.17, 1.022 and 1.37, 1.031 and 1.36, 1.036 and 1.54, 1.045 and 1.24, 1.043
// and 1.21, 1.125 and 1.27: central 548^2, 5 rows of pairs 15.4 us, 7 of single columns 14.1; DVM 128^2 7.3 -> 5.0,
// 256^2 8.6 -> 7.2; LBM 1024^2 23.1 -> 18.8; three-stage 850^2 72.3 -> 63.9.)
// Segments over 64 rows lose again (4096^2, 241 rows in one wave: 478 us): the rows in flight then
// lie all over the planes, more pages than the TLB holds.
// FP64: the FP64 unit of each scheduler issues a warp instruction in 64 cycles whatever the
// number of active lanes, so a step costs the rows of the busiest scheduler: the warps it gets
// times s + 2.5 rows (the rows at a segment's ends leave out what they do not need).
struct MarchPlan {
    int cols, rows, early, one_wave;
    double cost;   // of a step, as the rule sees it (FP64: in rows of a warp alone on its scheduler, 12.4 us)
    int mode() const { return (early ? MARCH_EARLY : 0) | (one_wave ? MARCH_ONE_WAVE : 0); }
};
// strips of a grid for lanes of `cols` columns, their width, segments of about `want` rows and
// their equal length
inline int march_strips(int cols, int nx) {
    return cols == 2 ? MarchTile<float2, float>::strips(nx) : MarchTile<float, float>::strips(nx);
}
inline int march_width(int cols, int nx) {   // (single columns: spread over the strips)
    const int n = march_strips(cols, nx);
    return cols == 2 ? MarchTile<float2, float>::TX : (nx + n - 1) / n;
}
inline int march_segments(int want, int ny) { return (ny + want - 1) / want; }
inline int march_segment_rows(int want, int ny) {
    const int n = march_segments(want, ny);
    return (ny + n - 1) / n;
}
// What the rule needs of a kernel with lanes of one width: resident warps an SM; in one wave, us a launch, more where
// the next kernel is not scheduled early, and a row's us: `row` and `more` for each warp of the fullest SM (counted in
// steps of `step`), of a segment's rows and `extra1`; in several waves, us a row of a full wave, rows that a segment
// costs past its own and the largest part of a wave that is lost; the part of a wave from which the next kernel
// is scheduled early, and the longest segments for which it is. The costs of a three-stage step are those of its two kernels.
struct MarchLanes {
    double slots, launch, late, row, more;
    int step;
    double extra1, unit, extra2, tail, early;
    int early_rows;
};
// For single columns and pairs; the part of a wave below which the next kernel is scheduled early too, and the rows that a
// segment costs past its own in FP64.
// Early scheduling of the next kernel hides its launch and velocity factors (512^2: 15.5 against 16.5 us). On a
// chip half full it costs instead, because the waiting warps fill some SMs and leave others idle (256^2, 860
// warps: 10.2 against 9.1), in long segments of pairs in the three-stage scheme (7 rows, 900 x 500 45.1 against 47.7;
// 9 rows, 768^2 59.3 against 51.1; 12 rows that fill the wave, central 900^2, 70.4 against 66), for the LBM within a wave (512^2, single columns of 6 rows, 11 against
// 9.4), and in FP64, where a scheduler with two warps takes twice as long.
struct MarchShape {
    int (*strips)(int cols, int nx);
    MarchLanes lanes[2];
    double few, extra64;
};
inline const MarchShape &march_shape(int stages, int flux) {
    static const MarchShape s[4] = {
        {march_strips,
         {{12, 4.9, 0.9, 0.62, 0.075, 4, 0, 1.12, 3.5, 0.7, 0.667, 64},
          {8, 5.7, 0.9, 0.98, 0.1175, 4, 0, 1.36, 3.5, 0.7, 0.52, 64}},
         0.15, 2.5},
        {march_strips,
         {{12, 4.08, 0, 0.81, 0.06, 1, 1.33, 1.02, 4.39, 0.67, 0.667, 64},
          {8, 0, 0, 1.49, 0.04, 1, 4.55, 1.36, 3.5, 0.7, 0.52, 64}},
         0.15, 2.5},
        {march_strips,
         {{12, 6.2, 0, 1.95, 0.13, 1, 0.57, 4.17, 3.44, 0.47, 0.667, 64},
          {8, 1.6, 0, 4.09, 0.06, 1, 1.75, 3.03, 6.04, 1.07, 0.52, 7}},
         0.15, 2.5},
        {march_strips,
         {{12, 8.06, 0, 1.57, 0.16, 1, 0.96, 2.73, 3.09, 0.59, 0.667, 64},
          {8, 0, 0, 3.25, 0.13, 1, 3.97, 3.14, 4.59, 0.64, 0.52, 7}},
         0.15, 2.5}};
    return s[(stages == 3 ? 2 : 0) + (flux == 1 ? 1 : 0)];
}
// the DVM: displacements below half a cell, from there up, and of one cell (the LBM)
inline const MarchShape &dvm_shape(double dt) {
    static const MarchShape s[3] = {
        {dvm_march_strips,
         {{16, 0.04, 0.42, 0.86, 0.04, 1, 2.99, 1.42, 4.91, 0.71, 1.0, 64},
          {12, 0.06, 1.04, 1.05, 0.04, 1, 2.73, 1.13, 2.54, 1.06, 0.667, 64}},
         0.1, 6.0},
        {dvm_march_strips,
         {{16, 0.67, 0.01, 0.79, 0.05, 1, 3.05, 1.31, 4.78, 0.65, 0.76, 64},
          {12, 0, 0.07, 1.18, 0.06, 1, 3.1, 1.43, 3.05, 0.72, 0.667, 64}},
         0.1, 6.0},
        {dvm_march_strips,
         {{16, 0.06, 0.14, 0.71, 0.03, 1, 4.25, 1.57, 2.75, 0.52, 1.3, 64},
          {12, 1.14, 0.39, 1.02, 0.07, 1, 1.99, 1.28, 2.44, 0.49, 1.05, 64}},
         0.15, 6.0}};
    return s[dt == 1.0 ? 2 : dt >= 0.5 ? 1 : 0];
}
// Strip segments that a set of grids gives, for every lane width (index: columns - 1) and segment length.
// Kept from one plan to the next where grids come and go one at a time.
constexpr int MARCH_ROWS = 64;
struct MarchWork {
    int64_t n[2][MARCH_ROWS + 1] = {};
    void count(const MarchShape &sh, int2 size, int sign) {
        const int64_t a = (int64_t)sign * sh.strips(1, size.x), b = (int64_t)sign * sh.strips(2, size.x);
        for (int want = 1; want <= MARCH_ROWS; want++) {
            const int64_t s = march_segments(want, size.y);
            n[0][want] += a * s;
            n[1][want] += b * s;
        }
    }
};
// For `count` grids of sizes (x, y) stepped together, whose segments are `work`. (A length that no grid's equal
// segments reach, because the longest of them has r < `want` rows, costs as much as r, which is met
// first: each grid has as many segments at r. So `want` stands for the rows of the longest, and a
// plan takes no pass over the grids, which cost 0.22 ms of the step call after each admission to 512 of them:
// 272 -> 34 us on the host, of 64 48 -> 19.)
inline MarchPlan march_plan(const MarchShape &sh, int variant, const MarchWork &work, const int2 *sizes, int count,
                            int precision, int sms) {
    static constexpr int fixed[6] = {16, 8, 0, 32, 0, 64};   // variants 2 and 4: by the rule
    MarchPlan m{precision == DUGKS_FP64 ? 1 : 2, 16, 0, 0, 0.0};
    double best = 1e300;
    const int forced = variant >= 0 && variant < 6 ? fixed[variant] : 0;
    const bool f64 = precision == DUGKS_FP64;
    int longest = 1;
    for (int i = 0; i < (forced ? count : 0); i++) longest = std::max(longest, march_segment_rows(forced, sizes[i].y));
    for (int cols = 1; cols <= (f64 ? 1 : 2); cols++) {
        const int c = cols - 1;
        const MarchLanes &q = sh.lanes[c];
        for (int want = forced ? forced : 1; want <= (forced ? forced : MARCH_ROWS); want++) {
            const double w = (double)work.n[c][want];
            const int rows = forced ? longest : want;
            const double W = w / (q.slots * sms), n = w / (4.0 * sms);
            const bool early = !f64 && (rows <= q.early_rows || (W > 0.965 && W <= 1.0)) && (W > q.early || W < sh.few);
            double cost;
            if (f64)
                cost = (n > 3.0 ? n + 0.5 : std::ceil(n)) * (rows + sh.extra64);
            else if (W <= 1.0)
                cost = q.launch + (early && !(rows == 1 && W > 0.9) ? 0.0 : q.late) +   // (no room for the next kernel's warps)
                       (rows + q.extra1) * (q.row + q.more * q.step * std::ceil(w / (q.step * (double)sms)));
            else
                cost = q.unit * (rows + q.extra2) * (W + std::min(q.tail, 1.4 / W));
            if (cost < best) {
                best = cost;
                // (FP64 warps on every scheduler of an SM: a row takes a tenth longer)
                m = MarchPlan{cols, want, early, W <= 1.0, f64 && n > 0.8 && n <= 1.0 ? 1.1 * cost : cost};
            }
        }
    }
    return m;
}

inline MarchPlan march_plan(const MarchShape &sh, int variant, int2 size, int precision, int sms) {
    MarchWork work;
    work.count(sh, size, 1);
    return march_plan(sh, variant, work, &size, 1, precision, sms);
}

// Whether the FP64 two-stage step of an nx * ny grid takes the tile kernel (tiles of w * h cells, one
// CTA an SM) and not the march. Both are bound by the FP64 unit and come in steps: the march by the
// rows of the busiest scheduler, the tiles in waves of 71 us, 5.75 rows. Measured (vortex, us, tile
// against march): 192^2 76.7 / 75.9, 198^2 77.0 / 81.0, 246^2 76.6 / 97.3, 252^2 143 / 97, 320^2 146 / 136,
// 360^2 146.6 / 150.3, 380^2 220 / 163. From three waves on the march was faster at every size.
inline bool tile64_pays(const MarchPlan &m, int nx, int ny, int w, int h, int sms) {
    const long long tiles = (long long)((nx + w - 1) / w) * ((ny + h - 1) / h), waves = (tiles + sms - 1) / sms;
    return waves <= 2 && 5.75 * (double)waves < m.cost;
}

// The expansions of the DVM's streaming (Eq. (12)) at the displacement d xi_k: rows of the
// stencil of xi = (1, 1) at (d, d) as weights of the row's sum, of R - 2 C + L and of R - L; px, pe as
// above with c = d; nu, nm: weights of the first and second difference over rows of L + 4 C + R.
template <typename T>
inline MarchCoefs<T> make_dvm_coefs(int order, double d) {
    MarchCoefs<T> m{};
    const double q = order >= 3 ? 1.0 : 0.0;
    for (int b = -1; b <= 1; b++) {
        const double l = taylor_w(order, d, d, -1, b), r = taylor_w(order, d, d, 1, b);
        m.dx[b + 1][0] = (T)(taylor_w(order, d, d, 0, b) + l + r);
        m.dx[b + 1][1] = (T)(0.5 * (r + l));
        m.dx[b + 1][2] = (T)(0.5 * (r - l));
    }
    m.px = (T)(d / 12.0);
    m.pe = (T)(q * d * d / 12.0);
    m.nu = (T)(d / 12.0);
    m.nm = (T)(q * d * d / 12.0);
    return m;
}

// ---- TMA tensor maps -----------------------------------------------------------
inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess && q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
        else
            cudaGetLastError();
    });
    return fn;
}

inline CUtensorMapDataType tma_type(size_t es, bool half) {
    if (half) return CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    return es == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
}

// planes of `es`-byte elements at base: dims (pitch, ny + 2 GHOST[, nplanes]),
// box (bw, bh[, nplanes]); the fill of out-of-range elements is zero
inline bool encode_plane_map(CUtensorMap *m, void *base, size_t es, bool half, int pitch, int ny, size_t plane,
                             int nplanes, int bw, int bh) {
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)pitch, (cuuint64_t)(ny + 2 * GHOST), (cuuint64_t)nplanes};
    const cuuint64_t strides[2] = {(cuuint64_t)pitch * es, (cuuint64_t)plane * es};
    const cuuint32_t box[3] = {(cuuint32_t)bw, (cuuint32_t)bh, (cuuint32_t)nplanes};
    const cuuint32_t estr[3] = {1, 1, 1};
    const cuuint32_t rank = nplanes > 1 ? 3 : 2;
    CUresult r = fn(m, tma_type(es, half), rank, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

// host doubles (ny * nx, x fastest) -> device plane (double or float) with the
// periodic ghost border; synchronous
// A ny * nx field written into a ghost-bordered plane of (ny + 2 GHOST) rows of
// `pitch` elements of type O: the border holds the periodic images, the padding
// past nx + 2 GHOST is zero.
template <typename O>
inline void fill_ghosted_plane(O *pad, const double *src, int nx, int ny, int pitch) {
    const int G = GHOST;
    for (int y = -G; y < ny + G; y++) {
        const int sy = ((y % ny) + ny) % ny;
        const double *row = src + (size_t)sy * nx;
        O *out = pad + (size_t)(y + G) * pitch;
        for (int x = -G; x < 0; x++) out[x + G] = (O)row[((x % nx) + nx) % nx];
        for (int x = 0; x < nx; x++) out[x + G] = (O)row[x];
        for (int x = nx; x < nx + G; x++) out[x + G] = (O)row[x % nx];
        for (int x = nx + 2 * G; x < pitch; x++) out[x] = O(0);
    }
}

inline cudaError_t upload_ghosted_plane(void *dst, const double *src, int nx, int ny, int pitch, bool fp64) {
    const size_t n = (size_t)(ny + 2 * GHOST) * pitch;
    if (fp64) {
        std::vector<double> pad(n);
        fill_ghosted_plane(pad.data(), src, nx, ny, pitch);
        return cudaMemcpy(dst, pad.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    }
    std::vector<float> f(n);
    fill_ghosted_plane(f.data(), src, nx, ny, pitch);
    return cudaMemcpy(dst, f.data(), n * sizeof(float), cudaMemcpyHostToDevice);
}

}  // namespace host
}  // namespace dugks
