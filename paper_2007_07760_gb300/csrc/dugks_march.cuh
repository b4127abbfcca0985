// dugks_march.cuh -- the DUGKS step for stencils of radius 1 (orders 2 and 3) as a
// row march (sm_103a): the two-stage step and the two kernels of the three-stage step.
//
// Same method as step_kernel (dugks_kernels.cuh; equation numbers are the paper's).
// One warp, which is one CTA, owns a strip of 60 columns (28 with one column a lane, as in FP64 and
// on small grids) and a segment of rows and walks up the rows with everything the step needs of
// the rows below in registers:
//  * a lane holds two adjacent columns, and all arithmetic is on that pair (packed
//    FP32: one instruction, two columns). The left and right neighbours of a pair
//    are one shuffle each for two cells; no shared-memory exchange and no barrier.
//  * the face values of Eqs. (24)-(26) are evaluated as expansions about each cell:
//    cell c gives its own contribution to its east, west, north and south faces, so
//    a face needs the 3 x 3 cells around one cell instead of 3 x 4 around a face.
//    An expansion is a sum over the three rows of row terms, so when row j arrives
//    it completes the expansions of row j - 1, adds the middle terms of row j and
//    starts row j + 1: each row of bar f^+ is formed and shuffled once.
//  * the directions normal to a face (the ties of Eq. (26)) enter only the face
//    moment phi_b, never the difference of a single bar f_k; their sums over the
//    three directions are taken before the stencil.
//  * rows arrive through a ring of per-lane cp.async copies two rows ahead.
// What bounds it: the issue of FP32 instructions on large grids (4096^2: 673 for a row of a warp, 399
// thread instructions a cell, against 876 in tiles), a row's latency in launches of one wave, and in FP64 that unit,
// one warp instruction in 64 cycles a scheduler. Rows of a segment are read and expanded with two extra rows
// on each side, so the segment length trades that overhead against the number of warps in flight
// (march_plan in dugks_host.h has the rule).
// Measured, us a step, shared-memory tiles -> march: FP32 256^2 9.4 -> 7.5, 512^2 14.8 -> 12.8, 1024^2 44.0 -> 35.1,
// 4096^2 617 -> 331; FP16 storage 1024^2 52.6 -> 38.6, 4096^2 738 -> 370; three-stage 512^2 33.4 -> 28.9, 1024^2
// 108.9 -> 87.5, 4096^2 1352 -> 885; FP64 (a step a call) 64^2 77 -> 47, 512^2 312 -> 256.
#pragma once

#include <type_traits>

#include "dugks_fast.cuh"

namespace dugks {

// Expansion coefficients of one reconstruction time h (host: make_march_coefs).
// Upwind, with c = 1/2 - h:
//   dx[b + 1][.]  row b of the expansion at (c, -h), the east face of xi = (1, 1): weights of
//                 C, R + L and R - L (FP64: of C, L and R, which saves the sums where every
//                 operation counts); dy: of the one at (-h, c), the north face. Mirrored for
//                 the other diagonals
//   px, pe           row term px (R - L) + pe (L - 2 C + R) of the expansion at (c, 0)
//   nu, nm, nd       weights of L + 4 C + R of the rows above, at and below at (0, c)
//   ge, gp, gd, b2   ties: see the row terms G, Q and B in the kernel
// Central: h, cu = 1/2 + h, cd = 1/2 - h, hk = h / 24.
template <typename T>
struct MarchCoefs {
    T dx[3][3], dy[3][3];
    T px, pe, nu, nm, nd, ge, gp, gd, b2;
    T h, cu, cd, hk;
};

// ---- a lane's columns of one row: a pair (float2, packed arithmetic) or one value -----
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 vfma(float a, float2 b, float2 c) { return __ffma2_rn(make_float2(a, a), b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vadd(float2 a, float b) { return __fadd2_rn(a, make_float2(b, b)); }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }   // (an operand modifier)
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return __fadd2_rn(a, vneg(b)); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float a, float2 b) { return __fmul2_rn(make_float2(a, a), b); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vneg(double a) { return -a; }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }

// Neighbouring columns: one shuffle a value or pair each way, and sums and differences
// taken per column (a pair built of a shuffled and an own value would cost the moves that
// line it up). Undefined at the warp's edges.
constexpr unsigned ALL = 0xffffffffu;
template <typename V>
struct Sides { V s, d; };   // right + left, right - left
__device__ __forceinline__ Sides<float2> vsides(float2 c) {
    const float l = __shfl_up_sync(ALL, c.y, 1), r = __shfl_down_sync(ALL, c.x, 1);
    return {make_float2(__fadd_rn(c.y, l), __fadd_rn(r, c.x)), make_float2(__fsub_rn(c.y, l), __fsub_rn(r, c.x))};
}
__device__ __forceinline__ float2 vless_left(float2 c) {    // c - left
    return make_float2(__fsub_rn(c.x, __shfl_up_sync(ALL, c.y, 1)), __fsub_rn(c.y, c.x));
}
__device__ __forceinline__ float2 vless_right(float2 c) {   // c - right
    return make_float2(__fsub_rn(c.x, c.y), __fsub_rn(c.y, __shfl_down_sync(ALL, c.x, 1)));
}
__device__ __forceinline__ float2 vplus_right(float2 a, float2 c) {   // a + right of c
    return make_float2(__fadd_rn(a.x, c.y), __fadd_rn(a.y, __shfl_down_sync(ALL, c.x, 1)));
}
template <typename V>
__device__ __forceinline__ Sides<V> vsides(V c) {
    const V l = __shfl_up_sync(ALL, c, 1), r = __shfl_down_sync(ALL, c, 1);
    return {vadd(r, l), vsub(r, l)};
}
template <typename V>
__device__ __forceinline__ V vless_left(V c) { return vsub(c, __shfl_up_sync(ALL, c, 1)); }
template <typename V>
__device__ __forceinline__ V vless_right(V c) { return vsub(c, __shfl_down_sync(ALL, c, 1)); }
template <typename V>
__device__ __forceinline__ V vplus_right(V a, V c) { return vadd(a, __shfl_down_sync(ALL, c, 1)); }

// columns of a lane: count, value of each, a pair of values
template <typename V>
struct Lane {
    using T = V;
    static constexpr int N = 1;
    __device__ static __forceinline__ V make(T a, T) { return a; }
    __device__ static __forceinline__ T first(V v) { return v; }
    __device__ static __forceinline__ T second(V v) { return v; }
};
template <>
struct Lane<float2> {
    using T = float;
    static constexpr int N = 2;
    __device__ static __forceinline__ float2 make(float a, float b) { return make_float2(a, b); }
    __device__ static __forceinline__ float first(float2 v) { return v.x; }
    __device__ static __forceinline__ float second(float2 v) { return v.y; }
};

// 1 / sqrt(g) for g well inside the normal range
__device__ __forceinline__ float rsqrt_n(float g) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(g));
    return r;
}
// 1 / sqrt(g), and 0 for g <= lim
__device__ __forceinline__ float vnorm(float g, float lim) { return g > lim ? rsqrt_n(g) : 0.0f; }
__device__ __forceinline__ double vnorm(double g, double lim) { return g > lim ? rsqrt(g) : 0.0; }
__device__ __forceinline__ float2 vnorm(float2 g, float lim) { return make_float2(vnorm(g.x, lim), vnorm(g.y, lim)); }

// a + b rounded stochastically (add_sr): the neighbour n of the rounded sum s on the side of
// the remainder e is taken with probability |e| / |n - s|; f: a uniform number in [1, 2)
// of 23 bits, half a bit of which is added
__device__ __forceinline__ float sr_next(float v, float r) {   // one step away from or toward zero
    return __int_as_float(__float_as_int(v) + (((__float_as_int(v) ^ __float_as_int(r)) >> 31) | 1));
}
__device__ __forceinline__ float sr_uniform(uint32_t bits) { return __uint_as_float((bits >> 9) | 0x3f800000u); }
__device__ __forceinline__ float vadd_sr(float a, float b, uint32_t cell, uint32_t seed) {
    const float s = vadd(a, b), bb = vsub(s, a), e = vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
    const float n = sr_next(s, e), t = vmul(vadd(sr_uniform(mix32(cell ^ seed)), -0.99999994f), vsub(n, s));
    return fabsf(t) < fabsf(e) ? n : s;
}
__device__ __forceinline__ float2 vadd_sr(float2 a, float2 b, uint32_t cell, uint32_t seed) {
    const float2 s = vadd(a, b), bb = vsub(s, a), e = vadd(vsub(a, vsub(s, bb)), vsub(b, bb));
    const float2 n = make_float2(sr_next(s.x, e.x), sr_next(s.y, e.y));
    const float2 f = make_float2(sr_uniform(mix32(cell ^ seed)), sr_uniform(mix32((cell + 1u) ^ seed)));
    const float2 t = vmul(vadd(f, -0.99999994f), vsub(n, s));
    return make_float2(fabsf(t.x) < fabsf(e.x) ? n.x : s.x, fabsf(t.y) < fabsf(e.y) ? n.y : s.y);
}

// ---- per-lane asynchronous copies ------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(uint32_t dst, const void *src) {
    static_assert(BYTES == 4 || BYTES == 8, "copy size");
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// sin and cos of pi x
__device__ __forceinline__ void sincospi_(float x, float &s, float &c) { sincospif(x, &s, &c); }
__device__ __forceinline__ void sincospi_(double x, double &s, double &c) { sincospi(x, &s, &c); }

template <typename T>
struct alignas(16) Row4 { T x, y, z, w; };

// Every prescribed velocity but the cell field is a product of a column and a row factor, u = cu(x)
// ru(y), v = cv(x) rv(y) (times the reversal factor). One sine and cosine serve both factors at an
// abscissa (ordinate) s: vortex sin^2(pi s / L), sin(2 pi s / L); deformation sin, cos(4 pi s / L).
template <typename T>
__device__ __forceinline__ void vel_waves(const StepParams<T> &p, T s, T &a, T &b) {
    T sn, cs;
    const bool def = p.vel_kind == VEL_DEFORM;
    sincospi_((def ? T(4) * s : s) / p.vp0, sn, cs);
    a = def ? sn : sn * sn;
    b = def ? cs : T(2) * sn * cs;
}
template <typename T>
__device__ __forceinline__ void vel_column(const StepParams<T> &p, T s, T &a, T &b) {
    if (p.vel_kind == VEL_VORTEX || p.vel_kind == VEL_DEFORM) {
        vel_waves(p, s, a, b);
        a *= -p.vp1;
        b *= p.vel_kind == VEL_DEFORM ? -p.vp1 : p.vp1;
    } else {
        a = p.vel_kind == VEL_UNIFORM ? p.vp0 : T(1);
        b = p.vel_kind == VEL_UNIFORM ? p.vp1 : p.vp2 * (s - p.vp0);
    }
}
template <typename T>
__device__ __forceinline__ void vel_row(const StepParams<T> &p, T s, T &a, T &b) {
    if (p.vel_kind == VEL_DEFORM) {
        vel_waves(p, s, a, b);
    } else if (p.vel_kind == VEL_VORTEX) {   // u takes sin(2 pi y / L), v sin^2(pi y / L)
        vel_waves(p, s, b, a);
    } else {
        a = p.vel_kind == VEL_UNIFORM ? T(1) : -p.vp2 * (s - p.vp1);
        b = T(1);
    }
}

// Geometry of a warp: 32 lanes x N columns; bar f^+ is valid on all of them, the expansions
// on all but the outer ones, and the cells but two columns from each edge are written: 60
// columns of 64, or 28 of 32. A strip of pairs starts at an odd column, x = 60 bx - 3 (lanes
// 1 to 30 are written, columns 60 bx - 1 to 60 bx + 58): with the ghost border of 5 a pair
// then lies on an 8-byte boundary of the plane (4 bytes in FP16 storage).
template <typename V, typename ST, int KIND = KIND_T2>
struct MarchTile {
    using T = typename Lane<V>::T;
    static constexpr int N = Lane<V>::N;
    static constexpr int TX = 32 * N - 4;                  // columns written (at most)
    // phi a plane of its own, or the sum of the state (FP64)
    static constexpr bool PHIP = Store<T, ST>::phi_plane;
    static constexpr int DEPTH = PHIP ? 3 : 4;             // rows in the ring
    // bytes of a lane's copy of the state (a single half value comes with its aligned pair)
    static constexpr int XB = N * (int)sizeof(ST) < 4 ? 4 : N * (int)sizeof(ST);
    static constexpr int PB = N * (int)sizeof(T);          // ... of phi
    static constexpr int oPo = 9 * 32 * XB;                // phi of the older level
    static constexpr int oP = oPo + 32 * PB;               // phi, one row ahead: columns -1 .. 32 N
    static constexpr int P0 = N;                           // index of column 0 there (aligned pairs)
    // (without phi planes: the state of the columns before and after the strip, 2 x 9 values)
    // second kernel of the three-stage scheme: the accumulator's moving directions and the plane
    // of its phi two rows below (without phi planes: all nine directions)
    static constexpr int oAcc = (oP + (PHIP ? 32 * N + P0 + N : 18) * (int)sizeof(T) + 15) / 16 * 16;
    static constexpr int slot = oAcc + (KIND == KIND_T3B ? 9 * 32 * PB : 0);
    // first kernel of the three-stage scheme: X + be (g - X) of its two outputs, rows j to j - 2
    static constexpr int oBase = DEPTH * slot;
    static constexpr int oRow = oBase + (KIND == KIND_T3A ? 3 * 16 * 32 * PB : 0);   // velocity factors of the segment's rows
    static constexpr int rows_extra = 4;                   // rows a segment reads past its own
    static constexpr int strips(int nx) { return (nx + (N == 2 ? 1 : 0) + TX - 1) / TX; }
    static constexpr int smem_bytes(int rows) { return oRow + (rows + rows_extra) * (int)sizeof(Row4<T>); }
};
static_assert(GHOST >= 5, "strips read 3 columns and rows past the grid");

// What a new row j gives: of row j - 1 the flux differences Dbar_k, without the differences over
// rows that wait for row j's own cells; those (e) of row j - 2 (upwind: the south faces, k = 6, 7, 8;
// central: the diagonals) and their sum; and the contributions of row j - 1 to the face moments
// phi_b of its four faces. Everything is a difference of face values, taken before it is
// added to anything: it vanishes where the state is uniform and keeps its digits elsewhere.
template <typename V>
struct RowOut {
    V D1, D2, D3, D4, D5, D6, D7, D8;
    V e2, e4, e6, e7, e8, es;
    V PE, PW, PN, PS;
};

// What a row j has to give (uniform over the warp): finished values of row j - 1, its flux
// differences, the middle terms of row j, the first terms of row j + 1. Only the first and
// last rows of a segment lack one.
struct Need { bool out, flux, mid, low; };

// The expansions of the rows in flight.
template <typename V, int FLUX>
struct March;

// Upwind faces (Eq. (26)). D_x, e, m below: (R - L) / 2, L - 2 C + R and (L + 4 C + R) / 6 of
// a row; the lattice-moment stencils are their products in the two directions, e.g.
// d/dx = (1 4 1)/6 (over rows) of D_x.
template <typename V>
struct March<V, 0> {
    using T = typename Lane<V>::T;
    // pending expansions: "a" of row j - 1 (waits for row j), "b" of row j (has row j - 1)
    struct Diag { V xa, xb, ya, yb; } g2, g4, g6, g8;
    V z1, q1, z5, q5, z3, m3p, z7, m7p, zA, vAp, zB, vBp, zN, gNp, qN1, qN2;
    V t3p, n2p, n4p, s6p, s7p, s8p;   // north- and south-face values of row j - 2

    __device__ __forceinline__ void clear(V z) {
        g2 = g4 = g6 = g8 = Diag{z, z, z, z};
        z1 = q1 = z5 = q5 = z3 = m3p = z7 = m7p = zA = vAp = zB = vBp = zN = gNp = qN1 = qN2 = z;
        t3p = n2p = n4p = s6p = s7p = s8p = z;
    }

    // a diagonal's row in the basis of its weights: C, R + L, R - L, or C, L, R
    struct Row { V c, u, v; };
    __device__ static __forceinline__ Row row(V C) {
        if constexpr (sizeof(T) == 8) {
            return Row{C, __shfl_up_sync(ALL, C, 1), __shfl_down_sync(ALL, C, 1)};
        } else {
            const Sides<V> q = vsides(C);
            return Row{C, q.s, q.d};
        }
    }
    template <int SX>
    __device__ static __forceinline__ V dot(const T (&w)[3], const Row &r, V acc) {
        if constexpr (sizeof(T) == 8) return vfma(w[SX > 0 ? 2 : 1], r.v, vfma(w[SX > 0 ? 1 : 2], r.u, vfma(w[0], r.c, acc)));
        else return vfma(T(SX) * w[2], r.v, vfma(w[1], r.u, vfma(w[0], r.c, acc)));
    }
    template <int SX>
    __device__ static __forceinline__ V dot(const T (&w)[3], const Row &r) {
        if constexpr (sizeof(T) == 8) return vfma(w[SX > 0 ? 2 : 1], r.v, vfma(w[SX > 0 ? 1 : 2], r.u, vmul(w[0], r.c)));
        else return vfma(T(SX) * w[2], r.v, vfma(w[1], r.u, vmul(w[0], r.c)));
    }
    // a diagonal direction (SX, SY): row b of the canonical stencil is row SY b here, and R - L
    // changes sign with SX
    template <int SX, int SY>
    __device__ static __forceinline__ void faces(const MarchCoefs<T> &cf, const Row &r, const Diag &g, V &ox, V &oy) {
        ox = dot<SX>(cf.dx[1 + SY], r, g.xa);
        oy = dot<SX>(cf.dy[1 + SY], r, g.ya);
    }
    // a row of a diagonal: the finished values at its two faces, and the pending sums
    template <int SX, int SY>
    __device__ static __forceinline__ void diagonal(const MarchCoefs<T> &cf, V C, Diag &g, V &ox, V &oy, Need n) {
        const Row r = row(C);
        if (n.out) faces<SX, SY>(cf, r, g, ox, oy);
        if (n.mid) {
            g.xa = dot<SX>(cf.dx[1], r, g.xb);
            g.ya = dot<SX>(cf.dy[1], r, g.yb);
        }
        if (n.low) {
            g.xb = dot<SX>(cf.dx[1 - SY], r);
            g.yb = dot<SX>(cf.dy[1 - SY], r);
        }
    }

    __device__ __forceinline__ void advance(const MarchCoefs<T> &cf, V F0, V F1, V F2, V F3, V F4, V F5, V F6, V F7,
                                            V F8, RowOut<V> &o, Need n) {
        V E2{}, E8{}, W4{}, W6{}, N2{}, N4{}, S6{}, S8{};
        diagonal<1, 1>(cf, F2, g2, E2, N2, n);
        diagonal<1, -1>(cf, F8, g8, E8, S8, n);
        diagonal<-1, 1>(cf, F4, g4, W4, N4, n);
        diagonal<-1, -1>(cf, F6, g6, W6, S6, n);
        const Sides<V> i0 = vsides(F0), i1 = vsides(F1), i5 = vsides(F5), i3 = vsides(F3), i7 = vsides(F7);
        // east face of k = 1, west face of k = 5
        const V e1 = vfma(T(-2), F1, i1.s), e5 = vfma(T(-2), F5, i5.s);
        V q = vfma(cf.px, i1.d, vmul(cf.pe, e1));
        const V T1 = vadd(z1, q);
        if (n.mid) z1 = vadd(vfma(T(4), q, F1), q1);
        q1 = q;
        q = vfma(-cf.px, i5.d, vmul(cf.pe, e5));
        const V T5 = vadd(z5, q);
        if (n.mid) z5 = vadd(vfma(T(4), q, F5), q5);
        q5 = q;
        // north face of k = 3, south face of k = 7
        const V m3 = vfma(T(4), F3, i3.s), m7 = vfma(T(4), F7, i7.s);
        const V T3 = vfma(cf.nu, m3, z3);
        if (n.mid) z3 = vfma(cf.nd, m3p, vfma(cf.nm, m3, F3));
        m3p = m3;
        const V T7 = vfma(cf.nd, m7, z7);
        if (n.mid) z7 = vfma(cf.nu, m7p, vfma(cf.nm, m7, F7));
        m7p = m7;
        // k = 0, 3, 7 at the east and west faces (weight 1/2 each): A even and B odd in x
        V A, B;
        {
            const V S = vadd(F0, vadd(F3, F7)), sS = vadd(i0.s, vadd(i3.s, i7.s));
            const V dS = vadd(i0.d, vadd(i3.d, i7.d)), dD = vsub(i7.d, i3.d);
            const V mP = vadd(m3, m7), mD = vsub(m7, m3);
            const V G = vfma(cf.ge, vfma(T(-2), S, sS), vmul(cf.gp, mP));
            A = vadd(zA, vfma(cf.gd, mD, G));
            if (n.mid) zA = vadd(vfma(T(0.5), S, vfma(T(4), G, vmul(T(-6) * cf.gp, mP))), vAp);
            if (n.low) vAp = vfma(-cf.gd, mD, G);
            const V u = vmul(T(1.0 / 48.0), dS);
            B = vadd(zB, vfma(cf.b2, dD, u));
            if (n.mid) zB = vfma(T(4), u, vBp);
            if (n.low) vBp = vfma(-cf.b2, dD, u);
        }
        if (n.flux) {
            o.PE = vadd(vadd(T1, vadd(E2, E8)), vadd(A, B));
            o.PW = vadd(vadd(T5, vadd(W4, W6)), vsub(A, B));
        }
        // k = 0, 1, 5 at the north and south faces
        {
            const V S = vadd(F0, vadd(F1, F5)), mS = vfma(T(4), S, vadd(i0.s, vadd(i1.s, i5.s)));
            const V dD = vsub(i5.d, i1.d), eP = vadd(e1, e5);
            const V G = vfma(cf.gd, dD, vfma(cf.gp, eP, vmul(cf.ge, mS)));
            A = vadd(zN, G);
            if (n.mid) zN = vadd(vfma(T(0.5), S, vfma(T(4), G, vmul(T(-6) * cf.ge, mS))), gNp);
            gNp = G;
            const V Q = vfma(T(1.0 / 48.0), mS, vmul(cf.b2, dD));
            B = vsub(Q, qN2);
            qN2 = qN1;
            qN1 = Q;
        }
        if (!n.out) return;
        o.PN = vadd(vadd(T3, vadd(N2, N4)), vadd(A, B));
        o.PS = vadd(vadd(T7, vadd(S6, S8)), vsub(A, B));
        // xi_y (f_N(c) - f_N(c - N)) for the directions that come from the row above
        o.e6 = vsub(s6p, S6);
        o.e7 = vsub(s7p, T7);
        o.e8 = vsub(s8p, S8);
        o.es = vadd(o.e7, vadd(o.e6, o.e8));
        s6p = S6;
        s7p = T7;
        s8p = S8;
        if (n.flux) {
            // Dbar_k = xi_x (f_E(c) - f_E(c - E)) + xi_y (f_N(c) - f_N(c - N))
            o.D1 = vless_left(T1);
            o.D5 = vless_right(T5);
            o.D2 = vadd(vless_left(E2), vsub(N2, n2p));
            o.D4 = vadd(vless_right(W4), vsub(N4, n4p));
            o.D3 = vsub(T3, t3p);
            o.D6 = vless_right(W6);
            o.D8 = vless_left(E8);
        }
        n2p = N2;
        n4p = N4;
        t3p = T3;
    }
};

// Central faces (Eq. (25)): f_E = (F_c + F_E) / 2 - h [xi_x (F_E - F_c) + xi_y (gy_c + gy_E) / 2] and
// likewise north: a part of each of the two cells. The face values are formed and then differenced,
// so that what one cell loses its neighbour gains whatever the coefficients' rounding. Their sums
// over k need the gradients of sum_k xi_y F_k and sum_k xi_x F_k only.
template <typename V>
struct March<V, 1> {
    using T = typename Lane<V>::T;
    struct Diag {
        V c1, m1, m2, zg, d1, nu, fn;   // C, m of row j - 1, m of row j - 2, gx pending, d; of f_N: own part of row j - 2, row j - 3
    } a2, a4, a6, a8;
    V q1, q5, z3, f3, z7, f7;       // Dbar of row j - 1 (k = 1, 5); own part of f_N of row j - 1, f_N of row j - 2 (k = 3, 7)
    V M0p, Mxp, Myp, my1, my2, zx, dx1;

    __device__ __forceinline__ void clear(V z) {
        a2 = a4 = a6 = a8 = Diag{z, z, z, z, z, z, z};
        q1 = q5 = z3 = f3 = z7 = f7 = M0p = Mxp = Myp = my1 = my2 = zx = dx1 = z;
    }

    // a row of a diagonal (SX, SY): the difference over columns of row j - 1, over rows of row j - 2
    template <int SX, int SY>
    __device__ static __forceinline__ void diagonal(const MarchCoefs<T> &cf, Diag &g, V C, V &D, V &e) {
        const Sides<V> q = vsides(C);
        const V m = vfma(T(4), C, q.s);
        const V gy = vmul(T(SY) * cf.hk, vsub(m, g.m2)), gx = vmul(T(SX) * cf.hk, vadd(g.zg, q.d));   // row j - 1
        // weights 1/2 + h, 1/2 - h of the upwind and the downwind cell
        const T up = cf.cu, dn = cf.cd;
        const V fE = vplus_right(vfma(SX > 0 ? up : dn, g.c1, vneg(gy)), vfma(SX > 0 ? dn : up, g.c1, vneg(gy)));
        const V own = vfma(SY > 0 ? up : dn, g.c1, vneg(gx)), south = vfma(SY > 0 ? dn : up, g.c1, vneg(gx));
        const V fN = vadd(g.nu, south);   // of row j - 2
        D = SX > 0 ? vless_left(fE) : vneg(vless_left(fE));
        e = SY > 0 ? vsub(fN, g.fn) : vsub(g.fn, fN);
        g.fn = fN;
        g.nu = own;
        g.c1 = C;
        g.m2 = g.m1;
        g.m1 = m;
        g.zg = vfma(T(4), q.d, g.d1);
        g.d1 = q.d;
    }

    __device__ __forceinline__ void advance(const MarchCoefs<T> &cf, V F0, V F1, V F2, V F3, V F4, V F5, V F6, V F7,
                                            V F8, RowOut<V> &o, Need) {
        const T h = cf.h, hk = cf.hk, up = cf.cu, dn = cf.cd;
        diagonal<1, 1>(cf, a2, F2, o.D2, o.e2);
        diagonal<-1, 1>(cf, a4, F4, o.D4, o.e4);
        diagonal<-1, -1>(cf, a6, F6, o.D6, o.e6);
        diagonal<1, -1>(cf, a8, F8, o.D8, o.e8);
        o.es = vadd(vadd(o.e2, o.e4), vadd(o.e6, o.e8));
        o.D1 = q1;
        o.D5 = vneg(q5);
        q1 = vless_left(vplus_right(vmul(up, F1), vmul(dn, F1)));
        q5 = vless_left(vplus_right(vmul(dn, F5), vmul(up, F5)));
        V f = vfma(dn, F3, z3);   // f_N of row j - 1
        o.D3 = vsub(f, f3);
        f3 = f;
        z3 = vmul(up, F3);
        f = vfma(up, F7, z7);
        o.D7 = vsub(f7, f);
        f7 = f;
        z7 = vmul(dn, F7);
        const V e = vadd(F2, F8), w = vadd(F4, F6), n = vadd(F2, F4), u = vadd(F6, F8);
        const V M0 = vadd(vadd(F0, vadd(F1, F5)), vadd(vadd(F3, F7), vadd(e, w)));
        const V Mx = vadd(vsub(F1, F5), vsub(e, w)), My = vadd(vsub(F3, F7), vsub(n, u));
        const V my = vfma(T(4), My, vsides(My).s);
        const V dx = vsides(Mx).d;
        const V bx = vfma(T(0.5), M0p, vmul(-hk, vsub(my, my2))), by = vfma(T(0.5), M0p, vmul(-hk, vadd(zx, dx)));
        o.PE = vfma(h, Mxp, bx);
        o.PW = vfma(-h, Mxp, bx);
        o.PN = vfma(h, Myp, by);
        o.PS = vfma(-h, Myp, by);
        my2 = my1;
        my1 = my;
        zx = vfma(T(4), dx, dx1);
        dx1 = dx;
        M0p = M0;
        Mxp = Mx;
        Myp = My;
    }
};

// One strip (rows y0 .. y0 + rows - 1) of one grid. FIELD: the velocity is given at cell
// centres (p.ufield, p.vfield). SUM_MASS: its sum of phi goes to mass_out; SUM_CHECK: a value that
// is not finite raises the status flag. (The sum is in FP64: a scheduler is busy with its conversions
// and additions for 256 cycles a row of pairs, of about 1200 in all.) KIND_T3A, KIND_T3B: the two kernels of the three-stage step
// (Sec. II.B.2),
//   T3A  out1 = X + be1 (g - X) + ga1 L (tilde f at t'), out2 = X + be2 (g - X) + ga2 L (the accumulator)
//   T3B  out1 = acc + be1 (g - X) + ga1 L (hat f at t_n + dt)
// with phi planes, phi of each output is that of its base plus the flux sum (two draws in T3A).
enum Sum { SUM_NONE, SUM_CHECK, SUM_MASS };
// launch mode: the next kernel may be scheduled at once; the launch fits into one wave of warps
enum MarchMode { MARCH_EARLY = 1, MARCH_ONE_WAVE = 2 };
// MID: rows 2 and 3 of a segment, which complete nothing, in a body of their own
template <typename V, typename ST, int FLUX, bool FIELD, int KIND, int SUM, bool MID = sizeof(V) == 4>
__device__ __forceinline__ void march_strip(const StepParams<typename Lane<V>::T> &p,
                                            const MarchCoefs<typename Lane<V>::T> &cf,
                                            const FastExtra<typename Lane<V>::T> &fe, int bx, int y0, int rows,
                                            double *mass_out, unsigned char *smem) {
    using T = typename Lane<V>::T;
    using LN = Lane<V>;
    using MT = MarchTile<V, ST, KIND>;
    constexpr bool T3A = KIND == KIND_T3A, T3B = KIND == KIND_T3B;
    constexpr bool DEV = Store<T, ST>::deviation;
    constexpr bool PHIP = MT::PHIP;
    // FP64 arithmetic is the scarce resource there: rows that complete nothing skip it
    constexpr bool SKIP = sizeof(T) == 8;
    constexpr int XB = MT::XB, PB = MT::PB, DEPTH = MT::DEPTH, N = LN::N;
    constexpr int LIGHT_ROWS = N == 2 && FLUX == 1 ? 0 : 2;
    static_assert(!MID || LIGHT_ROWS == 2, "the first four rows have bodies of their own");
    const int lane = threadIdx.x & 31;
    const int nx = p.nx, ny = p.ny;
    // the strip's width and the columns before it. FP64 strips of at most 26 columns leave out
    // the outermost lanes, whose phi needs a sum over the column past the strip
    const int tx = N == 2 ? MT::TX : p.tile_w;
    const bool wide = PHIP || tx > 26;
    const int hx = N == 2 || !wide ? 3 : 2;
    const int x = tx * bx - hx + N * lane;   // the lane's first column
    // element offset of the lane's columns in a row; lanes past the ghost border read padding
    const int col = min(x + GHOST, p.pitch - N);
    const bool wr = N == 2 ? lane >= 1 && lane <= 30 : lane >= hx && lane < hx + tx;
    const bool ok0 = wr && x >= 0 && x < nx, ok1 = N == 2 && wr && x + 1 >= 0 && x + 1 < nx;
    const int npk = rows + MT::rows_extra;

    // ---- velocity factors
    Row4<T> *sRow = reinterpret_cast<Row4<T> *>(smem + MT::oRow);
    const bool reversing = p.vel_kind == VEL_VORTEX || p.vel_kind == VEL_DEFORM;
    const T vct = reversing ? fe.vc_t : T(1), vco = reversing ? fe.vc_told : T(1), vcf = reversing ? fe.vc_tface : T(1);
    // flux terms carry the output's gamma; with two outputs they are kept without it
    const T ga = T3A ? T(1) : p.ga1;
    const T gc2 = ga * p.c2, hg3 = T(0.5) * ga * p.c3;
    const T f3 = T(3) * gc2;               // (face velocities carry 3 gamma c2)
    V cu{}, cv{}, cuE{}, cvE{};            // column factors at the centres and east faces
    if constexpr (!FIELD) {
        const T g0 = T(wrap_small(x, nx)), g1 = T(wrap_small(x + 1, nx)), ff = vcf * f3;
        T a0, b0, a1 = T(0), b1 = T(0);
        vel_column(p, g0 + T(0.5), a0, b0);
        if (N == 2) vel_column(p, g1 + T(0.5), a1, b1);
        cu = LN::make(a0, a1);
        cv = LN::make(b0, b1);
        vel_column(p, g0 + T(1), a0, b0);
        if (N == 2) vel_column(p, g1 + T(1), a1, b1);
        cuE = LN::make(a0 * ff, a1 * ff);
        cvE = LN::make(b0 * ff, b1 * ff);
        for (int i = lane; i < npk; i += 32) {
            const T g = T(wrap_small(y0 - 2 + i, ny));
            Row4<T> r;
            vel_row(p, g + T(0.5), r.x, r.y);
            vel_row(p, g + T(1), r.z, r.w);
            r.z *= ff;
            r.w *= ff;
            sRow[i] = r;
        }
    }
    pdl_wait();   // the previous kernel's output (launched with programmatic serialization)

    // ---- copies: packet i holds the state and phi_old of row y0 - 2 + i and phi of the row above
    // (without phi planes phi of the row above is summed from the next packet)
    const uint32_t ring = smem_u32(smem);
    const size_t row0 = (size_t)(y0 - 2 + GHOST) * p.pitch;
    const ST *gX = static_cast<const ST *>(p.X) + row0 + (DEV && N == 1 ? col & ~1 : col);
    const T *gPo = p.phi_old + row0 + col;
    const T *gP = PHIP ? p.phi_cur + row0 + p.pitch + col : nullptr;
    // lane 0 also fetches the column before the strip, lane 31 the one after it
    const int hcol = lane == 0 ? max(x + GHOST - 1, 0) : min(x + N + GHOST, p.pitch - 1);
    const T *gH = PHIP ? p.phi_cur + row0 + p.pitch + hcol : static_cast<const T *>(p.X) + row0 + hcol;
    const bool halo = wide && (lane == 0 || lane == 31);
    const uint32_t hdst = MT::oP + (PHIP ? lane == 0 ? MT::P0 - 1 : MT::P0 + 32 * N : lane == 0 ? 0 : 9) * (int)sizeof(T);
    const int packets = PHIP ? npk : npk + 1;
    const T *gA = T3B ? static_cast<const T *>(p.acc) + row0 + col : nullptr;
    const T *gPa = T3B && PHIP ? p.phi_acc + row0 - 2 * p.pitch + col : nullptr;
    const size_t plane = p.plane;
    int fetched = 0;
    uint32_t fslot = 0;   // byte offset of the slot the next packet goes to
    auto fetch = [&]() {
        if (fetched < packets) {
            const uint32_t s = ring + fslot;
#pragma unroll
            for (int k = 0; k < 9; k++) cp_async<XB>(s + k * 32 * XB + lane * XB, gX + k * plane);
            cp_async<PB>(s + MT::oPo + lane * PB, gPo);
            if constexpr (PHIP) {
                cp_async<PB>(s + MT::oP + (MT::P0 + N * lane) * (int)sizeof(T), gP);
                if (halo) cp_async<(int)sizeof(T)>(s + hdst, gH);
            } else if (halo) {
#pragma unroll
                for (int k = 0; k < 9; k++) cp_async<(int)sizeof(T)>(s + hdst + k * (int)sizeof(T), gH + k * plane);
            }
            if constexpr (T3B) {
#pragma unroll
                for (int k = PHIP ? 1 : 0; k < 9; k++)
                    cp_async<PB>(s + MT::oAcc + k * 32 * PB + lane * PB, gA + k * plane);
                if constexpr (PHIP) {
                    cp_async<PB>(s + MT::oAcc + lane * PB, gPa);
                    gPa += p.pitch;
                }
                gA += p.pitch;
            }
            gX += p.pitch;
            gPo += p.pitch;
            gP += p.pitch;
            gH += p.pitch;
            fetched++;
            fslot = fslot + MT::slot == DEPTH * MT::slot ? 0 : fslot + MT::slot;
        }
        cp_commit();   // (an empty group at the end keeps the count of groups in step)
    };
#pragma unroll
    for (int i = 0; i < DEPTH - 1; i++) fetch();

    // FIELD: the cell field is read from its planes a row at a time (rows j, j - 1, j - 2)
    const T *gU = nullptr, *gW = nullptr;
    V fu0{}, fv0{}, fu1{}, fv1{}, fu2{}, fv2{};
    if constexpr (FIELD) {
        gU = p.ufield + row0 + col;
        gW = p.vfield + row0 + col;
    }
    // V = theta n + 3 d(phi u)/dt: the second term is u_spatial (phi vD + phi_old vDo)
    const T vD = p.useD ? T(3) * p.inv_dtD * vct : T(0), vDo = p.useD ? T(-3) * p.inv_dtD * vco : T(0);
    const T v3 = T(3) * vct;

    // ---- rows below the first packet: phi of rows y0 - 3 and y0 - 2
    V pc1, pc2{}, pc3{};           // phi of rows j, j - 1, j - 2
    V pd1, pm1, pm0, pz;           // gradient rows: R - L, L + 4 C + R; 4 d(j) + d(j - 1)
    {
        auto row = [&](V c, T l, T r, V &d, V &m) {
            if constexpr (N == 2) {
                d = LN::make(LN::second(c) - l, r - LN::first(c));
                m = vfma(T(4), c, LN::make(LN::second(c) + l, r + LN::first(c)));
            } else {
                d = r - l;
                m = vfma(T(4), c, r + l);
            }
        };
        V d0, a, b;
        T al, ar, bl, br;
        if constexpr (PHIP) {
            const T *q = p.phi_cur + row0 - p.pitch + col;
            const int lo = x + GHOST - 1 < 0 ? 0 : -1, hi = col + N < p.pitch ? N : N - 1;
            a = *reinterpret_cast<const V *>(q);
            b = *reinterpret_cast<const V *>(q + p.pitch);
            al = q[lo];
            ar = q[hi];
            bl = q[p.pitch + lo];
            br = q[p.pitch + hi];
        } else {   // sum_k X_k, the outer lanes also of the columns past the strip
            auto sum = [&](const T *q) {
                T t = T(0);
#pragma unroll
                for (int k = 0; k < 9; k++) t += q[k * plane];
                return t;
            };
            const T *q = static_cast<const T *>(p.X) + row0 - p.pitch;
            a = sum(q + col);
            b = sum(q + p.pitch + col);
            T ha = T(0), hb = T(0);
            if (halo) {
                ha = sum(q + hcol);
                hb = sum(q + p.pitch + hcol);
            }
            al = __shfl_up_sync(ALL, a, 1);
            ar = __shfl_down_sync(ALL, a, 1);
            bl = __shfl_up_sync(ALL, b, 1);
            br = __shfl_down_sync(ALL, b, 1);
            if (lane == 0) al = ha, bl = hb;
            if (lane == 31) ar = ha, br = hb;
        }
        row(a, al, ar, d0, pm0);
        row(b, bl, br, pd1, pm1);
        pz = vfma(T(4), pd1, d0);
        pc1 = b;
    }
    const T gmc = ga * (T(1) - p.c2);
    March<V, FLUX> mx;
    mx.clear(V{});
    // rows in flight: X + be (g - X) of row j - 1; the same less the flux of row j - 2
    V b1{}, b2{}, b3{}, b4{}, b5{}, b6{}, b7{}, b8{};
    V r1{}, r2{}, r3{}, r4{}, r5{}, r6{}, r7{}, r8{};
    V sDp{}, phEp{}, pNp{};            // row j - 2: flux sum, phi_b east, own part of phi_b north
    V v0x{}, v0y{}, v1x{}, v1y{};      // V of rows j - 1, j - 2
    V f0p{}, f1p{}, f2p{};             // north-face moments of row j - 3
    double msum = 0.0;
    V check{};                         // 0, or NaN once a value was not finite
    V pa0{}, pa1{}, pa2{};             // T3B without phi planes: phi of the accumulator, rows j to j - 2
    uint32_t cslot = 0;
    const uint32_t seed = PHIP ? mix32(p.seed) : 0u;
    // lanes whose columns have images in the ghost border left or right of the grid
    const bool xedge = x < GHOST || x + N - 1 >= nx - GHOST;

    __syncwarp();
    // one row of the march; stage 0: the first two rows, which only enter the pending sums; stage 1:
    // the next two, which complete no row of the segment; stage 2: the others (and, where MID is false,
    // rows that the stages before would serve: they store nothing)
    auto row = [&](int it, auto stage) {
        constexpr bool LIGHT = decltype(stage)::value == 0, OUT = decltype(stage)::value == 2;
        cp_wait<1>();
        __syncwarp();
        fetch();
        const unsigned char *sl = smem + cslot;
        cslot = cslot + MT::slot == DEPTH * MT::slot ? 0 : cslot + MT::slot;

        // ---- phi of the row above, gradient and cell quantities of row j ------------
        V pc0;
        T pl, pr;
        if constexpr (PHIP) {
            const T *sP = reinterpret_cast<const T *>(sl + MT::oP) + MT::P0 + N * lane;
            pc0 = *reinterpret_cast<const V *>(sP);
            pl = sP[-1];
            pr = sP[N];
        } else {
            const unsigned char *sn = smem + cslot;   // the next packet
            pc0 = V{};
#pragma unroll
            for (int k = 0; k < 9; k++) pc0 = vadd(pc0, *reinterpret_cast<const V *>(sn + k * 32 * XB + lane * XB));
            T h = T(0);
            if (halo) {
                const T *q = reinterpret_cast<const T *>(sn + hdst);
#pragma unroll
                for (int k = 0; k < 9; k++) h = vadd(h, q[k]);
            }
            pl = __shfl_up_sync(ALL, pc0, 1);
            pr = __shfl_down_sync(ALL, pc0, 1);
            if (lane == 0) pl = h;
            if (lane == 31) pr = h;
        }
        V pd0, pmn;
        if constexpr (N == 2) {
            pd0 = LN::make(__fsub_rn(LN::second(pc0), pl), __fsub_rn(pr, LN::first(pc0)));
            pmn = vfma(T(4), pc0, LN::make(__fadd_rn(LN::second(pc0), pl), __fadd_rn(pr, LN::first(pc0))));
        } else {
            pd0 = vsub(pr, pl);
            pmn = vfma(T(4), pc0, vadd(pr, pl));
        }
        const V gx = vadd(pz, pd0), gy = vsub(pmn, pm0);   // 12 grad phi
        pz = vfma(T(4), pd0, pd1);
        pd1 = pd0;
        pm0 = pm1;
        pm1 = pmn;
        const V ph = pc1;
        V Vx, Vy, Px, Py;
        {
            // n = grad phi / |grad phi|; 0 where |grad phi|^2 <= 1e-24 (Eq. (2))
            V inv = vnorm(vfma(gx, gx, vmul(gy, gy)), T(144e-24));
            inv = vmul(inv, vmul(vmul(p.theta_c, vadd(ph, -p.phiA)), vadd(ph, -p.phiB)));   // theta of Eq. (4)
            const V po = *reinterpret_cast<const V *>(sl + MT::oPo + lane * PB);
            const V w = vfma(vD, ph, vmul(vDo, po));
            V us, vs;
            if constexpr (FIELD) {
                fu2 = fu1; fv2 = fv1; fu1 = fu0; fv1 = fv0;
                fu0 = *reinterpret_cast<const V *>(gU);
                fv0 = *reinterpret_cast<const V *>(gW);
                gU += p.pitch;
                gW += p.pitch;
                us = fu0;
                vs = fv0;
            } else {
                const Row4<T> rf = sRow[it];
                us = vmul(rf.x, cu);
                vs = vmul(rf.y, cv);
            }
            Vx = vfma(gx, inv, vmul(us, w));             // Eq. (14b)
            Vy = vfma(gy, inv, vmul(vs, w));
            const V p3 = vmul(v3, ph);
            Px = vfma(us, p3, vmul(p.tau, Vx));          // g_k = w_k (phi + xi_k . P)
            Py = vfma(vs, p3, vmul(p.tau, Vy));
        }

        // ---- bar f^+_k = X + b (g - X) and X + be (g - X) of row j -------------------
        V F0, F1, F2, F3, F4, F5, F6, F7, F8;
        V nb1, nb2, nb3, nb4, nb5, nb6, nb7, nb8;
        {
            // returns X + be (g - X) (T3B: with the accumulator in the place of X)
            auto cell = [&](int k, V g, V &F) -> V {
                const T wk = wq<T>(k);
                const unsigned char *q = sl + k * 32 * XB + lane * XB;
                V X, t;
                if constexpr (DEV) {
                    V h;
                    if constexpr (N == 2) h = __half22float2(*reinterpret_cast<const __half2 *>(q));
                    else h = __half2float(reinterpret_cast<const __half *>(q)[col & 1]);
                    X = vfma(p.qinv, h, ph);
                    t = vmul(wk, vsub(g, X));
                    X = vmul(wk, X);
                } else {
                    X = *reinterpret_cast<const V *>(q);
                    t = vfma(wk, g, vneg(X));
                }
                F = vfma(p.b, t, X);
                if (k == 0 || LIGHT || (SKIP && it > npk - 3)) return V{};
                if constexpr (T3A) {
                    V *q2 = reinterpret_cast<V *>(smem + MT::oBase + (it % 3) * 16 * 32 * PB) + (2 * k - 2) * 32 + lane;
                    q2[0] = vfma(p.be1, t, X);
                    q2[32] = vfma(p.be2, t, X);
                    return V{};
                } else if constexpr (T3B) {
                    return vfma(p.be1, t, *reinterpret_cast<const V *>(sl + MT::oAcc + k * 32 * PB + lane * PB));
                } else {
                    return vfma(p.be1, t, X);
                }
            };
            const V gp = vadd(ph, Px), gm = vsub(ph, Px);
            cell(0, ph, F0);
            nb1 = cell(1, gp, F1);
            nb2 = cell(2, vadd(gp, Py), F2);
            nb3 = cell(3, vadd(ph, Py), F3);
            nb4 = cell(4, vadd(gm, Py), F4);
            nb5 = cell(5, gm, F5);
            nb6 = cell(6, vsub(gm, Py), F6);
            nb7 = cell(7, vsub(ph, Py), F7);
            nb8 = cell(8, vsub(gp, Py), F8);
            if constexpr (T3B && !PHIP) {
                pa2 = pa1; pa1 = pa0;
                if (it >= 2 && it <= npk - 3) {
                    pa0 = V{};
#pragma unroll
                    for (int k = 0; k < 9; k++)
                        pa0 = vadd(pa0, *reinterpret_cast<const V *>(sl + MT::oAcc + k * 32 * PB + lane * PB));
                }
            }
        }

        V phn{}, phn2{}, pho{};
        V o[9], o2[9];
        const int y = y0 + it - 4;
        // ---- expansions: row j completes row j - 1 -----------------------------------
        RowOut<V> ro;
        mx.advance(cf, F0, F1, F2, F3, F4, F5, F6, F7, F8, ro,
                   LIGHT  ? Need{false, false, !SKIP || it >= 1, true}
                   : SKIP ? Need{true, it >= 3 && it <= npk - 2, it <= npk - 2, it <= npk - 3}
                          : Need{true, true, true, true});
        if constexpr (!LIGHT) {

        // ---- row j - 2 is complete: faces, flux and store ----------------------------
        // (FP32: computed in the next two rows too, where nothing is stored: one straight block)
        if (!SKIP || it >= 3) {
        const V phN = vadd(pNp, ro.PS), phE = phEp;
        // face moments: phi_b and (3 gamma c2 phi_b u_b + gamma c3 V_b) at the east and north faces
        const T hf = T(0.5) * f3;
        Row4<T> rf{};
        V uN, vN;
        if constexpr (FIELD) {
            uN = vmul(hf, vadd(fu2, fu1));
            vN = vmul(hf, vadd(fv2, fv1));
        } else {
            rf = sRow[max(it - 2, 0)];
            uN = vmul(rf.z, cu);
            vN = vmul(rf.w, cv);
        }
        const V y1 = vfma(phN, uN, vmul(hg3, vadd(v1x, v0x)));
        const V y2 = vfma(phN, vN, vmul(hg3, vadd(v1y, v0y)));
        if (OUT && (MID || !SKIP || it >= 4)) {
            V uE, vE;
            if constexpr (FIELD) {
                uE = vmul(hf, vplus_right(fu2, fu2));
                vE = vmul(hf, vplus_right(fv2, fv2));
            } else {
                uE = vmul(rf.x, cuE);
                vE = vmul(rf.y, cvE);
            }
            const V x1 = vfma(phE, uE, vmul(hg3, vplus_right(v1x, v1x)));
            const V x2 = vfma(phE, vE, vmul(hg3, vplus_right(v1y, v1y)));
            const V A1 = vmul(gc2, vless_left(phE)), A2 = vmul(gc2, vsub(phN, f0p));
            const V B1 = vless_left(x1), B2 = vadd(vless_left(x2), vsub(y1, f1p)), B3 = vsub(y2, f2p);
            const V S13 = vadd(B1, B3);
            // new phi = phi + gamma sum_k L_k (sum_k w_k xi_k = 0, sum_k w_k xi_a xi_b = delta_ab / 3)
            const V dph = vfma(T(-1.0 / 3.0), S13, vmul(-gmc, vadd(sDp, ro.es)));
            V phb = pc3;
            if constexpr (T3B) phb = PHIP ? *reinterpret_cast<const V *>(sl + MT::oAcc + lane * PB) : pa2;
            const V dph1 = T3A ? vmul(p.ga1, dph) : dph;
            if constexpr (PHIP) phn = vadd_sr(phb, dph1, (uint32_t)y * (uint32_t)nx + (uint32_t)x, seed);
            else phn = vadd(phb, dph1);
            if constexpr (T3A) {
                const V dph2 = vmul(p.ga2, dph);
                if constexpr (PHIP) phn2 = vadd_sr(phb, dph2, (uint32_t)y * (uint32_t)nx + (uint32_t)x, ~seed);
                else phn2 = vadd(phb, dph2);
            }
            {
                // gamma w_k (c2 Phi_k + c3 Psi_k) = w_k (xi_x A1 + xi_y A2 + xi_x^2 B1 + xi_x xi_y B2 + xi_y^2 B3)
                const T w1 = wq<T>(1), w2 = wq<T>(2);
                // (the differences over rows that waited)
                const V p7 = FLUX == 0 ? vfma(-gmc, ro.e7, r7) : r7;
                const V p6 = vfma(-gmc, ro.e6, r6), p8 = vfma(-gmc, ro.e8, r8);
                const V p2 = FLUX == 0 ? r2 : vfma(-gmc, ro.e2, r2), p4 = FLUX == 0 ? r4 : vfma(-gmc, ro.e4, r4);
                o[1] = vfma(-w1, vadd(B1, A1), r1);
                o[5] = vfma(-w1, vsub(B1, A1), r5);
                o[3] = vfma(-w1, vadd(B3, A2), r3);
                o[7] = vfma(-w1, vsub(B3, A2), p7);
                const V sp = vadd(S13, B2), sm = vsub(S13, B2), ap = vadd(A1, A2), am = vsub(A1, A2);
                o[2] = vfma(-w2, vadd(sp, ap), p2);
                o[6] = vfma(-w2, vsub(sp, ap), p6);
                o[8] = vfma(-w2, vadd(sm, am), p8);
                o[4] = vfma(-w2, vsub(sm, am), p4);
                if constexpr (T3A) {
                    const V *q2 = reinterpret_cast<const V *>(smem + MT::oBase + ((it + 1) % 3) * 16 * 32 * PB) + lane;
#pragma unroll
                    for (int k = 1; k < 9; k++) {
                        o2[k] = vfma(p.ga2, o[k], q2[(2 * k - 1) * 32]);
                        o[k] = vfma(p.ga1, o[k], q2[(2 * k - 2) * 32]);
                    }
                    o2[0] = vsub(phn2, vadd(vadd(vadd(o2[1], o2[2]), vadd(o2[3], o2[4])),
                                            vadd(vadd(o2[5], o2[6]), vadd(o2[7], o2[8]))));
                }
                // rest component: the new phi is exactly phn (up to this subtraction)
                o[0] = vsub(phn, vadd(vadd(vadd(o[1], o[2]), vadd(o[3], o[4])), vadd(vadd(o[5], o[6]), vadd(o[7], o[8]))));
            }
        }
        f0p = phN;
        f1p = y1;
        f2p = y2;
        }
        pho = PHIP ? phn : pc3;   // (without phi planes: phi of X, the next step's older level)
        // ---- row j - 1: X + be (g - X) - gamma (1 - c2) Dbar ---------------------------
        if (!SKIP || (it >= 3 && it <= npk - 2)) {
        // (b is 0 where the bases are kept apart: T3A)
        r1 = vfma(-gmc, ro.D1, b1);
        r2 = vfma(-gmc, ro.D2, b2);
        r3 = vfma(-gmc, ro.D3, b3);
        r4 = vfma(-gmc, ro.D4, b4);
        r5 = vfma(-gmc, ro.D5, b5);
        r6 = vfma(-gmc, ro.D6, b6);
        r7 = FLUX == 0 ? b7 : vfma(-gmc, ro.D7, b7);
        r8 = vfma(-gmc, ro.D8, b8);
        sDp = vadd(vadd(vadd(ro.D1, ro.D2), vadd(ro.D3, ro.D4)), vadd(vadd(ro.D5, ro.D6), FLUX == 0 ? ro.D8 : vadd(ro.D7, ro.D8)));
        phEp = vplus_right(ro.PE, ro.PW);
        }
        pNp = ro.PN;
        }
        b1 = nb1; b2 = nb2; b3 = nb3; b4 = nb4; b5 = nb5; b6 = nb6; b7 = nb7; b8 = nb8;
        v1x = v0x; v1y = v0y;
        v0x = Vx; v0y = Vy;
        pc3 = pc2; pc2 = pc1; pc1 = pc0;
        if constexpr (!OUT) return;

        // ---- store row j - 2 -----------------------------------------------------------
        const bool st0 = ok0 && (MID || it >= 4), st1 = ok1 && (MID || it >= 4);
        using OV = typename std::conditional<!DEV, V, typename std::conditional<N == 2, __half2, __half>::type>::type;
        const size_t g0 = (size_t)(y + GHOST) * p.pitch + (size_t)(x + GHOST);
        // nine values and (unless Q is null) phi; images: also into the ghost border
        auto store = [&](const OV (&ov)[9], ST *O, const V ph, T *Q, bool images) {
            // one column of this lane at element offset g
            auto put0 = [&](long long g) {
#pragma unroll
                for (int k = 0; k < 9; k++) {
                    if constexpr (N == 2) O[(long long)(k * plane) + g] = ov[k].x;
                    else O[(long long)(k * plane) + g] = ov[k];
                }
                if constexpr (!T3B || PHIP) Q[g] = LN::first(ph);
            };
            auto put1 = [&](long long g) {
                if constexpr (N == 2) {
#pragma unroll
                    for (int k = 0; k < 9; k++) O[(long long)(k * plane) + g + 1] = ov[k].y;
                    if constexpr (!T3B || PHIP) Q[g + 1] = LN::second(ph);
                }
            };
            if (st0 && (N == 1 || st1)) {
#pragma unroll
                for (int k = 0; k < 9; k++) *reinterpret_cast<OV *>(O + k * plane + g0) = ov[k];
                if constexpr (!T3B || PHIP) *reinterpret_cast<V *>(Q + g0) = ph;
            } else if (st0) {
                put0(g0);
            } else if (st1) {
                put1(g0);
            }
            // periodic images in the ghost border
            if (images && (st0 || st1) && (xedge || y < GHOST || y >= ny - GHOST)) {
#pragma unroll 1
                for (int im = 0; im < 9; im++) {
                    const int ay = im / 3 - 1, ax = im - 3 * (im / 3) - 1;
                    const int yy = y + ay * ny, xx = x + ax * nx;
                    if (im == 4 || yy < -GHOST || yy >= ny + GHOST) continue;
                    const long long gi = (long long)(yy + GHOST) * p.pitch + (xx + GHOST);
                    if (st0 && xx >= -GHOST && xx < nx + GHOST) put0(gi);
                    if (st1 && xx + 1 >= -GHOST && xx + 1 < nx + GHOST) put1(gi);
                }
            }
        };
        if constexpr (DEV) {
            OV ov[9];
#pragma unroll
            for (int k = 0; k < 9; k++) {
                const V q = vmul(p.qscale / wq<T>(k), vfma(-wq<T>(k), phn, o[k]));
                if constexpr (N == 2) ov[k] = __float22half2_rn(q);
                else ov[k] = __float2half_rn(q);
            }
            store(ov, static_cast<ST *>(p.out1), pho, p.phi_out, true);
        } else {
            store(o, static_cast<ST *>(p.out1), pho, p.phi_out, true);
            if constexpr (T3A) {   // the accumulator is read per cell only: no images
                if constexpr (PHIP) {
                    store(o2, p.out2, phn2, p.phi_out2, false);
                } else if (st0) {
#pragma unroll
                    for (int k = 0; k < 9; k++) p.out2[k * plane + g0] = o2[k];
                }
            }
        }
        if constexpr (SUM == SUM_MASS) {
            if (st0) msum += (double)LN::first(phn);
            if (st1) msum += (double)LN::second(phn);
        } else if constexpr (SUM == SUM_CHECK) {
            if (st0 || st1) check = vfma(T(0), phn, check);
        }
    };
    // (pairs with central faces: a second loop body costs registers, 4096^2 323 -> 371 us; else it
    // gives 256^2 9.1 -> 8.4, 1024^2 38.5 -> 37.6, 4096^2 354 -> 350 us. MID, single columns: 64^2
    // 4.8 -> 3.9, 256^2 7.9 -> 7.6, three-stage 64^2 11.8 -> 9.7 us; FP64 loses: 64^2 47.1 -> 48.8)
#pragma unroll 1
    for (int it = 0; it < LIGHT_ROWS; it++) row(it, std::integral_constant<int, 0>{});
    if constexpr (MID) {
#pragma unroll 1
        for (int it = 2; it < 4; it++) row(it, std::integral_constant<int, 1>{});
    }
    constexpr int UNROLL = sizeof(T) == 8 ? 1 : 2;   // (FP64: the arithmetic hides the moves that two rows would save)
#pragma unroll UNROLL
    for (int it = MID ? 4 : LIGHT_ROWS; it < npk; it++) row(it, std::integral_constant<int, 2>{});
    cp_wait<0>();
    if constexpr (SUM == SUM_MASS) {
        for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(ALL, msum, o);
        if (lane == 0) *mass_out = msum;
    } else if constexpr (SUM == SUM_CHECK) {
        const bool bad = (ok0 && !(LN::first(check) == T(0))) || (ok1 && !(LN::second(check) == T(0)));
        if (__any_sync(ALL, bad) && lane == 0) atomicOr(p.status, 1);
    }
}

// One grid: blockIdx.x = strip, blockIdx.y = segment of p.tile_h rows. MARCH_EARLY: dependents may
// be scheduled at once (a grid that leaves room for them on the chip: their velocity factors
// are ready when this grid ends).
template <typename V, typename ST, int FLUX, bool FIELD, int KIND, int SUM, bool MID>
__global__ void __launch_bounds__(32, (sizeof(V) == 4 ? 12 : 8))
step_march_kernel(const __grid_constant__ StepParams<typename Lane<V>::T> p,
                  const __grid_constant__ MarchCoefs<typename Lane<V>::T> cf,
                  const __grid_constant__ FastExtra<typename Lane<V>::T> fe, const int mode) {
    extern __shared__ __align__(128) unsigned char smem[];
    if (mode & MARCH_EARLY) pdl_trigger();
    const int y0 = blockIdx.y * p.tile_h;
    march_strip<V, ST, FLUX, FIELD, KIND, SUM, MID>(
        p, cf, fe, blockIdx.x, y0, min(p.tile_h, p.ny - y0),
        SUM == SUM_MASS ? p.mass_partial + blockIdx.y * p.tiles_x + blockIdx.x : nullptr, smem);
    if (!(mode & MARCH_EARLY)) pdl_trigger();
}

// ---- many grids per launch ----------------------------------------------------
// Steps that one replayed graph takes; the reversal factors of that many are kept ready.
constexpr int GRAPH_STEPS = 8;

// Per-grid descriptor of a batch, in device memory. `step` counts the grid's steps; with the
// launch's offset in its group it selects the ping-pong state set and the phi plane roles. It is
// advanced by batch_advance_kernel at the end of the group, so a captured sequence of launches
// stays valid while grids join and leave (their step counters differ).
template <typename T>
struct BatchGrid {
    void *X[2];              // state sets 0, 1
    T *phi[3];               // phi planes
    long long step, target;  // steps taken; the grid is frozen once step == target
    size_t plane;
    int nx, ny, pitch, tile_w;
    int vel_kind, pad_;
    double vp[3];            // velocity parameters (FP64; rounded per precision in the kernel)
    T vc[GRAPH_STEPS][3];    // single vortex: cos(pi t / T) at t, t - dt, t + dt/2 of the next steps
};

// Parameters common to every grid of a batch (same W, M, cfl, order, flux, precision).
template <typename T>
struct BatchUniform {
    T b, c2, c3, be1, ga1, tau, theta_c, phiA, phiB, inv_dt, qscale, qinv;
    double dt;
    int dtphiu;
    int *status;
};

// The parameters of a grid's step `ofs` of the group.
template <typename T, typename ST>
__device__ __forceinline__ void batch_step_params(const BatchUniform<T> &u, const BatchGrid<T> *G, int ofs,
                                                  StepParams<T> &p, FastExtra<T> &fe) {
    const long long step = G->step + ofs;
    p.nx = G->nx;
    p.ny = G->ny;
    p.pitch = G->pitch;
    p.plane = G->plane;
    p.tile_w = G->tile_w;
    p.status = u.status;
    p.ufield = p.vfield = nullptr;
    p.b = u.b;
    p.c2 = u.c2;
    p.c3 = u.c3;
    p.be1 = u.be1;
    p.ga1 = u.ga1;
    p.tau = u.tau;
    p.theta_c = u.theta_c;
    p.phiA = u.phiA;
    p.phiB = u.phiB;
    p.inv_dtD = u.inv_dt;
    p.useD = (u.dtphiu && step > 0) ? 1 : 0;
    p.seed = (uint32_t)step;
    p.vel_kind = G->vel_kind;
    p.vp0 = (T)G->vp[0];
    p.vp1 = (T)G->vp[1];
    p.vp2 = (T)G->vp[2];
    p.qscale = u.qscale;
    p.qinv = u.qinv;
    fe.vc_t = G->vc[ofs][0];
    fe.vc_told = G->vc[ofs][1];
    fe.vc_tface = G->vc[ofs][2];
    const int cur = (int)(step & 1);
    p.X = G->X[cur];
    p.out1 = G->X[1 - cur];
    int iPc = 0, iPo, iOut;
    if constexpr (Store<T, ST>::phi_plane) {   // roles rotate with period 3 (see the context API)
        iPc = (3 - (int)(step % 3)) % 3;
        iPo = (iPc + 1) % 3;
        iOut = (iPc + 2) % 3;
        p.phi_cur = G->phi[iPc];
    } else {
        iPo = cur;
        iOut = 1 - cur;
        p.phi_cur = nullptr;
    }
    p.phi_old = G->phi[iPo];
    p.phi_out = G->phi[iOut];
}

// Step `ofs` of the group: CTAs stride over the work list (grid, strip, first row, rows).
// (The descriptors are read with ordinary loads, not __restrict__: this kernel may be resident while
// the kernel ahead of it still writes them, and only a load that the wait orders sees the new counters.)
template <typename V, typename ST, int FLUX>
__global__ void __launch_bounds__(32, (sizeof(V) == 4 ? 12 : 8))
batch_march_kernel(const __grid_constant__ BatchUniform<typename Lane<V>::T> u,
                   const __grid_constant__ MarchCoefs<typename Lane<V>::T> cf,
                   const BatchGrid<typename Lane<V>::T> *grids, const int4 *items, int nitems, int ofs) {
    using T = typename Lane<V>::T;
    extern __shared__ __align__(128) unsigned char smem[];
    pdl_wait();   // the previous step's output, or the advanced descriptors
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const int4 w = items[it];
        const BatchGrid<T> *G = grids + w.x;
        if (G->step + ofs >= G->target) continue;   // frozen grid
        StepParams<T> p;
        FastExtra<T> fe;
        batch_step_params<T, ST>(u, G, ofs, p, fe);
        march_strip<V, ST, FLUX, false, KIND_T2, SUM_CHECK>(p, cf, fe, w.y, w.z, w.w, nullptr, smem);
        __syncwarp();   // the next strip's copies overwrite the ring
    }
    pdl_trigger();
}

// After a group of `n` steps (n = 0: after an upload of the descriptors): the step counters, and
// the reversal factors of the vortex for the next group. FP64 is slow on this chip and its cost
// does not fall with idle lanes: one lane a factor.
template <typename T>
__global__ void __launch_bounds__(32) batch_advance_kernel(BatchGrid<T> *grids, int n, double dt) {
    pdl_wait();
    BatchGrid<T> *G = grids + blockIdx.x;
    const long long step = n > 0 && G->step < G->target ? min(G->step + n, G->target) : G->step;
    __syncwarp();
    if (threadIdx.x == 0) G->step = step;
    if (G->vel_kind == VEL_VORTEX && threadIdx.x < 3 * GRAPH_STEPS) {
        const int i = threadIdx.x / 3, q = threadIdx.x - 3 * i;
        const double t = (double)(step + i) * dt;
        G->vc[i][q] = (T)cospi((q == 0 ? t : q == 1 ? t - dt : t + 0.5 * dt) / G->vp[2]);
    }
    pdl_trigger();
}

}  // namespace dugks
