// dugks_dvm.cuh -- the streaming-collision discrete velocity method (DVM) of
// Sec. II.B.1 on the GPU, and at C = 1 the lattice Boltzmann method.
//
// State: tilde f^+_k = f_k + (dt/2)(Omega_k + S_k) at the cell centres (Eq. (9)),
// 9 planes in the ghost-bordered layout, and phi of the state as a plane. One
// fused kernel per step, one CTA per 32 x 8 tile:
//   pass 1  streaming, Eq. (11a): tilde f'_k(x_c) = tilde f^+_k(x_c - xi_k dt), the
//           value at the back-traced point from the Taylor expansion of Eq. (12)
//           (value + d.grad + d d : H / 2 (+ d d d : T / 6 at order 4), the
//           isotropic stencils of the DUGKS path) about the centre x_n = x_c - s xi_k
//           of the cell that holds it (s = 1 for dt >= 1/2, else 0), so
//           d = xi_k (s - dt); phi(t + dt) = sum_k tilde f'_k (Eq. (13)) on the tile
//           plus the ring the gradient of phi needs. At dt = 1 the back-traced
//           point is the neighbour's centre: plain streaming, the LBM.
//   pass 2  cell quantities at t + dt from the new phi (Eqs. (2), (4), (14): n,
//           theta, d(phi u)/dt by the backward difference from t, f^eq, S) and the
//           collision of Eq. (11b): tilde f^+ = tilde f' + 2 dt/(2 tau + dt)
//           (f^eq + tau S - tilde f') for the moving directions, the rest direction
//           closing the moment phi(t + dt) (equal to Eq. (11b) up to rounding); the
//           new state, phi and an FP64 mass partial per tile are written.
// The state tile (halo 2R + 1: the phi ring, the shift, the Taylor stencil; R + 1
// for the LBM) is read with plain coalesced loads; the ghost border makes it one
// rectangle. That kernel serves order 4; orders 2 and 3 (stencils of radius 1) march
// up the rows of a strip as the DUGKS step does (dugks_march.cuh), see dvm_strip.
#pragma once

#include "dugks_march.cuh"

namespace dugks {

// Per-run constants of the DVM step.
template <typename T>
struct DvmExtra {
    T d;      // displacement of the back-traced point from x_n per unit lattice velocity: s - dt
    T beta;   // collision factor 2 dt / (2 tau + dt)
    int s;    // shift of the expansion cell: x_n = x_c - s xi_k
    int early;   // row march: dependents may be scheduled at once
};

// (order 4)
template <typename T, bool LBM>
struct DvmTile {
    static constexpr int TX = 32, TY = 8, NT = TX * TY;
    static constexpr int R = 2;                           // stencil radius
    static constexpr int HS = LBM ? R + 1 : 2 * R + 1;    // state halo
    static constexpr int SW = TX + 2 * HS, SH = TY + 2 * HS;
    static constexpr int PW = TX + 2 * R, PH = TY + 2 * R;   // phi(t + dt) region
    static constexpr int RING = PW * PH - TX * TY;
    static constexpr size_t oP = sizeof(T) * 9 * SW * SH;
    static constexpr size_t oRed = (oP + sizeof(T) * PW * PH + 15) / 16 * 16;
    static constexpr size_t smem_bytes = oRed + sizeof(double) * 32;
    static_assert(HS <= GHOST, "the halo fits the ghost border");
    static_assert(RING <= NT, "one ring cell per thread");
};

template <typename T, bool LBM>
__global__ void __launch_bounds__(256) dvm_step_kernel(const StepParams<T> p, const DvmExtra<T> dv) {
    using DT = DvmTile<T, LBM>;
    constexpr int TX = DT::TX, TY = DT::TY, HS = DT::HS, SW = DT::SW, SH = DT::SH, R = DT::R;
    constexpr int PW = DT::PW, PH = DT::PH;
    extern __shared__ __align__(128) unsigned char smem[];
    T *sF = reinterpret_cast<T *>(smem);
    T *sP = reinterpret_cast<T *>(smem + DT::oP);
    double *sred = reinterpret_cast<double *>(smem + DT::oRed);
    const int tid = threadIdx.x, x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int nx = p.nx, ny = p.ny;

    // the state tile with its halo (cells beyond the ghost border, needed by no
    // cell of the grid, are clamped to it)
    const T *X = static_cast<const T *>(p.X);
    for (int i = tid; i < 9 * SW * SH; i += DT::NT) {
        const int k = i / (SW * SH), r = i - k * (SW * SH), yy = r / SW, xx = r - yy * SW;
        const int gx = min(x0 + xx - HS, nx + GHOST - 1), gy = min(y0 + yy - HS, ny + GHOST - 1);
        sF[i] = X[k * p.plane + gidx(p, gx, gy)];
    }
    __syncthreads();

    // pass 1: streaming of cell (x, y) of the tile frame (Eqs. (11a), (12)), phi(t + dt)
    auto stream = [&](int x, int y, T (&fs)[9]) -> T {
        T phi = T(0);
#pragma unroll
        for (int k = 0; k < 9; k++) {
            const T *F = sF + k * SW * SH;
            if constexpr (LBM) {
                fs[k] = F[(y - ey(k) + HS) * SW + (x - ex(k) + HS)];
            } else {
                const int xn = x - dv.s * ex(k), yn = y - dv.s * ey(k);
                fs[k] = taylor<T, 4>(F + (yn + HS) * SW + (xn + HS), SW, dv.d * T(ex(k)), dv.d * T(ey(k)));
            }
            phi += fs[k];   // Eq. (13), the unweighted sum
        }
        return phi;
    };
    const int tx = tid & 31, ty = tid >> 5;
    T fs[9];
    sP[(ty + R) * PW + (tx + R)] = stream(tx, ty, fs);
    if (tid < DT::RING) {   // the ring of the phi region: rows above and below, then the side columns
        int rx, ry;
        if (tid < 2 * R * PW) {
            const int band = tid / PW;
            ry = band < R ? band - R : TY + band - R;
            rx = tid - band * PW - R;
        } else {
            const int e = tid - 2 * R * PW, col = e / TY;
            rx = col < R ? col - R : TX + col - R;
            ry = e - col * TY;
        }
        T tmp[9];
        sP[(ry + R) * PW + (rx + R)] = stream(rx, ry, tmp);
    }
    __syncthreads();

    // pass 2: cell quantities at t + dt and the collision (Eqs. (2), (4), (14), (11b))
    const int gx = x0 + tx, gy = y0 + ty;
    double msum = 0.0;
    if (gx < nx && gy < ny) {
        const T *P = sP + (ty + R) * PW + (tx + R);
        const T ph = P[0];
        T gxp, gyp;
        grad_p<T, 4>(P, PW, gxp, gyp);
        const T g2 = gxp * gxp + gyp * gyp;
        T nxv = T(0), nyv = T(0);
        if (g2 > T(1e-24)) {
            const T inv = T(1) / sqrt(g2);
            nxv = gxp * inv;
            nyv = gyp * inv;
        }
        const T theta = p.theta_c * (ph - p.phiA) * (ph - p.phiB);
        T u, v;
        vel_cell(p, gx, gy, p.t, u, v);   // at t + dt
        T Dx = T(0), Dy = T(0);
        const size_t g = gidx(p, gx, gy);
        if (p.useD) {   // d(phi u)/dt between t and t + dt
            T uo, vo;
            vel_cell(p, gx, gy, p.t_old, uo, vo);
            const T po = p.phi_old[g];
            Dx = (ph * u - po * uo) * p.inv_dtD;
            Dy = (ph * v - po * vo) * p.inv_dtD;
        }
        const T Vx = theta * nxv + T(3) * Dx, Vy = theta * nyv + T(3) * Dy;
        T *O = static_cast<T *>(p.out1);
        // the rest component closes the sum (sum_k f^eq_k = phi, sum_k S_k = 0): the state
        // keeps the moment phi(t + dt) up to one rounding, as the DUGKS kernels do
        T rest = ph;
#pragma unroll
        for (int k = 1; k < 9; k++) {
            const T xu = T(ex(k)) * u + T(ey(k)) * v, xv = T(ex(k)) * Vx + T(ey(k)) * Vy;
            const T gk = wq<T>(k) * (ph * (T(1) + T(3) * xu) + p.tau * xv);   // f^eq + tau S
            const T o = fs[k] + dv.beta * (gk - fs[k]);
            rest -= o;
            put_cell(p, O + k * p.plane, gx, gy, o);
        }
        put_cell(p, O, gx, gy, rest);
        p.phi_out[g] = ph;
        msum = (double)ph;
    }
    const double s = block_sum(msum, sred);
    if (tid == 0 && p.mass_partial) p.mass_partial[blockIdx.y * p.tiles_x + blockIdx.x] = s;
}

// ---- orders 2 and 3 as a row march ---------------------------------------------
// A row j that arrives completes the expansions of row j - 1 (Eq. (12); the row terms of
// March<V, 0>, one expansion a direction). With the shift (MODE 1) the value expanded at
// cell c is tilde f'_k of cell c + xi_k: a shuffle over columns, and rows j - 2, j - 1, j for
// xi_y = -1, 0, 1, so that row j - 2 of tilde f' and of phi(t + dt) is then complete, and row j - 3
// has its gradient and is written. Without it (MODE 0) row j - 1 is complete; at dt = 1 (MODE 2, the
// LBM) the rows themselves are shifted. Bound by a row's latency in one wave of warps, then by instruction
// issue; measured in FP32, order 3, dt = 0.8, a step, against the tile kernel that it replaced (every tap read from
// shared memory, sines and cosines for every cell): 128^2 5.0 us, 14.4 before; 512^2 11.8, 30.1; 1024^2 25.1, 96.3;
// LBM 1024^2 18.8, 72.8.
template <typename V>
struct DvmMarch {
    using T = typename Lane<V>::T;
    static constexpr int N = Lane<V>::N;
    // columns written: lanes 2 to 29 of pairs, 3 to 28 of single columns
    static constexpr int TX = N == 2 ? 56 : 26, HX = N == 2 ? 5 : 3, LO = N == 2 ? 2 : 3, HI = 31 - LO;
    static constexpr int DEPTH = 3, LB = N * (int)sizeof(T);
    static constexpr int slot = 10 * 32 * LB;   // the state and phi_old of the row that it completes
    static constexpr int oRow = DEPTH * slot;
    static constexpr int strips(int nx) { return (nx + (N == 2 ? 1 : 0) + TX - 1) / TX; }
    static constexpr int smem_bytes(int rows) { return oRow + (rows + 6) * (int)sizeof(Row4<T>); }
};

template <typename V, int MODE, bool MASS>
__device__ __forceinline__ void dvm_strip(const StepParams<typename Lane<V>::T> &p, const DvmExtra<typename Lane<V>::T> &dv,
                                          const MarchCoefs<typename Lane<V>::T> &cf,
                                          const FastExtra<typename Lane<V>::T> &fe, int bx, int y0, int rows,
                                          double *mass_out, unsigned char *smem) {
    using T = typename Lane<V>::T;
    using LN = Lane<V>;
    using DM = DvmMarch<V>;
    constexpr int N = LN::N, LB = DM::LB;
    constexpr int LAG = MODE == 1 ? 3 : 2;   // row j completes row j - LAG
    const int lane = threadIdx.x & 31, nx = p.nx, ny = p.ny;
    const int x = DM::TX * bx - DM::HX + N * lane;
    const int col = min(x + GHOST, p.pitch - N);
    const bool wr = lane >= DM::LO && lane <= DM::HI;
    const bool ok0 = wr && x >= 0 && x < nx, ok1 = N == 2 && wr && x + 1 >= 0 && x + 1 < nx;
    const int first = y0 - LAG, npk = rows + 2 * LAG;

    // velocity factors (dugks_march.cuh) at the cell centres, at t + dt (rows y, sRow.x, .y)
    Row4<T> *sRow = reinterpret_cast<Row4<T> *>(smem + DM::oRow);
    const bool reversing = p.vel_kind == VEL_VORTEX || p.vel_kind == VEL_DEFORM;
    const T vct = reversing ? fe.vc_t : T(1), vco = reversing ? fe.vc_told : T(1);
    V cu{}, cv{};
    const bool field = p.vel_kind == VEL_FIELD;
    if (!field) {
        T a0, b0, a1 = T(0), b1 = T(0);
        vel_column(p, T(wrap_small(x, nx)) + T(0.5), a0, b0);
        if (N == 2) vel_column(p, T(wrap_small(x + 1, nx)) + T(0.5), a1, b1);
        cu = LN::make(a0, a1);
        cv = LN::make(b0, b1);
        for (int i = lane; i < rows; i += 32) {
            Row4<T> r{};
            vel_row(p, T(y0 + i) + T(0.5), r.x, r.y);
            sRow[i] = r;
        }
    }
    pdl_wait();

    // packet i: the state of row first + i and phi_old of the row that it completes
    const uint32_t ring = smem_u32(smem);
    const size_t plane = p.plane;
    const T *gX = static_cast<const T *>(p.X) + (size_t)(first + GHOST) * p.pitch + col;
    const T *gPo = p.phi_old + (size_t)(y0 + GHOST) * p.pitch + col;   // from row y0 on
    int fetched = 0;
    uint32_t fslot = 0;
    auto fetch = [&]() {
        if (fetched < npk) {
            const uint32_t s = ring + fslot + lane * LB;
#pragma unroll
            for (int k = 0; k < 9; k++) cp_async<LB>(s + k * 32 * LB, gX + k * plane);
            if (fetched >= 2 * LAG) {
                cp_async<LB>(s + 9 * 32 * LB, gPo);
                gPo += p.pitch;
            }
            gX += p.pitch;
            fetched++;
            fslot = fslot + DM::slot == DM::DEPTH * DM::slot ? 0 : fslot + DM::slot;
        }
        cp_commit();
    };
#pragma unroll
    for (int i = 0; i < DM::DEPTH - 1; i++) fetch();

    // pending expansions (as in March<V, 0>)
    struct Diag { V a, b, c; } g2{}, g4{}, g6{}, g8{};
    V z1{}, q1{}, z5{}, q5{}, z3{}, m3{}, d3{}, z7{}, m7{}, d7{};
    // rows in flight: north-going values of the two rows before, rest and axial ones
    V n2{}, n3{}, n4{}, o2{}, o3{}, o4{}, c0{}, c1{}, c5{}, d0{};
    V f1{}, f2{}, f3{}, f4{}, f5{}, f6{}, f7{}, f8{};   // tilde f' of the row that is written next
    V pc1{}, pd1{}, pm1{}, pm0{}, pz{};                 // phi(t + dt): that row, and its gradient
    const T vD = p.useD ? T(3) * p.inv_dtD * vct : T(0), vDo = p.useD ? T(-3) * p.inv_dtD * vco : T(0);
    const T v3 = T(3) * vct;
    double msum = 0.0;
    uint32_t cslot = 0;
    const bool xedge = x < GHOST || x + N - 1 >= nx - GHOST;
    // the value one column to the left / right (towards which xi_x points away)
    auto from_left = [&](V c) -> V {
        if constexpr (N == 2) return LN::make(__shfl_up_sync(ALL, LN::second(c), 1), LN::first(c));
        else return __shfl_up_sync(ALL, c, 1);
    };
    auto from_right = [&](V c) -> V {
        if constexpr (N == 2) return LN::make(LN::second(c), __shfl_down_sync(ALL, LN::first(c), 1));
        else return __shfl_down_sync(ALL, c, 1);
    };
    const T *gU = field ? p.ufield + (size_t)(y0 + GHOST) * p.pitch + col : nullptr;
    const T *gW = field ? p.vfield + (size_t)(y0 + GHOST) * p.pitch + col : nullptr;

#pragma unroll 1
    for (int it = 0; it < npk; it++) {
        cp_wait<1>();
        __syncwarp();
        fetch();
        const unsigned char *sl = smem + cslot + lane * LB;
        cslot = cslot + DM::slot == DM::DEPTH * DM::slot ? 0 : cslot + DM::slot;
        auto state = [&](int k) -> V { return *reinterpret_cast<const V *>(sl + k * 32 * LB); };

        // ---- pass 1: tilde f' and phi(t + dt) of the newly complete row ----------------
        V t[9];
        if constexpr (MODE == 2) {   // rows j (south-going), j - 1, j - 2 (north-going)
            t[0] = c0;
            t[1] = from_left(c1);
            t[5] = from_right(c5);
            t[2] = from_left(o2);
            t[3] = o3;
            t[4] = from_right(o4);
            o2 = n2; o3 = n3; o4 = n4;
            c0 = state(0);
            c1 = state(1);
            c5 = state(5);
            n2 = state(2);
            n3 = state(3);
            n4 = state(4);
            t[6] = from_right(state(6));
            t[7] = state(7);
            t[8] = from_left(state(8));
        } else {
            V e[9];   // expansions of row j - 1
            // Expansions are written in differences of cells, so that they sum to the same mass whatever
            // the weights' rounding: rows of a diagonal as W (C(r) - C(0)) + w1 (R - 2 C + L) + w2 (R - L)
            auto diag = [&](V C, auto sx, auto sy, Diag &g) -> V {
                constexpr int SX = decltype(sx)::value, SY = decltype(sy)::value;
                const Sides<V> q = vsides(C);
                const V e = vfma(T(-2), C, q.s), up = vsub(C, g.c);
                auto row = [&](int r, V acc) { return vfma(T(SX) * cf.dx[r][2], q.d, vfma(cf.dx[r][1], e, acc)); };
                const V out = row(1 + SY, vfma(cf.dx[1 + SY][0], up, g.a));
                g.a = row(1, vadd(vfma(-cf.dx[1 - SY][0], up, C), g.b));
                g.b = vfma(T(SX) * cf.dx[1 - SY][2], q.d, vmul(cf.dx[1 - SY][1], e));
                g.c = C;
                return out;
            };
            using P1 = std::integral_constant<int, 1>;
            using M1 = std::integral_constant<int, -1>;
            e[2] = diag(state(2), P1{}, P1{}, g2);
            e[4] = diag(state(4), M1{}, P1{}, g4);
            e[6] = diag(state(6), M1{}, M1{}, g6);
            e[8] = diag(state(8), P1{}, M1{}, g8);
            V C = state(1);
            Sides<V> q = vsides(C);
            V w = vfma(cf.px, q.d, vmul(cf.pe, vfma(T(-2), C, q.s)));
            e[1] = vadd(z1, w);
            z1 = vadd(vfma(T(4), w, C), q1);
            q1 = w;
            C = state(5);
            q = vsides(C);
            w = vfma(-cf.px, q.d, vmul(cf.pe, vfma(T(-2), C, q.s)));
            e[5] = vadd(z5, w);
            z5 = vadd(vfma(T(4), w, C), q5);
            q5 = w;
            C = state(3);
            w = vfma(T(4), C, vsides(C).s);
            // value + nu (m(+) - m(-)) + nm (m(+) - 2 m(0) + m(-)), m = L + 4 C + R
            V up = vsub(w, m3);
            e[3] = vfma(cf.nu, vadd(up, d3), vfma(cf.nm, vsub(up, d3), z3));
            z3 = C;
            m3 = w;
            d3 = up;
            C = state(7);
            w = vfma(T(4), C, vsides(C).s);
            up = vsub(w, m7);
            e[7] = vfma(-cf.nu, vadd(up, d7), vfma(cf.nm, vsub(up, d7), z7));
            z7 = C;
            m7 = w;
            d7 = up;
            if constexpr (MODE == 0) {
                t[0] = c0;
                c0 = state(0);
#pragma unroll
                for (int k = 1; k < 9; k++) t[k] = e[k];
            } else {
                t[0] = d0;
                d0 = c0;
                c0 = state(0);
                t[1] = c1;
                t[5] = c5;
                c1 = from_left(e[1]);
                c5 = from_right(e[5]);
                t[2] = o2;
                t[3] = o3;
                t[4] = o4;
                o2 = n2; o3 = n3; o4 = n4;
                n2 = from_left(e[2]);
                n3 = e[3];
                n4 = from_right(e[4]);
                t[6] = from_right(e[6]);
                t[7] = e[7];
                t[8] = from_left(e[8]);
            }
        }
        // Eq. (13), the unweighted sum
        const V pc0 = vadd(vadd(vadd(vadd(t[0], t[1]), vadd(t[2], t[3])), vadd(vadd(t[4], t[5]), vadd(t[6], t[7]))), t[8]);
        const Sides<V> ps = vsides(pc0);
        const V pmn = vfma(T(4), pc0, ps.s);
        const V gx = vadd(pz, ps.d), gy = vsub(pmn, pm0);   // 12 grad phi of row j - LAG
        pz = vfma(T(4), ps.d, pd1);
        pd1 = ps.d;
        pm0 = pm1;
        pm1 = pmn;

        // ---- pass 2: cell quantities at t + dt and the collision of row j - LAG ----------
        const V ph = pc1;
        const V h1 = f1, h2 = f2, h3 = f3, h4 = f4, h5 = f5, h6 = f6, h7 = f7, h8 = f8;
        f1 = t[1]; f2 = t[2]; f3 = t[3]; f4 = t[4]; f5 = t[5]; f6 = t[6]; f7 = t[7]; f8 = t[8];
        pc1 = pc0;
        if (it < 2 * LAG) continue;
        const int i = it - 2 * LAG, y = y0 + i;
        V us, vs;
        if (field) {
            us = *reinterpret_cast<const V *>(gU + (size_t)i * p.pitch);
            vs = *reinterpret_cast<const V *>(gW + (size_t)i * p.pitch);
        } else {
            const Row4<T> rf = sRow[i];
            us = vmul(rf.x, cu);
            vs = vmul(rf.y, cv);
        }
        V inv = vnorm(vfma(gx, gx, vmul(gy, gy)), T(144e-24));
        inv = vmul(inv, vmul(vmul(p.theta_c, vadd(ph, -p.phiA)), vadd(ph, -p.phiB)));
        const V po = *reinterpret_cast<const V *>(sl + 9 * 32 * LB);
        const V w = vfma(vD, ph, vmul(vDo, po));   // 3 d(phi u)/dt without u's spatial part
        const V Vx = vfma(gx, inv, vmul(us, w)), Vy = vfma(gy, inv, vmul(vs, w));
        const V p3 = vmul(v3, ph);
        const V Px = vfma(us, p3, vmul(p.tau, Vx)), Py = vfma(vs, p3, vmul(p.tau, Vy));   // f^eq + tau S = w (phi + xi . P)
        V o[9];
        auto collide = [&](int k, V f, V g) { o[k] = vfma(dv.beta, vfma(wq<T>(k), g, vneg(f)), f); };
        const V gp = vadd(ph, Px), gm = vsub(ph, Px);
        collide(1, h1, gp);
        collide(2, h2, vadd(gp, Py));
        collide(3, h3, vadd(ph, Py));
        collide(4, h4, vadd(gm, Py));
        collide(5, h5, gm);
        collide(6, h6, vsub(gm, Py));
        collide(7, h7, vsub(ph, Py));
        collide(8, h8, vsub(gp, Py));
        // the rest component closes the sum (sum_k f^eq_k = phi, sum_k S_k = 0): the state
        // keeps the moment phi(t + dt) up to one rounding, as the DUGKS kernels do
        o[0] = vsub(ph, vadd(vadd(vadd(o[1], o[2]), vadd(o[3], o[4])), vadd(vadd(o[5], o[6]), vadd(o[7], o[8]))));
        T *O = static_cast<T *>(p.out1);
        auto put0 = [&](long long g) {
#pragma unroll
            for (int k = 0; k < 9; k++) O[(long long)(k * plane) + g] = LN::first(o[k]);
        };
        auto put1 = [&](long long g) {
#pragma unroll
            for (int k = 0; k < 9; k++) O[(long long)(k * plane) + g + 1] = LN::second(o[k]);
        };
        const size_t g = (size_t)(y + GHOST) * p.pitch + (size_t)(x + GHOST);
        if (ok0 && (N == 1 || ok1)) {
#pragma unroll
            for (int k = 0; k < 9; k++) *reinterpret_cast<V *>(O + k * plane + g) = o[k];
            *reinterpret_cast<V *>(p.phi_out + g) = ph;
        } else if (ok0) {
            put0(g);
            p.phi_out[g] = LN::first(ph);
        } else if (ok1) {
            put1(g);
            p.phi_out[g + 1] = LN::second(ph);
        }
        if constexpr (MASS) {
            if (ok0) msum += (double)LN::first(ph);
            if (ok1) msum += (double)LN::second(ph);
        }
        // periodic images in the ghost border
        if ((ok0 || ok1) && (xedge || y < GHOST || y >= ny - GHOST)) {
#pragma unroll 1
            for (int im = 0; im < 9; im++) {
                const int ay = im / 3 - 1, ax = im - 3 * (im / 3) - 1;
                const int yy = y + ay * ny, xx = x + ax * nx;
                if (im == 4 || yy < -GHOST || yy >= ny + GHOST) continue;
                const long long gi = (long long)(yy + GHOST) * p.pitch + (xx + GHOST);
                if (ok0 && xx >= -GHOST && xx < nx + GHOST) put0(gi);
                if (ok1 && xx + 1 >= -GHOST && xx + 1 < nx + GHOST) put1(gi);
            }
        }
    }
    cp_wait<0>();
    if constexpr (MASS) {
        for (int o = 16; o > 0; o >>= 1) msum += __shfl_down_sync(ALL, msum, o);
        if (lane == 0) *mass_out = msum;
    }
}

template <typename V, int MODE, bool MASS>
__global__ void __launch_bounds__(32, (sizeof(V) == 4 ? 16 : 8))
dvm_march_kernel(const __grid_constant__ StepParams<typename Lane<V>::T> p,
                 const __grid_constant__ DvmExtra<typename Lane<V>::T> dv,
                 const __grid_constant__ MarchCoefs<typename Lane<V>::T> cf,
                 const __grid_constant__ FastExtra<typename Lane<V>::T> fe) {
    extern __shared__ __align__(128) unsigned char smem[];
    if (dv.early) pdl_trigger();
    const int y0 = blockIdx.y * p.tile_h;
    dvm_strip<V, MODE, MASS>(p, dv, cf, fe, blockIdx.x, y0, min(p.tile_h, p.ny - y0),
                             MASS ? p.mass_partial + blockIdx.y * p.tiles_x + blockIdx.x : nullptr, smem);
    if (!dv.early) pdl_trigger();
}

}  // namespace dugks
