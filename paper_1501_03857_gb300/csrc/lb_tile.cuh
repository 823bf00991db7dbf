// The tiled form of the fused step (the other is lb_march.cuh): for domains
// too small to keep the GPU busy, where a step lasts as long as one block's
// chain of dependent work.
//
// A block computes one tile of NW * K rows x 64 columns, 5 of them on each
// side halo, all stages at once: five barriers per tile instead of five per
// two rows. Warp w owns K consecutive rows of all 64 columns: lane l holds
// columns l and l + 32 in one float2, so a row's conditions are the warp's
// and the paired instructions need no repacking. What a thread's own cells
// need again (populations, rho, theta, RK coefficients and sums) stays in
// its registers; the fields whose neighbours are read (psi, rho, v, theta and
// the RK stage inputs, which reuse the first three) are shared rows of 34
// float2: slot -1 and 32 repeat the other half's edge column, written by
// lanes 31 and 0.
//
// The first rows and columns out are recomputed by every tile that needs
// them (7.1 cells computed per cell written at 12 rows, 4.1 at 14, 3.2 at 16,
// 2.0 at 24), which an idle GPU has to spare. A tile's time is its warps' work
// on one SM plus the chain of stages, so on a domain that leaves SMs empty
// smaller tiles are faster while they still come to one wave: a step of
// 100 x 100 takes 4.25 us with 12 one-row warps (100 blocks), 4.6 with 14
// (50), 4.9 with 16 (34), 6.5 with 12 two-row warps (16), and 15.2 us
// marching; 300 x 100 takes 7.3 us with 12 (300 blocks, two waves), 4.8 with
// 14 (150) and 5.0 with 16; 600 x 150 6.7 us with 24 rows (132 blocks), 8.4
// us with 16 (300), 17.6 us marching. From about 500 x 1000 on marching is
// faster (24.8 against 28.3 us).
#pragma once

#include "lb_common.cuh"

namespace lbgpu {

namespace {

constexpr int TILE_OUT = TILE_W - 2 * HALO;  // columns it writes

template <int NW, int K>
struct TileShape {
    static constexpr int rows = NW * K;                  // rows a tile computes
    static constexpr int out = rows - 2 * HALO;          // rows it writes
    static constexpr int field = (rows + 2) * TILE_ROW;  // float2 per shared field
    static constexpr int slots = 5 * field;
};

// Output rows [ys, ye) and columns [x0, x0 + nv) of the step.
template <int NW, int K, bool REC, bool OUT, bool QF>
__device__ __forceinline__ void tile_rows(const StepParams& P, const StepParams& C, int x0, int nv, int ys, int ye,
                                          const RecomputeOut* R, float2* sm, bool& eos_bad, bool& nonfinite) {
    using Sh = TileShape<NW, K>;
    const int Lx = P.Lx, Ly = P.Ly;
    const int lane = threadIdx.x & 31, j0 = (threadIdx.x >> 5) * K;
    const bool periodic = P.bc == BC_PERIODIC;
    const bool thermal = !P.isothermal;
    Cols c;
    {
        const int xs = x0 - HALO + lane;
        c.a = wrap(xs, Lx);
        c.b = wrap(xs + 32, Lx);
        c.am = c.a == 0 ? Lx - 1 : c.a - 1;
        c.ap = c.a == Lx - 1 ? 0 : c.a + 1;
        c.bm = c.b == 0 ? Lx - 1 : c.b - 1;
        c.bp = c.b == Lx - 1 ? 0 : c.b + 1;
    }
    const bool outa = lane >= HALO && lane < HALO + nv;
    const bool outb = lane + 32 < TILE_W - HALO && lane + 32 < HALO + nv;
    const int r0 = ys - HALO + j0;  // this thread's first row
    auto in = [&](int d, int r) {  // rows [ys - d, ye + d) of the domain
        if (periodic) return r >= ys - d && r < ye + d;
        return r >= max(ys - d, 0) && r < min(ye + d, Ly);
    };
    // whether any of the warp's rows is needed at distance d from the tile's
    // output rows; a warp works on all its rows or none (values of rows and
    // columns further out are never read by those that count)
    auto any = [&](int d) {
        if (periodic) return r0 + K > ys - d && r0 < ye + d;
        return r0 + K > max(ys - d, 0) && r0 < min(ye + d, Ly);
    };
    auto phys = [&](int r) { return periodic ? wrap_row(r, Ly) : min(max(r, 0), Ly - 1); };
    auto interior = [&](int r) { return periodic || (r > 0 && r < Ly - 1); };
    float2* const own = sm + (j0 + 1) * TILE_ROW + 1 + lane;
    enum { PSI = 0, RHO = 1, VX = 2, VY = 3, TH = 4, U2 = PSI, U3 = RHO, U4 = VX };
    const int edge = lane == 0 || lane == 31;
    // the other half's edge slot, in floats from this thread's own: lane 0's
    // upper column is column 32 (slot 32's lower half), lane 31's lower column
    // 31 (slot -1's upper half)
    const int eo = lane == 0 ? 64 : -63;
    auto at = [&](float2* q) { return smem_at(q, -lane - 1, 32 - lane, sm, Sh::slots, P.acc); };
    auto put = [&](int F, int k, P2 v) {
        float2* q = at(own + F * Sh::field + k * TILE_ROW);
        *q = v.f2();
        if (edge) reinterpret_cast<float*>(q)[eo] = lane == 0 ? v.y() : v.x();
    };
    auto row = [&](int F, int k) {
        const float2* q = at(own + F * Sh::field + k * TILE_ROW);
        return Row3{P2(q[-1]), P2(q[0]), P2(q[1])};
    };
    auto save = [&](float* plane, int y, P2 v) {
        float* p = plane + y * P.pitch;
        lb_st_if(outa, p + c.a, v.x(), plane, (size_t)P.plane, P.acc);
        lb_st_if(outb, p + c.b, v.y(), plane, (size_t)P.plane, P.acc);
    };
    const P2 zero = P2::bc(0.f);

    // the warp that holds the bottom wall row needs theta_b at the end
    const bool bottom = !periodic && r0 <= 0 && r0 + K > 0;
    P2 thb = zero;
    if (OUT && bottom && thermal) thb = P2(lb_ldg(P.thb + c.a, P.thb, P.pitch, P.acc), lb_ldg(P.thb + c.b, P.thb, P.pitch, P.acc));
    // ---- P: pull, wall fill, rho, psi
    P2 f[K][9], rho[K], th[K];
    if (any(HALO)) {
#pragma unroll
        for (int k = 0; k < K; ++k) load_row2<false>(P, phys(r0 + k), c, f[k], th[k]);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int y = r0 + k;
            if (!periodic) {
                const P2 d = 0.5f * (f[k][1] - f[k][3]);
                const bool lo = y == 0, hi = P.bc == BC_WALLS && y == Ly - 1;
                // Zou-He walls, u = 0
                f[k][2] = sel(lo, f[k][4], f[k][2]);
                f[k][5] = sel(lo, f[k][7] - d, f[k][5]);
                f[k][6] = sel(lo, f[k][8] + d, f[k][6]);
                f[k][4] = sel(hi, f[k][2], f[k][4]);
                f[k][7] = sel(hi, f[k][5] + d, f[k][7]);
                f[k][8] = sel(hi, f[k][6] - d, f[k][8]);
            }
            rho[k] = ((f[k][0] + f[k][1]) + (f[k][2] + f[k][3])) + ((f[k][4] + f[k][5]) + (f[k][6] + f[k][7])) + f[k][8];
            bool bad = false;
            const P2 psi = eos_psi2(rho[k], th[k] + P2(C.kp[KP_TS]), C, bad);
            eos_bad |= bad && in(HALO, y);
            put(PSI, k, psi);
            put(RHO, k, rho[k]);
            put(TH, k, th[k]);
            if constexpr (REC) {
                if (in(0, y)) {
                    save(R->rho, phys(y), rho[k]);
                    save(R->psi, phys(y), psi);
                }
            }
        }
    }
    __syncthreads();

    // ---- bottom-wall heat flux of level t (Sec. 3.2), one term per column, by
    // a warp whose rows lie below the wall
    if (QF && !periodic && ys == 0 && threadIdx.x < 32) {
        float2* q0 = at(sm + (HALO + 1) * TILE_ROW + 1 + lane);  // row y = 0
        const float2 rw = q0[RHO * Sh::field];
        const float2 t0 = q0[TH * Sh::field], t1 = q0[TH * Sh::field + TILE_ROW], t2 = q0[TH * Sh::field + 2 * TILE_ROW];
        if (outa) lb_st(P.qpart + c.a, heat_term(rw.x, t0.x, t1.x, t2.x), P.qpart, P.Lx, P.acc);
        if (outb) lb_st(P.qpart + c.b, heat_term(rw.y, t0.y, t1.y, t2.y), P.qpart, P.Lx, P.acc);
    }

    // ---- B: forces and velocity
    P2 vx[K], vy[K], Fx[K], Fy[K], g2[K];
    if (any(4)) {
        Row3 m = row(PSI, -1), o = row(PSI, 0);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const Row3 p = row(PSI, k + 1);
            const int y = r0 + k;
            const bool wall = !periodic && (y == 0 || y == Ly - 1);
            const P2(&g)[9] = f[k];
            const P2 jx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
            const P2 jy = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
            Row3 ps = m, pn = p;
            if (!periodic) {  // the ghost layer beyond a wall copies the wall row
                ps = Row3{sel(y == 0, o.w, m.w), sel(y == 0, o.c, m.c), sel(y == 0, o.e, m.e)};
                pn = Row3{sel(y == Ly - 1, o.w, p.w), sel(y == Ly - 1, o.c, p.c), sel(y == Ly - 1, o.e, p.e)};
            }
            const St2 d = stencil2(ps, o, pn, false);  // 12 sum_a w_a psi(x + e_a) e_a, Eq. 7
            const P2 mG = P2(C.kp[KP_GN12]) * o.c;
            Fx[k] = mG * d.dx;
            Fy[k] = mG * d.dy;
            g2[k] = fma2(d.dx, d.dx, d.dy * d.dy);
            {
                const bool off = wall && !P.ghost;
                Fx[k] = sel(off, zero, Fx[k]);
                Fy[k] = sel(off, zero, Fy[k]);
                g2[k] = sel(off, zero, g2[k]);
                if (!periodic) Fy[k] = sel(y == 1, fma2(P2(P.kp[KP_GW6]), o.c * o.c, Fy[k]), Fy[k]);  // Eq. 22
            }
            const P2 Fb = fma2(P2(C.kp[KP_GN]), rho[k] - P2(P.kp[KP_RHOAVE]), Fy[k]);  // Eq. 9
            Fy[k] = sel(wall, Fy[k], Fb);
            const P2 irho = rcp2(rho[k]);
            vx[k] = fma2(P2::bc(0.5f), Fx[k], jx) * irho;  // Eq. 6
            vy[k] = fma2(P2::bc(0.5f), Fy[k], jy) * irho;
            put(VX, k, vx[k]);
            put(VY, k, vy[k]);
            m = o;
            o = p;
        }
    }
    __syncthreads();

    // ---- B: collision (nothing waits for it, so it follows the barrier)
    if (OUT && any(0)) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            if (K == 1 || in(0, r0 + k)) {
                P2 w[9];
                collide2(f[k], rho[k], vx[k], vy[k], Fx[k], Fy[k], g2[k], C, w);
                const int pl = P.plane;
                float* out = P.f_out + phys(r0 + k) * P.pitch;
                nonfinite |= (outa && !finite_f(rho[k].x())) || (outb && !finite_f(rho[k].y()));
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    lb_st_if(outa, out + (a * pl + c.a), w[a].x(), P.f_out, 9 * (size_t)pl, P.acc);
                    lb_st_if(outb, out + (a * pl + c.b), w[a].y(), P.f_out, 9 * (size_t)pl, P.acc);
                }
            }
        }
    }

    P2 acc[K];
    Coef2 co[K];
    if (thermal) {
        // ---- C: frozen-flow coefficients and RK stage 1
        if (any(3)) {
            Row3 rm = row(RHO, -1), ro = row(RHO, 0), xm = row(VX, -1), xo = row(VX, 0), ym = row(VY, -1), yo = row(VY, 0);
            Row3 tm = row(TH, -1), to = row(TH, 0);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const Row3 rp = row(RHO, k + 1), xp = row(VX, k + 1), yp = row(VY, k + 1), tp = row(TH, k + 1);
                const int y = r0 + k;
                const St2 gr = stencil2(rm, ro, rp, false);
                const St2 gvx = stencil2(xm, xo, xp, false);
                const St2 gvy = stencil2(ym, yo, yp, false);
                const P2 q = P2(C.kp[KP_CHI144]) * rcp2(gr.c);
                const P2 divv = gvx.dx + gvy.dy;  // 12 div v
                const P2 br = P2(C.kp[KP_B]) * gr.c;
                Coef2 kC;  // ax, ay divided by 12
                kC.ax = fma2(q, gr.dx, P2::bc(-1.f / 12.f) * gvx.c);
                kC.ay = fma2(q, gr.dy, P2::bc(-1.f / 12.f) * gvy.c);
                kC.cA = P2(C.kp[KP_RCV12]) * divv * rcp2(P2::bc(1.f) - br);
                kC.cB = P2(C.kp[KP_ACV12]) * (divv * gr.c) * rcp2(fma2(br, P2::bc(2.f) - br, P2::bc(1.f)));
                co[k] = kC;
                acc[k] = rhs_K2(stencil2(tm, to, tp, true), kC, C);
                const P2 u2 = sel(interior(y), fma2(P2::bc(0.5f), acc[k], th[k]), th[k]);
                put(U2, k, u2);
                if constexpr (REC) {
                    if (in(0, y)) {  // weighted gradients, unscaled coefficients
                        const int yy = phys(y);
                        const bool fl = interior(y);
                        const P2 w12 = P2::bc(1.f / 12.f), t12 = P2::bc(12.f);
                        save(R->drx, yy, sel(fl, w12 * gr.dx, zero));
                        save(R->dry, yy, sel(fl, w12 * gr.dy, zero));
                        save(R->divv, yy, sel(fl, w12 * divv, zero));
                        save(R->ax, yy, sel(fl, t12 * kC.ax, zero));
                        save(R->ay, yy, sel(fl, t12 * kC.ay, zero));
                        save(R->u2, yy, u2);
                    }
                }
                rm = ro;
                ro = rp;
                xm = xo;
                xo = xp;
                ym = yo;
                yo = yp;
                tm = to;
                to = tp;
            }
        }
        __syncthreads();
        // ---- D: RK stage 2
        if (any(2)) {
            Row3 m = row(U2, -1), o = row(U2, 0);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const Row3 p = row(U2, k + 1);
                const int y = r0 + k;
                const P2 h2 = rhs_K2(stencil2(m, o, p, true), co[k], C);
                P2 u3 = fma2(P2::bc(0.5f), h2, th[k]);
                u3 = sel(interior(y), u3, th[k]);
                acc[k] = fma2(P2::bc(2.f), h2, acc[k]);
                put(U3, k, u3);
                if constexpr (REC) {
                    if (in(0, y)) save(R->u3, phys(y), u3);
                }
                m = o;
                o = p;
            }
        }
        __syncthreads();
        // ---- E: RK stage 3
        if (any(1)) {
            Row3 m = row(U3, -1), o = row(U3, 0);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const Row3 p = row(U3, k + 1);
                const int y = r0 + k;
                const P2 h3 = rhs_K2(stencil2(m, o, p, true), co[k], C);
                P2 u4 = th[k] + h3;
                u4 = sel(interior(y), u4, th[k]);
                acc[k] = fma2(P2::bc(2.f), h3, acc[k]);
                put(U4, k, u4);
                if constexpr (REC) {
                    if (in(0, y)) save(R->u4, phys(y), u4);
                }
                m = o;
                o = p;
            }
        }
        __syncthreads();
    }
    // ---- F: RK stage 4, theta^{t+1}
    if (OUT && any(0)) {
        Row3 m, o;
        if (thermal) {
            m = row(U4, -1);
            o = row(U4, 0);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int y = r0 + k;
            P2 tnew = th[k];
            if (thermal) {
                const Row3 p = row(U4, k + 1);
                const P2 h4 = rhs_K2(stencil2(m, o, p, true), co[k], C);
                tnew = fma2(acc[k] + h4, P2::bc(1.f / 6.f), th[k]);
                if (!periodic) {
                    tnew = sel(y == 0, thb, tnew);
                    tnew = sel(y == Ly - 1, zero, tnew);
                }
                m = o;
                o = p;
            }
            if (K == 1 || in(0, y)) {
                float* out = P.th_out + phys(y) * P.pitch;
                nonfinite |= (outa && !finite_f(tnew.x())) || (outb && !finite_f(tnew.y()));
                lb_st_if(outa, out + c.a, tnew.x(), P.th_out, (size_t)P.plane, P.acc);
                lb_st_if(outb, out + c.b, tnew.y(), P.th_out, (size_t)P.plane, P.acc);
            }
        }
    }
}

// The whole step for block `block`: strip block % nstrips, and the rows of its
// segment (P.seg_h, normally one tile's). K = C supplies the model constants
// (see lb_step_batch.cu); fold: the previous step's q(t) is still to be folded.
template <int NW, int K, bool REC, bool OUT, bool QF>
__device__ __forceinline__ void tile_body(const StepParams& P, const StepParams& C, const int block, const int fold,
                                          const RecomputeOut* R) {
    extern __shared__ float2 sm2[];
    using Sh = TileShape<NW, K>;
    bool eos_bad = false, nonfinite = false;
    // by a warp that has no rows of its own in the tile above the bottom wall
    if (QF && fold && block == 0 && P.bc != BC_PERIODIC && threadIdx.x < 32) fold_heat(P, threadIdx.x);
    const int x0 = block % P.nstrips * TILE_OUT, seg = block / P.nstrips;
    const int nv = min(TILE_OUT, P.Lx - x0);
    const int s1 = min((seg + 1) * P.seg_h, P.Ly);
    for (int ys = seg * P.seg_h; ys < s1; ys += Sh::out) {
        if (ys > seg * P.seg_h) __syncthreads();
        tile_rows<NW, K, REC, OUT, QF>(P, C, x0, nv, ys, min(ys + Sh::out, s1), R, sm2, eos_bad, nonfinite);
    }
    if (eos_bad) atomicOr(&P.acc->err, ERR_EOS);
    if (nonfinite) atomicOr(&P.acc->err, ERR_NONFINITE);
}

}  // namespace

}  // namespace lbgpu
