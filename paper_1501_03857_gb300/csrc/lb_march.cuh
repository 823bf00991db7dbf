// The marching form of the fused step (the other is lb_tile.cuh): for domains
// that fill the GPU.
//
// A block of 64 threads owns two adjacent strips of 54 columns and a segment
// of rows, thread lc the column lc of both (5 halo columns per side), and
// marches up the segment two rows per iteration through a pipeline of stages,
// each one row behind the previous; every population and temperature value is
// read from HBM once and written once:
//
//   P  rows L, L+1     : wall fill, rho, psi(rho, T^t)        (Eqs. 3, 6, 21)
//   B  rows L-1, L     : F_m, F_ads, F_b, v, MRT collision, store f*  (Eqs. 2-9, 22);
//                        then the loads of rows L+2, L+3
//   C  rows L-2, L-1   : grad rho, div v, RK stage 1 of Eq. 18 (Eqs. 18-20)
//   D  rows L-3, L-2   : RK stage 2
//   E  rows L-4, L-3   : RK stage 3
//   F  rows L-5, L-4   : RK stage 4, store theta^{t+1}
//
// Every stage writes two rows of its field into one half of a four-row shared
// ring, and the next stage reads that half and the one before it: the four
// rows its two stencils need. Two rows per iteration share two thirds of the
// neighbour loads and the barriers, and their independent arithmetic fills
// each other's latencies. A thread reads its own column's values back from
// registers (carried from the iteration that made them), the RK coefficients
// of a row once for the two stages that follow each other on it.
//
// What bounds it: eight warps per SM (240 registers) keep the FP32 pipe 54 %
// and the shared-memory path 54 % busy, with fixed-latency waits as the first
// stall; twelve warps (168 registers) measure the same. On 4096^2: one row
// per iteration 351 us; two rows 325 us; square root and stores without
// branches, so that the two rows interleave, 320 us; own values from
// registers, 302 us (392 instructions per cell instead of 541, shared-load
// wavefronts 56 instead of 110 per cell-warp); coherent loads 306 us, between
// the collisions 298 us.
#pragma once

#include "lb_common.cuh"

namespace lbgpu {

namespace {

constexpr int MARCH_T = 64;                            // threads
constexpr int MARCH_COLS = 2 * (MARCH_T - 2 * HALO);  // columns a block writes

struct MarchSmem {
    static constexpr int MT = MARCH_T, MW = MT + 2;  // float2 slots of a ring row (one beyond each side)
    // four-row rings (two halves of two rows), theta with eight rows, and the
    // own-column RK coefficients (three halves), in float2
    enum { PSI = 0, RHO = 4 * MW, VX = 8 * MW, VY = 12 * MW, U2 = 16 * MW, U3 = 20 * MW, U4 = 24 * MW, TH = 28 * MW, CO = 36 * MW };
    static constexpr int HALF = 2 * MW;             // float2 of half a ring
    static constexpr int CHALF = 2 * 4 * MT;        // float2 of the coefficients of two rows
    static constexpr int total = CO + 3 * CHALF;
};

// The whole step for block `block`: column pair block % npair, segment of
// P.seg_h rows. C supplies the model constants (see lb_step_batch.cu); fold: the
// previous step's q(t) is still to be folded.
// EARLY: the next rows' loads between the collisions instead of after the
// stores: a load does not overtake a store that it might alias, so it waits
// where it stands. One domain: 4096^2 298 us instead of 306, 2048^2 86.4
// instead of 88.4, 517 x 1003 24.6 instead of 24.8. Not for batches: 48 uneven
// domains take 0.9 % longer with it, and in 168 registers it spills 200 bytes
// more.
template <bool REC, bool OUT, bool QF, bool EARLY>
__device__ __forceinline__ void march_body(const StepParams& P, const StepParams& C, const int block, const int fold,
                                           const RecomputeOut* R) {
    extern __shared__ float2 sm2[];
    using M = MarchSmem;
    constexpr int MT = M::MT, MW = M::MW, NO = MT - 2 * HALO;
    const int Lx = P.Lx, Ly = P.Ly;
    const int npair = (Lx + 2 * NO - 1) / (2 * NO);
    const int strip = block % npair, seg = block / npair;
    const int x0 = strip * 2 * NO;
    const int nva = min(NO, Lx - x0), nvb = min(NO, Lx - x0 - NO);
    const int lc = threadIdx.x;
    const bool periodic = P.bc == BC_PERIODIC;
    const bool thermal = !P.isothermal;
    Cols c;
    c.a = wrap(x0 - HALO + lc, Lx);
    c.b = wrap(x0 + NO - HALO + lc, Lx);
    c.am = c.a == 0 ? Lx - 1 : c.a - 1;
    c.ap = c.a == Lx - 1 ? 0 : c.a + 1;
    c.bm = c.b == 0 ? Lx - 1 : c.b - 1;
    c.bp = c.b == Lx - 1 ? 0 : c.b + 1;
    const bool outa = lc >= HALO && lc < HALO + nva;
    const bool outb = lc >= HALO && lc < HALO + nvb;
    const int ys = seg * P.seg_h, ye = min(ys + P.seg_h, Ly);
    bool eos_bad = false, nonfinite = false;

    auto at = [&](float2* q, int lo, int hi) { return smem_at(q, lo, hi, sm2, M::total, P.acc); };
    auto phys = [&](int r) { return periodic ? wrap_row(r, Ly) : min(max(r, 0), Ly - 1); };
    auto interior = [&](int r) { return periodic || (r > 0 && r < Ly - 1); };
    auto mine = [&](int r) { return r >= ys && r < ye; };
    auto save = [&](float* plane, int y, P2 v) {
        float* p = plane + y * P.pitch;
        lb_st_if(outa, p + c.a, v.x(), plane, (size_t)P.plane, P.acc);
        lb_st_if(outb, p + c.b, v.y(), plane, (size_t)P.plane, P.acc);
    };
    const P2 zero = P2::bc(0.f);

    // this thread's slot in the current and the previous half of the rings,
    // the four halves of theta, the three of the coefficients
    float2* bc = sm2 + 1 + lc;
    float2* bp = bc + M::HALF;
    float2 *t0 = sm2 + M::TH + 1 + lc, *t1 = t0 + M::HALF, *t2 = t1 + M::HALF, *t3 = t2 + M::HALF;
    float2 *k0 = sm2 + M::CO + lc, *k1 = k0 + M::CHALF, *k2 = k1 + M::CHALF;
    // a ring row's three columns around this one, the own from a register
    auto rowc = [&](float2* q0, P2 c) {
        const float2* q = at(q0, -1, 1);
        return Row3{P2(q[-1]), c, P2(q[1])};
    };
    auto row = [&](float2* q0) {
        const float2* q = at(q0, -1, 1);
        return Row3{P2(q[-1]), P2(q[0]), P2(q[1])};
    };
    auto own = [&](float2* q) { return P2(*at(q, 0, 0)); };
    auto put = [&](float2* q, P2 v) { *at(q, 0, 0) = v.f2(); };

    P2 fp[9], f0[9], f1[9], th0, th1;  // populations of rows L - 1, L, L + 1; theta of L, L + 1
    P2 rhop = zero;
    P2 accD0 = zero, accD1 = zero, accE = zero, accF0 = zero, accF1 = zero;
#pragma unroll
    for (int a = 0; a < 9; ++a) fp[a] = zero;
    const int L0 = periodic ? ys - HALO : max(ys - HALO, 0);
    load_row2<false>(P, phys(L0), c, f0, th0);
    load_row2<false>(P, phys(L0 + 1), c, f1, th1);
    // own values of the previous half's rows
    P2 cpsi0 = zero, cpsi1 = zero, cvx = zero, cvy0 = zero, cvy1 = zero, crho0 = zero, crho1 = zero;
    P2 cu20 = zero, cu21 = zero, cu30 = zero, cu31 = zero, cu40 = zero, cu41 = zero;
    P2 acc_m1 = zero;  // row L - 3's accumulator, made by C one iteration ago

    auto iter = [&](const int L, auto steady) {
        constexpr bool S = decltype(steady)::value;
        // ---- P: rows L, L + 1
        P2 rho0, rho1;
        auto stageP = [&](P2 (&f)[9], P2 th, int y, int s, P2& rho, P2& psi) {
            if (!S && !periodic) {
                const P2 d = 0.5f * (f[1] - f[3]);
                const bool lo = y == 0, hi = P.bc == BC_WALLS && y == Ly - 1;
                f[2] = sel(lo, f[4], f[2]);
                f[5] = sel(lo, f[7] - d, f[5]);
                f[6] = sel(lo, f[8] + d, f[6]);
                f[4] = sel(hi, f[2], f[4]);
                f[7] = sel(hi, f[5] + d, f[7]);
                f[8] = sel(hi, f[6] - d, f[8]);
            }
            rho = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
            bool bad = false;
            psi = eos_psi2(rho, th + P2(C.kp[KP_TS]), C, bad);
            if (S) eos_bad |= bad;
            else eos_bad |= bad && (periodic ? y < ye + HALO : y < min(ye + HALO, Ly));
            put(bc + M::PSI + s * MW, psi);
            put(t0 + s * MW, th);
            if constexpr (REC) {
                if (mine(y)) {
                    save(R->rho, phys(y), rho);
                    save(R->psi, phys(y), psi);
                }
            }
        };
        P2 psi0, psi1;
        stageP(f0, th0, L, 0, rho0, psi0);
        stageP(f1, th1, L + 1, 1, rho1, psi1);
        const P2 thL = th0;
        __syncthreads();

        // ---- bottom-wall heat flux of level t (Sec. 3.2), one term per column
        if (QF && !S && !periodic && ys == 0 && L == 2) {
            const P2 r0 = own(bp + M::RHO + MW), a0 = own(t1), a1 = own(t1 + MW), a2 = own(t0);
            if (outa) lb_st(P.qpart + c.a, heat_term(r0.x(), a0.x(), a1.x(), a2.x()), P.qpart, P.Lx, P.acc);
            if (outb) lb_st(P.qpart + c.b, heat_term(r0.y(), a0.y(), a1.y(), a2.y()), P.qpart, P.Lx, P.acc);
        }

        // ---- B: rows L - 1, L
        P2 vx0, vy0, vx1, vy1, rhob = rho0, rhoa = rhop;
        {
            const Row3 w0 = rowc(bp + M::PSI, cpsi0), w1 = rowc(bp + M::PSI + MW, cpsi1), w2 = rowc(bc + M::PSI, psi0), w3 = rowc(bc + M::PSI + MW, psi1);
            struct Flow {
                P2 rho, vx, vy, Fx, Fy, g2;
            };
            auto flow = [&](const Row3& m, const Row3& o, const Row3& p, const P2 (&g)[9], P2 rho, int y, int s) {
                const bool wall = !S && !periodic && (y == 0 || y == Ly - 1);
                const P2 jx = (g[1] - g[3]) + (g[5] - g[6]) + (g[8] - g[7]);
                const P2 jy = (g[2] - g[4]) + (g[5] + g[6]) - (g[7] + g[8]);
                Row3 ps = m, pn = p;
                if (!S && !periodic) {
                    ps = Row3{sel(y == 0, o.w, m.w), sel(y == 0, o.c, m.c), sel(y == 0, o.e, m.e)};
                    pn = Row3{sel(y == Ly - 1, o.w, p.w), sel(y == Ly - 1, o.c, p.c), sel(y == Ly - 1, o.e, p.e)};
                }
                const St2 d = stencil2(ps, o, pn, false);  // 12 sum_a w_a psi(x + e_a) e_a, Eq. 7
                const P2 mG = P2(C.kp[KP_GN12]) * o.c;
                Flow q;
                q.rho = rho;
                q.Fx = mG * d.dx, q.Fy = mG * d.dy;
                q.g2 = fma2(d.dx, d.dx, d.dy * d.dy);
                if (!S) {
                    const bool off = wall && !P.ghost;
                    q.Fx = sel(off, zero, q.Fx);
                    q.Fy = sel(off, zero, q.Fy);
                    q.g2 = sel(off, zero, q.g2);
                    if (!periodic) q.Fy = sel(y == 1, fma2(P2(P.kp[KP_GW6]), o.c * o.c, q.Fy), q.Fy);  // Eq. 22
                }
                const P2 Fb = fma2(P2(C.kp[KP_GN]), rho - P2(P.kp[KP_RHOAVE]), q.Fy);  // Eq. 9
                q.Fy = S ? Fb : sel(wall, q.Fy, Fb);
                const P2 irho = rcp2(rho);
                q.vx = fma2(P2::bc(0.5f), q.Fx, jx) * irho;  // Eq. 6
                q.vy = fma2(P2::bc(0.5f), q.Fy, jy) * irho;
                put(bc + M::VX + s * MW, q.vx);
                put(bc + M::VY + s * MW, q.vy);
                put(bc + M::RHO + s * MW, rho);
                return q;
            };
            auto store = [&](const P2 (&w)[9], P2 rho, int y) {
                const int pl = P.plane;
                float* out = P.f_out + (S ? y : phys(y)) * P.pitch;
                nonfinite |= (outa && !finite_f(rho.x())) || (outb && !finite_f(rho.y()));
#pragma unroll
                for (int a = 0; a < 9; ++a) {
                    lb_st_if(outa, out + (a * pl + c.a), w[a].x(), P.f_out, 9 * (size_t)pl, P.acc);
                    lb_st_if(outb, out + (a * pl + c.b), w[a].y(), P.f_out, 9 * (size_t)pl, P.acc);
                }
            };
            const Flow qa = flow(w0, w1, w2, fp, rhop, L - 1, 0);
            const Flow qb = flow(w1, w2, w3, f0, rho0, L, 1);
            vx0 = qa.vx, vy0 = qa.vy, vx1 = qb.vx, vy1 = qb.vy;
            // the next two rows' loads, most of an iteration ahead
            const bool more = S || L + 2 < ye + HALO;
            auto shift = [&] {
#pragma unroll
                for (int a = 0; a < 9; ++a) fp[a] = f1[a];
                rhop = rho1;
            };
            auto load0 = [&] { load_row2<S>(P, S ? L + 2 : phys(L + 2), c, f0, th0); };
            auto load1 = [&] { load_row2<S>(P, S ? L + 3 : phys(L + 3), c, f1, th1); };
            const bool sa = OUT && (S || mine(L - 1)), sb = OUT && (S || mine(L));
            P2 wa[9], wb[9];
            if (sa) {
                collide2(fp, qa.rho, qa.vx, qa.vy, qa.Fx, qa.Fy, qa.g2, C, wa);
                store(wa, qa.rho, L - 1);
            }
            if (EARLY) {
                shift();
                if (more) load1();
            }
            if (sb) collide2(f0, qb.rho, qb.vx, qb.vy, qb.Fx, qb.Fy, qb.g2, C, wb);
            if (EARLY && more) load0();
            if (sb) store(wb, qb.rho, L);
            if (!EARLY) {
                shift();
                if (more) {
                    load0();
                    load1();
                }
            }
        }
        __syncthreads();

        P2 accC0 = zero, accC1 = zero;
        if (thermal) {
            // ---- C: rows L - 2, L - 1
            Coef2 ka, kb;
            P2 u2a, u2b, tha;
            {
                P2 da, db;
                {
                    const Row3 m = rowc(bp + M::VX, zero), o = rowc(bp + M::VX + MW, cvx), p = rowc(bc + M::VX, vx0), q = rowc(bc + M::VX + MW, vx1);
                    const St2 A = stencil2(m, o, p, false), B = stencil2(o, p, q, false);
                    da = A.dx;
                    db = B.dx;
                    ka.ax = P2::bc(-1.f / 12.f) * A.c;
                    kb.ax = P2::bc(-1.f / 12.f) * B.c;
                }
                {
                    const Row3 m = rowc(bp + M::VY, cvy0), o = rowc(bp + M::VY + MW, cvy1), p = rowc(bc + M::VY, vy0), q = rowc(bc + M::VY + MW, vy1);
                    const St2 A = stencil2(m, o, p, false), B = stencil2(o, p, q, false);
                    da = da + A.dy;  // 12 div v
                    db = db + B.dy;
                    ka.ay = P2::bc(-1.f / 12.f) * A.c;
                    kb.ay = P2::bc(-1.f / 12.f) * B.c;
                }
                auto coef = [&](const St2& g, P2 divv, Coef2& k) {  // ax, ay divided by 12
                    const P2 q = P2(C.kp[KP_CHI144]) * rcp2(g.c);
                    const P2 br = P2(C.kp[KP_B]) * g.c;
                    k.ax = fma2(q, g.dx, k.ax);
                    k.ay = fma2(q, g.dy, k.ay);
                    k.cA = P2(C.kp[KP_RCV12]) * divv * rcp2(P2::bc(1.f) - br);
                    k.cB = P2(C.kp[KP_ACV12]) * (divv * g.c) * rcp2(fma2(br, P2::bc(2.f) - br, P2::bc(1.f)));
                };
                {
                    const Row3 m = rowc(bp + M::RHO, crho0), o = rowc(bp + M::RHO + MW, crho1), p = rowc(bc + M::RHO, rhoa), q = rowc(bc + M::RHO + MW, rhob);
                    const St2 A = stencil2(m, o, p, false), B = stencil2(o, p, q, false);
                    coef(A, da, ka);
                    coef(B, db, kb);
                    if constexpr (REC) {
                        auto rec = [&](const St2& g, P2 divv, const Coef2& k, int y) {
                            if (!mine(y)) return;
                            const bool fl = interior(y);
                            const int yy = phys(y);
                            const P2 w12 = P2::bc(1.f / 12.f), t12 = P2::bc(12.f);
                            save(R->drx, yy, sel(fl, w12 * g.dx, zero));
                            save(R->dry, yy, sel(fl, w12 * g.dy, zero));
                            save(R->divv, yy, sel(fl, w12 * divv, zero));
                            save(R->ax, yy, sel(fl, t12 * k.ax, zero));
                            save(R->ay, yy, sel(fl, t12 * k.ay, zero));
                        };
                        rec(A, da, ka, L - 2);
                        rec(B, db, kb, L - 1);
                    }
                }
                auto keep = [&](float2* q0, const Coef2& k) {
                    float2* q = at(q0, 0, 3 * MT);
                    q[0] = k.ax.f2();
                    q[MT] = k.ay.f2();
                    q[2 * MT] = k.cA.f2();
                    q[3 * MT] = k.cB.f2();
                };
                keep(k0, ka);
                keep(k0 + 4 * MT, kb);
                {
                    const Row3 m = row(t2 + MW), o = row(t1), p = row(t1 + MW), q = rowc(t0, thL);
                    accC0 = rhs_K2(stencil2(m, o, p, true), ka, C);
                    accC1 = rhs_K2(stencil2(o, p, q, true), kb, C);
                    P2 ua = fma2(P2::bc(0.5f), accC0, o.c), ub = fma2(P2::bc(0.5f), accC1, p.c);
                    if (!S) {
                        ua = sel(interior(L - 2), ua, o.c);
                        ub = sel(interior(L - 1), ub, p.c);
                    }
                    u2a = ua, u2b = ub, tha = o.c;
                    put(bc + M::U2, ua);
                    put(bc + M::U2 + MW, ub);
                    if constexpr (REC) {
                        if (mine(L - 2)) save(R->u2, phys(L - 2), ua);
                        if (mine(L - 1)) save(R->u2, phys(L - 1), ub);
                    }
                }
            }
            __syncthreads();
            auto coefs = [&](float2* q0) {
                const float2* q = at(q0, 0, 3 * MT);
                return Coef2{P2(q[0]), P2(q[MT]), P2(q[2 * MT]), P2(q[3 * MT])};
            };
            // ---- D: rows L - 3, L - 2
            const Coef2 kd = coefs(k1 + 4 * MT);  // row L - 3, for D and E
            const P2 td = own(t2 + MW);
            P2 u3a, u3b;
            {
                const Row3 m = rowc(bp + M::U2, cu20), o = rowc(bp + M::U2 + MW, cu21), p = rowc(bc + M::U2, u2a), q = rowc(bc + M::U2 + MW, u2b);
                const P2 ta = td, tb = tha;
                const P2 ha = rhs_K2(stencil2(m, o, p, true), kd, C);
                const P2 hb = rhs_K2(stencil2(o, p, q, true), ka, C);
                P2 ua = fma2(P2::bc(0.5f), ha, ta), ub = fma2(P2::bc(0.5f), hb, tb);
                if (!S) {
                    ua = sel(interior(L - 3), ua, ta);
                    ub = sel(interior(L - 2), ub, tb);
                }
                accD0 = fma2(P2::bc(2.f), ha, acc_m1);  // row L - 3
                accD1 = fma2(P2::bc(2.f), hb, accC0);   // row L - 2
                u3a = ua, u3b = ub;
                put(bc + M::U3, ua);
                put(bc + M::U3 + MW, ub);
                if constexpr (REC) {
                    if (mine(L - 3)) save(R->u3, phys(L - 3), ua);
                    if (mine(L - 2)) save(R->u3, phys(L - 2), ub);
                }
            }
            __syncthreads();
            // ---- E: rows L - 4, L - 3
            P2 eb, u4a, u4b;
            const Coef2 ke = coefs(k1);  // row L - 4, for E and F
            const P2 te = own(t2);
            {
                const Row3 m = rowc(bp + M::U3, cu30), o = rowc(bp + M::U3 + MW, cu31), p = rowc(bc + M::U3, u3a), q = rowc(bc + M::U3 + MW, u3b);
                const P2 ta = te, tb = td;
                const P2 ha = rhs_K2(stencil2(m, o, p, true), ke, C);
                const P2 hb = rhs_K2(stencil2(o, p, q, true), kd, C);
                P2 ua = ta + ha, ub = tb + hb;
                if (!S) {
                    ua = sel(interior(L - 4), ua, ta);
                    ub = sel(interior(L - 3), ub, tb);
                }
                accF1 = fma2(P2::bc(2.f), ha, accE);   // row L - 4
                eb = fma2(P2::bc(2.f), hb, accD0);     // row L - 3
                u4a = ua, u4b = ub;
                put(bc + M::U4, ua);
                put(bc + M::U4 + MW, ub);
                if constexpr (REC) {
                    if (mine(L - 4)) save(R->u4, phys(L - 4), ua);
                    if (mine(L - 3)) save(R->u4, phys(L - 3), ub);
                }
            }
            __syncthreads();
            // ---- F: rows L - 5, L - 4
            if (OUT) {
                const Row3 m = rowc(bp + M::U4, cu40), o = rowc(bp + M::U4 + MW, cu41), p = rowc(bc + M::U4, u4a), q = rowc(bc + M::U4 + MW, u4b);
                const P2 ta = own(t3 + MW), tb = te;
                const P2 ha = rhs_K2(stencil2(m, o, p, true), coefs(k2 + 4 * MT), C);
                const P2 hb = rhs_K2(stencil2(o, p, q, true), ke, C);
                P2 na = fma2(accF0 + ha, P2::bc(1.f / 6.f), ta), nb = fma2(accF1 + hb, P2::bc(1.f / 6.f), tb);
                auto store = [&](P2 v, int y) {
                    if (!S) {
                        if (!mine(y)) return;
                        if (!periodic) {
                            if (y == 0) v = P2(lb_ldg(P.thb + c.a, P.thb, P.pitch, P.acc), lb_ldg(P.thb + c.b, P.thb, P.pitch, P.acc));
                            if (y == Ly - 1) v = zero;
                        }
                    }
                    float* out = P.th_out + (S ? y : phys(y)) * P.pitch;
                    nonfinite |= (outa && !finite_f(v.x())) || (outb && !finite_f(v.y()));
                    lb_st_if(outa, out + c.a, v.x(), P.th_out, (size_t)P.plane, P.acc);
                    lb_st_if(outb, out + c.b, v.y(), P.th_out, (size_t)P.plane, P.acc);
                };
                store(na, L - 5);
                store(nb, L - 4);
            }
            cu20 = u2a, cu21 = u2b, cu30 = u3a, cu31 = u3b, cu40 = u4a, cu41 = u4b;
            accF0 = eb;      // row L - 3 = the next iteration's L - 5
            accE = accD1;    // row L - 2 = the next iteration's L - 4
            acc_m1 = accC1;  // row L - 1 = the next iteration's L - 3
        } else if (OUT) {
            auto store = [&](P2 v, int y) {
                if (!mine(y)) return;
                float* out = P.th_out + phys(y) * P.pitch;
                nonfinite |= (outa && !finite_f(v.x())) || (outb && !finite_f(v.y()));
                lb_st_if(outa, out + c.a, v.x(), P.th_out, (size_t)P.plane, P.acc);
                lb_st_if(outb, out + c.b, v.y(), P.th_out, (size_t)P.plane, P.acc);
            };
            store(own(t3 + MW), L - 5);
            store(own(t2), L - 4);
        }
        cpsi0 = psi0, cpsi1 = psi1, cvx = vx1, cvy0 = vy0, cvy1 = vy1, crho0 = rhoa, crho1 = rhob;
        // rotate the halves
        float2* s = bc;
        bc = bp;
        bp = s;
        s = t3;
        t3 = t2;
        t2 = t1;
        t1 = t0;
        t0 = s;
        s = k2;
        k2 = k1;
        k1 = k0;
        k0 = s;
    };
    // steady iterations: stored rows L - 5 .. L in the segment; with walls the
    // rows L - 5 .. L + 1 off the walls and above the first fluid row; the
    // rows the next loads pull from, up to L + 4, inside
    const int Ls = ys + HALO + (ys == 0 && !periodic ? 2 : 0);
    const int Le = min(ye, Ly - 4);
    int L = L0;
    for (; L < Ls; L += 2) iter(L, std::false_type{});
    for (; L < Le; L += 2) iter(L, std::true_type{});
    for (; L <= ye + HALO - 1; L += 2) iter(L, std::false_type{});
    if (eos_bad) atomicOr(&P.acc->err, ERR_EOS);
    if (nonfinite) atomicOr(&P.acc->err, ERR_NONFINITE);
    // (at the block's end, where it delays nothing)
    if (QF && fold && !periodic && block == 0 && lc < 32) fold_heat(P, lc);
}

}  // namespace

}  // namespace lbgpu
