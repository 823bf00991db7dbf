// One reverse step of a small domain in one launch (included by
// lb_adjoint.cu, whose two column-marching kernels serve the larger ones).
//
// A block computes NW * K rows of 64 columns, 6 of them halo on each side,
// through every part of the transposed step: the four RK stages (R4 .. R1,
// each one cell further in), the coefficients, the collision with the pull
// (C) and the transposed force sums and EOS (P); six barriers per tile, in
// place of five per row and two launches. The layout is the tiled step's
// (lb_tile.cuh): lane l holds columns l and l + 32 in one float2, warp w owns K
// rows, what only the own cell needs stays in registers, fields read at the
// neighbours are shared rows whose edge slots repeat the other half's column.
// The seven planes that the marching kernels pass between them never leave the
// block. A domain's last rows get the halo's room of the missing side: the
// first and the last tile write NW * K - 6 rows, the others NW * K - 12.

constexpr int RV_HALO = 6, RV_COLS = TILE_W - 2 * RV_HALO;  // 52 output columns

template <int NW, int K>
struct RevShape2 {
    static constexpr int rows = NW * K, out = rows - 2 * RV_HALO, edge = rows - RV_HALO;
    static constexpr int field = (rows + 2) * TILE_ROW, slots = 10 * field;
    static_assert(edge - out + 1 >= 2 && rows - edge + 1 >= 2, "the top two rows share a tile");
};

// Tiles in y of a domain of Ly rows, and the rows [ys, ye) of tile i. The top
// two rows always share a tile (the outflow top adds to what row Ly - 2
// stored): with two tiles or more the last has at least edge - out + 1 rows.
template <class Sh>
__host__ __device__ __forceinline__ int rev_tiles(int Ly) {
    if (Ly <= Sh::rows) return 1;
    const int mid = Ly - 2 * Sh::edge;
    return 2 + (mid > 0 ? (mid + Sh::out - 1) / Sh::out : 0);
}
template <class Sh>
__host__ __device__ __forceinline__ void rev_rows(int Ly, int i, int nt, int& ys, int& ye) {
    auto start = [&](int k) {
        if (k == 0) return 0;
        if (k == nt) return Ly;
        return Sh::edge + (k - 1) * Sh::out;
    };
    ys = start(i);
    ye = start(i + 1);
}

template <int NW, int K>
__global__ void __launch_bounds__(NW * 32) rev_tile(const StepParams P, AdjFields A, float lq) {
    using Sh = RevShape2<NW, K>;
    extern __shared__ float2 sm2[];
    grid_start();
    const int Lx = P.Lx, Ly = P.Ly, pitch = P.pitch, pl = P.plane;
    const int lane = threadIdx.x & 31, j0 = (threadIdx.x >> 5) * K;
    const int nstrips = (Lx + RV_COLS - 1) / RV_COLS;
    const int x0 = blockIdx.x % nstrips * RV_COLS, nv = min(RV_COLS, Lx - x0);
    int ys, ye;
    rev_rows<Sh>(Ly, blockIdx.x / nstrips, gridDim.x / nstrips, ys, ye);
    const int r0 = max(ys - RV_HALO, 0) + j0;  // this thread's first row
    Cols c;
    c.a = wrap(x0 - RV_HALO + lane, Lx);
    c.b = wrap(x0 - RV_HALO + lane + 32, Lx);
    c.am = c.a == 0 ? Lx - 1 : c.a - 1;
    c.ap = c.a == Lx - 1 ? 0 : c.a + 1;
    c.bm = c.b == 0 ? Lx - 1 : c.b - 1;
    c.bp = c.b == Lx - 1 ? 0 : c.b + 1;
    const bool outa = lane >= RV_HALO && lane < RV_HALO + nv;
    const bool outb = lane + 32 < TILE_W - RV_HALO && lane + 32 < RV_HALO + nv;
    auto any = [&](int d) { return r0 + K > max(ys - d, 0) && r0 < min(ye + d, Ly); };
    auto mine = [&](int r) { return r >= ys && r < ye; };
    auto isrow = [&](int r) { return r < Ly; };  // (r >= 0 always)
    auto wallrow = [&](int r) { return r == 0 || r == Ly - 1; };
    const P2 zero = P2::bc(0.f);

    // shared fields; the flow part's reuse the thermal part's
    enum { MU0, MU1, AX, AY, U4, U3, U2, TH, LR, PSI, LDRX = U4, LDRY = U3, LDIV = U2, QX = MU0, QY = MU1 };
    float2* const own = sm2 + (j0 + 1) * TILE_ROW + 1 + lane;
    const bool edge = lane == 0 || lane == 31;
    const int eo = lane == 0 ? 64 : -63;  // as in lb_tile.cuh
    auto at = [&](float2* q) { return smem_at(q, -lane - 1, 32 - lane, sm2, Sh::slots, P.acc); };
    auto put = [&](int F, int k, P2 v) {
        float2* q = at(own + F * Sh::field + k * TILE_ROW);
        *q = v.f2();
        if (edge) reinterpret_cast<float*>(q)[eo] = lane == 0 ? v.y() : v.x();
    };
    auto row = [&](int F, int k) {
        const float2* q = at(own + F * Sh::field + k * TILE_ROW);
        return Row3{P2(q[-1]), P2(q[0]), P2(q[1])};
    };
    auto cell = [&](int F, int k) { return P2(*at(own + F * Sh::field + k * TILE_ROW)); };
    auto load = [&](const float* p, int r) {  // (rows beyond the wall: the wall row's value)
        const int i = min(r, Ly - 1) * pitch;
        return P2(LB_LD(p, i + c.a, pl), LB_LD(p, i + c.b, pl));
    };
    auto store = [&](float* p, int i, int xa, int xb, P2 v, size_t n) {
        lb_st_if(outa, p + (i + xa), v.x(), p, n, P.acc);
        lb_st_if(outb, p + (i + xb), v.y(), p, n, P.acc);
    };

    // ---- inputs of the thermal part, and the flow part's two rings
    P2 lbar[K], cA[K], cB[K], rho[K], divv[K], th[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        lbar[k] = cA[k] = cB[k] = zero;
        rho[k] = P2::bc(1.f);
        divv[k] = th[k] = zero;
    }
    if (any(RV_HALO)) {
        P2 v[K][8];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int r = r0 + k;
            lbar[k] = load(A.lt_in, r);
            v[k][0] = load(A.ax, r);
            v[k][1] = load(A.ay, r);
            v[k][2] = load(A.u4, r);
            v[k][3] = load(A.u3, r);
            v[k][4] = load(A.u2, r);
            v[k][5] = load(A.lr_in, r);
            v[k][6] = load(A.psi, r);
            rho[k] = load(A.rho, r);
            divv[k] = load(A.divv, r);
            th[k] = load(A.theta, r);
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int r = r0 + k;
            if (r == 0 && mine(0)) {  // lambda of theta_b: what the step's wall row took
                if (outa) LB_ADD(A.dTb, c.a, pitch, (double)lbar[k].x());
                if (outb) LB_ADD(A.dTb, c.b, pitch, (double)lbar[k].y());
            }
            lbar[k] = sel(wallrow(r) || !isrow(r), zero, lbar[k]);
            put(MU0, k, (1.f / 6.f) * lbar[k]);
            put(AX, k, v[k][0]);
            put(AY, k, v[k][1]);
            put(U4, k, v[k][2]);
            put(U3, k, v[k][3]);
            put(U2, k, v[k][4]);
            put(LR, k, v[k][5]);
            put(PSI, k, v[k][6]);
            put(TH, k, th[k]);
            // the coefficients of the source term as the step forms them (Eq. 18)
            const P2 br = P.b * rho[k];
            cA[k] = (P.R * P.inv_cv) * divv[k] * rcp2(P2::bc(1.f) - br);
            cB[k] = (P.a * P.inv_cv) * (divv[k] * rho[k]) * rcp2(fma2(br, P2::bc(2.f) - br, P2::bc(1.f)));
        }
    }
    __syncthreads();

    // ---- the RK stages transposed (see rev_thermal_fused): lambda_u = -Dx[ax
    // mu] - Dy[ay mu] + chi Lap[mu] + the source's local part, from the stage's
    // mu (field M) and input u (field U); the next stage's mu goes to field N
    P2 lax[K], lay[K], lcA[K], lcB[K], lth[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        lax[k] = lay[k] = lcA[k] = lcB[k] = zero;
        lth[k] = lbar[k];
    }
    auto stage = [&](int d, int M, int U, int N, float ab, float bb) {
        if (!any(d)) return;
        Row3 xm = row(AX, -1), xc = row(AX, 0), ym = row(AY, -1), yc = row(AY, 0);
        Row3 mm = row(M, -1), mc = row(M, 0), um = row(U, -1), uc = row(U, 0);
        // the shared row below the tile's first holds no cell
        if (j0 == 0) xm = ym = mm = um = Row3{zero, zero, zero};
#pragma unroll
        for (int k = 0; k < K; ++k) {
            Row3 xp = row(AX, k + 1), yp = row(AY, k + 1), mp = row(M, k + 1), up = row(U, k + 1);
            if (j0 + k + 1 == Sh::rows || r0 + k + 1 >= Ly) xp = yp = mp = up = Row3{zero, zero, zero};
            const P2 four = P2::bc(4.f);
            const P2 dxp = fma2(four, fma2(xc.e, mc.e, -(xc.w * mc.w)),
                                fma2(xm.e, mm.e, -(xm.w * mm.w)) + fma2(xp.e, mp.e, -(xp.w * mp.w)));
            const P2 dyp = fma2(four, fma2(yp.c, mp.c, -(ym.c * mm.c)),
                                fma2(yp.e, mp.e, yp.w * mp.w) - fma2(ym.e, mm.e, ym.w * mm.w));
            const P2 lap = fma2(P2::bc(-20.f), mc.c, fma2(four, (mc.e + mc.w) + (mm.c + mp.c), (mm.e + mm.w) + (mp.e + mp.w)));
            P2 lu = fma2(P2::bc(P.chi * (1.f / 6.f)), lap, P2::bc(-1.f / 12.f) * (dxp + dyp));
            const P2 m = mc.c;
            const P2 T = uc.c + P2::bc(P.Ts);
            const P2 rsq = rsqrt2(T);
            const P2 dphi = fma2(P2::bc(-P.k0k1), rsq, P2::bc(P.k1k1));
            const P2 d2phi = P2::bc(0.5f * P.k0k1) * (rsq * rsq * rsq);
            lu = fma2(fma2(T * cB[k], d2phi, fma2(cB[k], dphi, -cA[k])), m, lu);
            const P2 d1 = up.e - um.w, d2 = um.e - up.w;
            lax[k] = fma2(P2::bc(1.f / 12.f) * fma2(four, uc.e - uc.w, d1 + d2), m, lax[k]);
            lay[k] = fma2(P2::bc(1.f / 12.f) * fma2(four, up.c - um.c, d1 - d2), m, lay[k]);
            lcA[k] = fma2(-T, m, lcA[k]);
            lcB[k] = fma2(T * dphi, m, lcB[k]);
            lth[k] = lth[k] + lu;
            if (N >= 0) {
                const P2 next = fma2(P2::bc(bb), lu, ab * lbar[k]);
                put(N, k, sel(wallrow(r0 + k) || !isrow(r0 + k), zero, next));
            }
            xm = xc, xc = xp, ym = yc, yc = yp, mm = mc, mc = mp, um = uc, uc = up;
        }
    };
    stage(5, MU0, U4, MU1, 1.f / 3.f, 1.f);
    __syncthreads();
    stage(4, MU1, U3, MU0, 1.f / 3.f, 0.5f);
    __syncthreads();
    stage(3, MU0, U2, MU1, 1.f / 6.f, 0.5f);
    __syncthreads();
    stage(2, MU1, TH, -1, 0.f, 0.f);

    // ---- the coefficients -> lambda of grad rho and div v (shared), and the
    // local parts of lambda_rho (lambda_v is -lax, -lay)
    P2 lrho[K];
    if (any(2)) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int r = r0 + k;
            const bool none = wallrow(r) || !isrow(r);
            P2 drx = zero, dry = zero;
            if (mine(r)) {  // (lambda_rho matters on the own rows only)
                drx = load(A.drx, r);
                dry = load(A.dry, r);
            }
            const P2 irho = rcp2(rho[k]), br = P.b * rho[k];
            const P2 i1 = rcp2(P2::bc(1.f) - br);
            const P2 D = fma2(br, P2::bc(2.f) - br, P2::bc(1.f)), iD = rcp2(D);
            const P2 dD = (2.f * P.b) * (P2::bc(1.f) - br);
            const P2 wA = (P.R * P.inv_cv) * lcA[k], wB = (P.a * P.inv_cv) * lcB[k];
            put(LDRX, k, sel(none, zero, P.chi * (lax[k] * irho)));
            put(LDRY, k, sel(none, zero, P.chi * (lay[k] * irho)));
            put(LDIV, k, sel(none, zero, fma2(wA, i1, wB * (rho[k] * iD))));
            const P2 g = (-P.chi) * (fma2(drx, lax[k], dry * lay[k]) * (irho * irho));
            const P2 e = fma2(P.b * wA, i1 * i1, wB * ((D - rho[k] * dD) * (iD * iD)));
            lrho[k] = sel(none, zero, fma2(e, divv[k], g));
            lax[k] = sel(none, zero, lax[k]);
            lay[k] = sel(none, zero, lay[k]);
        }
    }
    __syncthreads();

    // ---- C: collision, velocity, forces, pull (see rev_flow_fused)
    P2 lpsi[K], wlf[9];
#pragma unroll
    for (int a = 0; a < 9; ++a) wlf[a] = zero;
    const float G = P.G;
    if (any(1)) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const int y = r0 + k;
            P2 n_lpsi = zero, q0 = zero, q1 = zero;
            if (isrow(y) && y + 1 >= ys && y < ye + 1) {
                const bool wall = wallrow(y);
                P2 f[9], lo[9], t;
                load_row2<false>(P, y, c, f, t);
#pragma unroll
                for (int a = 0; a < 9; ++a)
                    lo[a] = P2(LB_LD(A.lf_in, a * pl + y * pitch + c.a, 9 * (size_t)pl),
                               LB_LD(A.lf_in, a * pl + y * pitch + c.b, 9 * (size_t)pl));
                {
                    const P2 d = 0.5f * (f[1] - f[3]);
                    const bool b = y == 0, tp = P.bc == BC_WALLS && y == Ly - 1;
                    f[2] = sel(b, f[4], f[2]);
                    f[5] = sel(b, f[7] - d, f[5]);
                    f[6] = sel(b, f[8] + d, f[6]);
                    f[4] = sel(tp, f[2], f[4]);
                    f[7] = sel(tp, f[5] + d, f[7]);
                    f[8] = sel(tp, f[6] - d, f[8]);
                }
                // lambda of f*^{n+1}: lf part + lr of the cell that pulled it
                // (rows beyond the walls hold no cell)
                Row3 lm = row(LR, k - 1), lc = row(LR, k), lp = row(LR, k + 1);
                Row3 pm = row(PSI, k - 1), pc = row(PSI, k), pn = row(PSI, k + 1);
                Row3 xm = row(LDRX, k - 1), xc = row(LDRX, k), xp = row(LDRX, k + 1);
                Row3 ym = row(LDRY, k - 1), yp = row(LDRY, k + 1);
                Row3 vm = row(LDIV, k - 1), vc = row(LDIV, k), vp = row(LDIV, k + 1);
                const Row3 none{zero, zero, zero};
                if (y == 0) lm = xm = ym = vm = none, pm = pc;
                if (y == Ly - 1) lp = xp = yp = vp = none, pn = pc;
                lo[0] = lo[0] + lc.c;
                lo[1] = lo[1] + lc.e;
                lo[2] = lo[2] + lp.c;
                lo[3] = lo[3] + lc.w;
                lo[4] = lo[4] + lm.c;
                lo[5] = lo[5] + lp.e;
                lo[6] = lo[6] + lp.w;
                lo[7] = lo[7] + lm.w;
                lo[8] = lo[8] + lm.e;
                const P2 psi = pc.c;
                P2 Fmx = zero, Fmy = zero;
                if (!wall || P.ghost) {
                    const St2 g = stencil2(pm, pc, pn, false);
                    const P2 mG = (-G * (1.f / 12.f)) * psi;
                    Fmx = mG * g.dx;
                    Fmy = mG * g.dy;
                }
                const P2 w12 = P2::bc(-1.f / 12.f);
                const P2 lr_c = w12 * (stencil2(xm, xc, xp, false).dx + stencil2(ym, none, yp, false).dy);
                const St2 dv = stencil2(vm, vc, vp, false);
                const P2 rh = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7])) + f[8];
                const P2 jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
                const P2 jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
                const P2 Fx = Fmx;
                P2 Fy = Fmy;
                const P2 psi2 = psi * psi;
                if (!wall) {
                    if (y == 1) Fy = fma2(P2::bc(P.gw6), psi2, Fy);
                    Fy = fma2(P2::bc(-P.g), rh - P2::bc(P.rho_ave), Fy);
                }
                const P2 irho = rcp2(rh), half = P2::bc(0.5f);
                const P2 vx = fma2(half, Fx, jx) * irho, vy = fma2(half, Fy, jy) * irho;
                // lambda_dm = diag(1/9, 1/36, ...) M lambda_f*
                const P2 sa = (lo[1] + lo[3]) + (lo[2] + lo[4]), sd = (lo[5] + lo[7]) + (lo[6] + lo[8]);
                const P2 ex = lo[1] - lo[3], ey = lo[2] - lo[4];
                const P2 dx = (lo[5] - lo[7]) + (lo[8] - lo[6]), dy = (lo[5] - lo[7]) + (lo[6] - lo[8]);
                const P2 ldm1 = (1.f / 36.f) * (fma2(P2::bc(2.f), sd, -sa) - 4.f * lo[0]);
                const P2 ldm2 = (1.f / 36.f) * (fma2(P2::bc(-2.f), sa, sd) + 4.f * lo[0]);
                const P2 ldm3 = (1.f / 6.f) * (ex + dx), ldm4 = (1.f / 12.f) * fma2(P2::bc(-2.f), ex, dx);
                const P2 ldm5 = (1.f / 6.f) * (ey + dy), ldm6 = (1.f / 12.f) * fma2(P2::bc(-2.f), ey, dy);
                const P2 ldm7 = 0.25f * ((lo[1] + lo[3]) - (lo[2] + lo[4]));
                const P2 ldm8 = 0.25f * ((lo[5] + lo[7]) - (lo[6] + lo[8]));
                // forward quantities of dm
                const P2 v2 = fma2(vx, vx, vy * vy), vd = fma2(vx, vx, -(vy * vy)), vp2 = vx * vy;
                const P2 ne7 = ((f[1] + f[3]) - (f[2] + f[4])) - rh * vd;
                const P2 ne8 = ((f[5] + f[7]) - (f[6] + f[8])) - rh * vp2;
                const P2 ipsi2 = P2(psi2.x() > 0.f ? rcp_approx(psi2.x()) : 0.f, psi2.y() > 0.f ? rcp_approx(psi2.y()) : 0.f);
                const P2 R = fma2(Fmx, Fmx, Fmy * Fmy) * ipsi2;
                const P2 S7 = 2.f * fma2(vx, Fx, -(vy * Fy)), S8 = fma2(vx, Fy, vy * Fx);
                const P2 sr = P.inv_drho * (rh - P2::bc(P.rho_v));
                const P2 sfr(__saturatef(sr.x()), __saturatef(sr.y()));
                const P2 snu = rcp2(fma2(P2::bc(P.dtau), sfr, P2::bc(P.tau_v)));
                // dm = -Lambda (m - meq) + (I - Lambda/2) S, momentum rows dm_j = F
                const P2 lne1 = -P.s_e * ldm1, lS1 = (1.f - 0.5f * P.s_e) * ldm1;
                const P2 lne2 = -P.s_z * ldm2, lS2 = (1.f - 0.5f * P.s_z) * ldm2;
                const P2 lne4 = -P.s_q * ldm4, lne6 = -P.s_q * ldm6;
                P2 lFx = fma2(P2::bc(0.5f * P.s_q - 1.f), ldm4, ldm3);
                P2 lFy = fma2(P2::bc(0.5f * P.s_q - 1.f), ldm6, ldm5);
                const P2 hnu = fma2(P2::bc(-0.5f), snu, P2::bc(1.f));
                const P2 lne7 = -(snu * ldm7), lS7 = hnu * ldm7;
                const P2 lne8 = -(snu * ldm8), lS8 = hnu * ldm8;
                const P2 lsnu = -fma2(fma2(half, S7, ne7), ldm7, fma2(half, S8, ne8) * ldm8);
                P2 lf[9];
                {
                    const P2 ax_ = fma2(P2::bc(-2.f), lne2, -lne1), dg = fma2(P2::bc(2.f), lne1, lne2);
                    lf[0] = fma2(P2::bc(4.f), lne2 - lne1, lo[0]);
                    lf[1] = lo[1] + ((ax_ - 2.f * lne4) + lne7);
                    lf[2] = lo[2] + ((ax_ - 2.f * lne6) - lne7);
                    lf[3] = lo[3] + ((ax_ + 2.f * lne4) + lne7);
                    lf[4] = lo[4] + ((ax_ + 2.f * lne6) - lne7);
                    lf[5] = lo[5] + ((dg + lne4) + (lne6 + lne8));
                    lf[6] = lo[6] + ((dg - lne4) + (lne6 - lne8));
                    lf[7] = lo[7] + ((dg - lne4) - (lne6 - lne8));
                    lf[8] = lo[8] + ((dg + lne4) - (lne6 + lne8));
                }
                // meq part (lambda_meq = -lambda_ne)
                const P2 q12 = lne2 - lne1;  // q1 - q2
                P2 n_lrho = fma2(P2::bc(2.f), lne1, -lne2) + fma2(3.f * q12, v2, fma2(lne4, vx, lne6 * vy)) -
                            fma2(lne7, vd, lne8 * vp2);
                P2 lvx = rh * (fma2(6.f * q12, vx, lne4) - fma2(2.f * lne7, vx, lne8 * vy));
                P2 lvy = rh * (fma2(6.f * q12, vy, lne6) + fma2(2.f * lne7, vy, -(lne8 * vx)));
                // S (Eq. 8): S1 = 6 vF + sig_e R, S2 = -6 vF - sig_z R, S7, S8
                const P2 lvF = 6.f * (lS1 - lS2);
                const P2 lR = fma2(P2::bc(P.sig_e), lS1, -P.sig_z * lS2);
                const P2 l7 = 2.f * lS7;
                lvx = lvx + fma2(lvF + l7, Fx, lS8 * Fy);
                lvy = lvy + fma2(lvF - l7, Fy, lS8 * Fx);
                lFx = lFx + fma2(lvF + l7, vx, lS8 * vy);
                lFy = lFy + fma2(lvF - l7, vy, lS8 * vx);
                const P2 w = 2.f * (lR * ipsi2);  // (0 where psi is)
                P2 lFmx = w * Fmx, lFmy = w * Fmy;
                n_lpsi = -(w * (R * psi));
                {  // snu(rho)
                    const P2 s = (-P.dtau * P.inv_drho) * (lsnu * (snu * snu));
                    n_lrho = n_lrho + P2(sr.x() > 0.f && sr.x() < 1.f ? s.x() : 0.f, sr.y() > 0.f && sr.y() < 1.f ? s.y() : 0.f);
                }
                // velocity v = (j + F/2) / rho with the thermal part's lambda_v
                lvx = lvx + fma2(w12, dv.dx, -lax[k]);
                lvy = lvy + fma2(w12, dv.dy, -lay[k]);
                n_lrho = n_lrho + (lrho[k] + lr_c);
                const P2 ljx = lvx * irho, ljy = lvy * irho;
                lFx = fma2(half, ljx, lFx);
                lFy = fma2(half, ljy, lFy);
                n_lrho = n_lrho - fma2(ljx, vx, ljy * vy);
                lf[1] = lf[1] + ljx;
                lf[2] = lf[2] + ljy;
                lf[3] = lf[3] - ljx;
                lf[4] = lf[4] - ljy;
                lf[5] = lf[5] + (ljx + ljy);
                lf[6] = lf[6] + (ljy - ljx);
                lf[7] = lf[7] - (ljx + ljy);
                lf[8] = lf[8] + (ljx - ljy);
                // forces: F = F_m + F_ads + F_b on fluid rows; on wall rows F_m
                // with the ghost layer, else none
                if (!wall || P.ghost) {
                    lFmx = lFmx + lFx;
                    lFmy = lFmy + lFy;
                    if (!wall) {
                        n_lrho = fma2(P2::bc(-P.g), lFy, n_lrho);  // F_b (Eq. 9)
                        if (y == 1) {                              // F_ads (Eq. 22) on the first fluid row
                            n_lpsi = fma2((2.f * P.gw6) * psi, lFy, n_lpsi);
                            const P2 d = (1.f / 6.f) * (psi2 * lFy);
                            if (mine(y) && outa) LB_ADD(A.dGwx, c.a, pitch, (double)d.x());
                            if (mine(y) && outb) LB_ADD(A.dGwx, c.b, pitch, (double)d.y());
                        }
                    }
                    const P2 ip(psi.x() > 0.f ? rcp_approx(psi.x()) : 0.f, psi.y() > 0.f ? rcp_approx(psi.y()) : 0.f);
                    n_lpsi = fma2(fma2(Fmx, lFmx, Fmy * lFmy), ip, n_lpsi);  // own factor of F_m
                } else {
                    lFmx = lFmy = zero;
                }
                q0 = psi * lFmx;
                q1 = psi * lFmy;
                lrho[k] = n_lrho;
                rho[k] = rh;
                if (mine(y)) {
                    if (wall) {  // completed in P
#pragma unroll
                        for (int a = 0; a < 9; ++a) wlf[a] = lf[a];
                    } else {  // pull-streaming transposed: lambda of f*_a(y - e_a), always inside
#pragma unroll
                        for (int a = 0; a < 9; ++a)
                            store(A.lf_out, a * pl + (y - EYd[a]) * pitch, EXd[a] == 0 ? c.a : EXd[a] > 0 ? c.am : c.ap,
                                  EXd[a] == 0 ? c.b : EXd[a] > 0 ? c.bm : c.bp, lf[a], 9 * (size_t)pl);
                    }
                }
            }
            lpsi[k] = n_lpsi;
            put(QX, k, q0);
            put(QY, k, q1);
        }
    }
    __syncthreads();

    // ---- P: F_m's neighbour sums, psi, q(t) and rho transposed; wall rows
    if (!any(0)) return;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int r = r0 + k;
        if (!mine(r)) continue;
        const bool wall = wallrow(r);
        Row3 xm = row(QX, k - 1), xc = row(QX, k), xp = row(QX, k + 1);
        Row3 ym = row(QY, k - 1), yc = row(QY, k), yp = row(QY, k + 1);
        const Row3 none{zero, zero, zero};
        const bool ghost = P.ghost && wall;  // the ghost row copies the wall row: its cells read psi here too
        if (r == 0) xm = ghost ? xc : none, ym = none;
        if (r == Ly - 1) xp = ghost ? xc : none, yp = none;
        auto yrow = [](const Row3& q) { return fma2(P2::bc(4.f), q.c, q.e + q.w); };
        P2 dq = fma2(P2::bc(4.f), xc.e - xc.w, (xm.e - xm.w) + (xp.e - xp.w)) + (yrow(yp) - yrow(ym));
        if (ghost) dq = r == 0 ? dq + yrow(yc) : dq - yrow(yc);
        const P2 lp = fma2(P2::bc(G * (1.f / 12.f)), dq, lpsi[k]);
        const P2 psi = cell(PSI, k);
        P2 lr = lrho[k], lt = lth[k];
        {  // psi^2 = 2 (p_EOS - rho/3) / G and its derivatives (Eq. 21)
            const P2 rh = rho[k], T = th[k] + P2::bc(P.Ts);
            const P2 rs = rsqrt2(T);
            const P2 base = fma2(P2::bc(-P.k1), T * rs, P2::bc(P.k0));
            const P2 aphi = P.a * (base * base), adphi = P.a * fma2(P2::bc(-P.k0k1), rs, P2::bc(P.k1k1));
            const P2 br = P.b * rh, i1 = rcp2(P2::bc(1.f) - br);
            const P2 D = fma2(br, P2::bc(2.f) - br, P2::bc(1.f)), iD = rcp2(D);
            const P2 dD = (2.f * P.b) * (P2::bc(1.f) - br);
            const P2 p_rho = fma2(P.R * T, i1 * i1, -((aphi * rh) * ((2.f * D - rh * dD) * (iD * iD))));
            const P2 p_T = fma2(P.R * rh, i1, -((adphi * (rh * rh)) * iD));
            const P2 q(psi.x() > 0.f ? lp.x() * rcp_approx(G * psi.x()) : 0.f, psi.y() > 0.f ? lp.y() * rcp_approx(G * psi.y()) : 0.f);
            lr = fma2(q, p_rho - P2::bc(1.f / 3.f), lr);
            lt = fma2(q, p_T, lt);
        }
        // q(t) = (1/Lx) sum_x -cvchi rho(x,0) (-3 th0 + 4 th1 - th2) / 2 (Sec. 3.2)
        if (lq != 0.f && r <= 2) {
            const float cq = lq / (float)Lx * (-P.cvchi);
            const P2 rho0 = r == 0 ? rho[k] : load(A.rho, 0);
            if (r == 0) {
                const P2 t1 = load(A.theta, 1), t2 = load(A.theta, 2);
                lr = lr + (0.5f * cq) * (fma2(P2::bc(-3.f), th[k], 4.f * t1) - t2);
            }
            lt = lt + (cq * (r == 0 ? -1.5f : r == 1 ? 2.f : -0.5f)) * rho0;
        }
        store(A.lt_out, r * pitch, c.a, c.b, lt, pl);
        store(A.lr_out, r * pitch, c.a, c.b, wall ? zero : lr, pl);
        if (wall) {
            P2 lf[9];
#pragma unroll
            for (int a = 0; a < 9; ++a) lf[a] = wlf[a] + lr;
            // Zou-He fill transposed: the filled populations pass their
            // adjoint to the known ones they were built from
            if (r == 0) {
                lf[4] = lf[4] + lf[2];
                lf[7] = lf[7] + lf[5];
                lf[1] = lf[1] + 0.5f * (lf[6] - lf[5]);
                lf[3] = lf[3] + 0.5f * (lf[5] - lf[6]);
                lf[8] = lf[8] + lf[6];
                lf[2] = lf[5] = lf[6] = zero;
            } else if (P.bc == BC_WALLS) {
                lf[2] = lf[2] + lf[4];
                lf[5] = lf[5] + lf[7];
                lf[1] = lf[1] + 0.5f * (lf[7] - lf[8]);
                lf[3] = lf[3] + 0.5f * (lf[8] - lf[7]);
                lf[6] = lf[6] + lf[8];
                lf[4] = lf[7] = lf[8] = zero;
            }
            // pull-streaming transposed as a scatter; where y + e_a lies
            // beyond the wall f*_a of this cell has no consumer: 0
#pragma unroll
            for (int a = 0; a < 9; ++a) {
                const int t = r - EYd[a], u = r + EYd[a];
                if (t >= 0 && t < Ly)
                    store(A.lf_out, a * pl + t * pitch, EXd[a] == 0 ? c.a : EXd[a] > 0 ? c.am : c.ap,
                          EXd[a] == 0 ? c.b : EXd[a] > 0 ? c.bm : c.bp, lf[a], 9 * (size_t)pl);
                if (u < 0 || u >= Ly) store(A.lf_out, a * pl + r * pitch, c.a, c.b, zero, 9 * (size_t)pl);
            }
            // the outflow top pulled populations 4, 7, 8 from its own row: a
            // second consumer besides the cell one row down, whose share row
            // Ly - 2 of this tile stored in C
            if (P.bc == BC_TOP_OUTFLOW && r == Ly - 1) {
                auto more = [&](int a, int xa, int xb) {
                    if (outa) LB_ADD(A.lf_out, a * pl + r * pitch + xa, 9 * (size_t)pl, lf[a].x());
                    if (outb) LB_ADD(A.lf_out, a * pl + r * pitch + xb, 9 * (size_t)pl, lf[a].y());
                };
                more(4, c.a, c.b);
                more(7, c.ap, c.bp);
                more(8, c.am, c.bm);
            }
        }
    }
}
