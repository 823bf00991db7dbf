// Device-side definitions shared by the kernels of the GB300 boiling step.
//
// Lattice: D2Q9 with e0=(0,0) e1=(1,0) e2=(0,1) e3=(-1,0) e4=(0,-1)
// e5=(1,1) e6=(-1,1) e7=(-1,-1) e8=(1,-1) (Sec. 2). Fields are pitched
// row-major [y][pitch] FP32, populations are 9 such planes (SoA).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lbgpu {

constexpr int HALO = 5;    // x-halo columns per side recomputed by a block
constexpr int TILE_COLS = 54;    // columns of a strip (64 less the halos); the marching form's blocks own two
constexpr int TILE24_ROWS = 14;  // rows a tile of 24 / 16 / 14 / 12 computed rows writes
constexpr int TILE16_ROWS = 6, TILE14_ROWS = 4, TILE12_ROWS = 2;

enum { BC_WALLS = 0, BC_TOP_OUTFLOW = 1, BC_PERIODIC = 2 };
enum : unsigned { ERR_EOS = 1u, ERR_NONFINITE = 2u, ERR_BOUNDS = 4u, ERR_TIMEOUT = 8u };

// FP64 device accumulators (wall heat flux of Sec. 3.2, mass, fault flags).
struct Acc {
    double spare;
    double q_last;      // q(t) of the last completed step
    double q_sum, q_sum2, q_n;
    double mass;
    unsigned int count; // unused (part of the saved-state record)
    unsigned int err;   // ERR_* bits
    double pad[2];
};

// Everything one launch of the step needs, passed by value.
struct StepParams {
    const float* f_in;
    float* f_out;
    const float* th_in;
    float* th_out;
    const float* thb;   // theta_b(x) = T_b(x) - T_s on the bottom wall
    Acc* acc;
    // the columns' terms of q(t) (fold_heat, lb_common.cuh): written by this step,
    // and those of the step before
    double* qpart;
    const double* qprev;
    double qscale;  // -c_v chi / (2 Lx)
    int Lx, Ly, pitch, plane;
    int bc, ghost, isothermal;
    int nstrips, seg_h;
    // Peng-Robinson EOS (Eq. 21): phi(T) = (k0 - k1 sqrt(T))^2 with
    // k0 = 1 + kappa, k1 = kappa / sqrt(Tc); psi^2 = two_over_G (p - rho/3).
    float Ts, a, b, R, two_over_G, k0, k1, G;
    float k0k1, k1k1;  // phi'(T) = k1^2 - k0 k1 / sqrt(T)
    // MRT collision (Eqs. 2, 4, 8)
    float s_e, s_z, s_q, sig_e, sig_z;
    float rho_v, inv_drho, tau_v, dtau;
    // forces (Eqs. 9, 22); gw6 = G_w/6 is -G_w sum_a omega_a s e_a,y on row 1
    float g, rho_ave, gw6;
    // temperature (Eq. 18): chi = c_v chi / c_v, cvchi = c_v chi
    float chi, cvchi, inv_cv;
    // the constants of the paired FP32 arithmetic, each duplicated into a
    // float2 so that a paired instruction can take it from the parameter
    // bank as it is (set_pairs)
    float2 kp[28];
};

enum {
    KP_TS, KP_K1N, KP_K0, KP_B, KP_R, KP_A, KP_2G, KP_K0K1N, KP_K1K1, KP_CHI6,
    KP_SE36N, KP_KE6, KP_KESIG, KP_SZ12N, KP_KZ6N, KP_KZSIGN, KP_SQ6, KP_SQ12N, KP_DTAU4, KP_TAUV4,
    KP_GN12, KP_GW6, KP_GN, KP_RHOAVE, KP_CHI144, KP_RCV12, KP_ACV12, KP_PSI, KP_COUNT
};

// Fill kp from the scalar fields (after any of them changes).
inline void set_pairs(StepParams& P) {
    static_assert(KP_COUNT == sizeof(P.kp) / sizeof(P.kp[0]), "kp size");
    const float G2 = P.G * P.G * (1.f / 144.f);
    // psi^2 is formed times 4^k, with |2 / G| 4^k in [2^54, 2^56): the smallest
    // |p - rho/3|, 2^-149, then gives at least 2^-95, and only beyond 2^72 does
    // it overflow
    const float tg = fabsf(P.two_over_G);
    const int k = tg > 0.f && tg <= 3.402823466e38f ? (55 - ilogbf(tg)) >> 1 : 0;
    const float ke = (1.f - 0.5f * P.s_e) * (1.f / 36.f), kz = (1.f - 0.5f * P.s_z) * (1.f / 36.f);
    const float v[KP_COUNT] = {P.Ts, -P.k1, P.k0, P.b, P.R, P.a, ldexpf(P.two_over_G, 2 * k), -P.k0k1, P.k1k1, P.chi * (1.f / 6.f),
                               -P.s_e * (1.f / 36.f), 6.f * ke, ke * P.sig_e * G2, -P.s_z * (1.f / 12.f), -6.f * kz,
                               -kz * P.sig_z * G2, P.s_q * (1.f / 6.f), -P.s_q * (1.f / 12.f), 4.f * P.dtau,
                               4.f * P.tau_v, -P.G * (1.f / 12.f), P.gw6, -P.g, P.rho_ave, P.chi * (1.f / 144.f),
                               P.R * P.inv_cv * (1.f / 12.f), P.a * P.inv_cv * (1.f / 12.f), ldexpf(1.f, -k)};
    for (int i = 0; i < KP_COUNT; ++i) P.kp[i] = make_float2(v[i], v[i]);
}

__device__ __forceinline__ int wrap(int v, int n) {
    int r = v % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ bool finite_f(float v) { return fabsf(v) <= 3.402823466e38f; }

// Checked build (-DLB_CHECKED, liblbboil_checked.so): every global and
// shared-memory access of the fused step goes through these; an address
// outside its buffer sets ERR_BOUNDS and the access is skipped (a load reads
// 0) instead of faulting. In the normal build they are the plain accesses.
// Loads of the state, which another grid or block writes while this kernel
// runs (kernels overlap their predecessor, grid_start; the persistent batch's
// blocks exchange buffers), are plain coherent ones (lb_ldco): after the wait
// they see those writes, where the read-only path (lb_ldg, for the wall
// temperature, which only copies write) may serve data it cached before; the
// terms of q(t) are read at L2 (lb_ldcg).
#ifdef LB_CHECKED
__device__ __forceinline__ bool lb_inside(const void* p, const void* base, size_t bytes, size_t width, Acc* acc) {
    const char* c = static_cast<const char*>(p);
    const char* b = static_cast<const char*>(base);
    if (base != nullptr && c >= b && c + width <= b + bytes) return true;
    atomicOr(&acc->err, ERR_BOUNDS);
    return false;
}
template <class T>
__device__ __forceinline__ T lb_ldg(const T* p, const T* base, size_t n, Acc* acc) {
    return lb_inside(p, base, n * sizeof(T), sizeof(T), acc) ? __ldg(p) : T(0);
}
template <class T>
__device__ __forceinline__ void lb_st(T* p, T v, const T* base, size_t n, Acc* acc) {
    if (lb_inside(p, base, n * sizeof(T), sizeof(T), acc)) *p = v;
}
template <class T>
__device__ __forceinline__ T lb_ldco(const T* p, const T* base, size_t n, Acc* acc) {
    return lb_inside(p, base, n * sizeof(T), sizeof(T), acc) ? *p : T(0);
}
template <class T>
__device__ __forceinline__ T lb_ldcg(const T* p, const T* base, size_t n, Acc* acc) {
    return lb_inside(p, base, n * sizeof(T), sizeof(T), acc) ? __ldcg(p) : T(0);
}
#else
template <class T>
__device__ __forceinline__ T lb_ldg(const T* p, const T*, size_t, Acc*) { return __ldg(p); }
template <class T>
__device__ __forceinline__ void lb_st(T* p, T v, const T*, size_t, Acc*) { *p = v; }
template <class T>
__device__ __forceinline__ T lb_ldco(const T* p, const T*, size_t, Acc*) { return *p; }
template <class T>
__device__ __forceinline__ T lb_ldcg(const T* p, const T*, size_t, Acc*) { return __ldcg(p); }
#endif
// A store that only lanes with `on` make, as one predicated instruction: a
// branch around a group of stores would end the basic block and with it the
// compiler's freedom to interleave two rows' arithmetic.
__device__ __forceinline__ void lb_st_if(bool on, float* p, float v, const float* base, size_t n, Acc* acc) {
#ifdef LB_CHECKED
    if (on) lb_st(p, v, base, n, acc);
#else
    asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q st.global.f32 [%0], %1; }" ::"l"(p), "f"(v), "r"((unsigned)on));
#endif
}
// psi(rho, T) = sqrt(2 (p_EOS - rho c_s^2) / G), c = 1 (Sec. 2 and Eq. 21).
__device__ __forceinline__ float eos_psi(float rho, float T, const StepParams& P, bool& bad) {
    const float sT = sqrtf(T);
    float ph = P.k0 - P.k1 * sT;
    ph *= ph;
    const float br = P.b * rho;
    const float p = rho * P.R * T / (1.f - br) - P.a * ph * rho * rho / (1.f + 2.f * br - br * br);
    float arg = P.two_over_G * (p - rho * (1.f / 3.f));
    if (arg < 0.f) {
        bad = true;
        arg = 0.f;
    }
    return sqrtf(arg);
}

// Pulled populations of row y at column x (Eq. 3: f_a(x) = f*_a(x - e_a)).
// Populations whose source lies outside a wall are left 0 and filled by
// Zou-He; with the outflow top the source row is clamped to the top row.
__device__ __forceinline__ void load_row(const StepParams& P, int y, int x, int xm, int xp,
                                         float (&f)[9], float& th) {
    const float* __restrict__ F = P.f_in;
    const int pl = P.plane, pitch = P.pitch;
    int ym = y - 1, yp = y + 1;
    bool okm = true, okp = true;
    if (P.bc == BC_PERIODIC) {
        if (ym < 0) ym += P.Ly;
        if (yp >= P.Ly) yp -= P.Ly;
    } else {
        okm = ym >= 0;
        if (yp >= P.Ly) {
            if (P.bc == BC_TOP_OUTFLOW) yp = P.Ly - 1;
            else okp = false;
        }
    }
    const int rc = y * pitch, rm = ym * pitch, rp = yp * pitch;
    f[0] = __ldg(F + 0 * pl + rc + x);
    f[1] = __ldg(F + 1 * pl + rc + xm);
    f[3] = __ldg(F + 3 * pl + rc + xp);
    f[2] = okm ? __ldg(F + 2 * pl + rm + x) : 0.f;
    f[5] = okm ? __ldg(F + 5 * pl + rm + xm) : 0.f;
    f[6] = okm ? __ldg(F + 6 * pl + rm + xp) : 0.f;
    f[4] = okp ? __ldg(F + 4 * pl + rp + x) : 0.f;
    f[7] = okp ? __ldg(F + 7 * pl + rp + xp) : 0.f;
    f[8] = okp ? __ldg(F + 8 * pl + rp + xm) : 0.f;
    th = __ldg(P.th_in + rc + x);
}

// Zou-He no-slip (u = 0) fill of the unknown populations on the wall rows
// (Sec. 3.1): zero momentum and bounce-back of the normal non-equilibrium
// part. Bottom unknowns 2, 5, 6; top unknowns 4, 7, 8 (walls only).
__device__ __forceinline__ void wall_fill(const StepParams& P, int y, float (&f)[9]) {
    if (P.bc != BC_PERIODIC && y == 0) {
        const float d = 0.5f * (f[1] - f[3]);
        f[2] = f[4];
        f[5] = f[7] - d;
        f[6] = f[8] + d;
    }
    if (P.bc == BC_WALLS && y == P.Ly - 1) {
        const float d = 0.5f * (f[1] - f[3]);
        f[4] = f[2];
        f[7] = f[5] + d;
        f[8] = f[6] - d;
    }
}

// sum_a w_a psi(x + e_a) e_a with w = 1/3 (axis), 1/12 (diagonal), Eq. 7;
// pm, pc, pn point at column x of rows y-1, y, y+1.
__device__ __forceinline__ void psi_sum(const float* pm, const float* pc, const float* pn,
                                        float& sx, float& sy) {
    sx = (pc[1] - pc[-1]) * (1.f / 3.f) + ((pn[1] - pm[-1]) + (pm[1] - pn[-1])) * (1.f / 12.f);
    sy = (pn[0] - pm[0]) * (1.f / 3.f) + ((pn[1] - pm[-1]) + (pn[-1] - pm[1])) * (1.f / 12.f);
}

}  // namespace lbgpu
