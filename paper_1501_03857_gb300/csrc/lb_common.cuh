// What the kernels share beside a cell's arithmetic: the
// pulled loads, the wall heat flux and its fold, shared-memory checks, launches.
#pragma once

#include "lb_cell.cuh"
#include "lb_internal.h"

namespace lbgpu {

namespace {

constexpr int TILE_W = 64;    // columns a tiled kernel's block computes
constexpr int TILE_ROW = 34;  // float2 slots of its shared rows

// y = v mod n for pipeline rows (|v| is within a few rows of [0, n)).
__device__ __forceinline__ int wrap_row(int v, int n) {
    if (v < 0) v += n;
    if (v >= n) v -= n;
    if ((unsigned)v >= (unsigned)n) v = wrap(v, n);
    return v;
}

// columns of this thread's two cells and their x neighbours
struct Cols {
    int a, am, ap, b, bm, bp;
};

// Pulled populations (Eq. 3: f_a(x) = f*_a(x - e_a)) and theta of row y for
// the two columns. S: rows y - 1 .. y + 1 lie inside. Otherwise the source
// rows are clamped to the domain (the outflow top's zero-gradient condition;
// on wall rows the Zou-He fill replaces what was pulled from there). Coherent
// loads (lb_ldco): the step before, still running when this kernel starts,
// writes these planes.
template <bool S>
__device__ __forceinline__ void load_row2(const StepParams& P, int y, const Cols& c, P2 (&f)[9], P2& th) {
    const float* F = P.f_in;
    const int pl = P.plane, pitch = P.pitch;
    const size_t nF = 9 * (size_t)pl;
    int ym = y - 1, yp = y + 1;
    if (!S) {
        if (P.bc == BC_PERIODIC) {
            if (ym < 0) ym += P.Ly;
            if (yp >= P.Ly) yp -= P.Ly;
        } else {
            ym = max(ym, 0);
            yp = min(yp, P.Ly - 1);
        }
    }
    auto ld = [&](int a, int row, int xa, int xb) {
        const int o = a * pl + row * pitch;
        return P2(lb_ldco(F + (o + xa), F, nF, P.acc), lb_ldco(F + (o + xb), F, nF, P.acc));
    };
    f[0] = ld(0, y, c.a, c.b);
    f[1] = ld(1, y, c.am, c.bm);
    f[3] = ld(3, y, c.ap, c.bp);
    f[2] = ld(2, ym, c.a, c.b);
    f[5] = ld(5, ym, c.am, c.bm);
    f[6] = ld(6, ym, c.ap, c.bp);
    f[4] = ld(4, yp, c.a, c.b);
    f[7] = ld(7, yp, c.ap, c.bp);
    f[8] = ld(8, yp, c.am, c.bm);
    const int o = y * pitch;
    th = P2(lb_ldco(P.th_in + (o + c.a), P.th_in, (size_t)pl, P.acc), lb_ldco(P.th_in + (o + c.b), P.th_in, (size_t)pl, P.acc));
}

__device__ __forceinline__ P2 sel(bool c, P2 a, P2 b) { return P2(c ? a.x() : b.x(), c ? a.y() : b.y()); }

// q(t) of the previous step: its columns' terms (P.qprev) summed in an order
// that no launch shape changes and added to the statistics; by one warp. A
// step writes its own terms and folds its predecessor's, off its critical
// path (a fold kernel follows the last step of a call): folding inside the
// step that made the terms took a counter, two fences and three trips to L2
// after the slowest block, 2.2 us of the 6.9 us of a 100 x 100 step.
__device__ __forceinline__ void fold_heat(const StepParams& P, const int lane) {
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int x = lane; x < P.Lx; x += 512) {  // 16 loads in flight
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = x + 32 * j < P.Lx ? lb_ldcg(P.qprev + x + 32 * j, P.qprev, P.Lx, P.acc) : 0.0;
#pragma unroll
        for (int j = 0; j < 16; ++j) s[j & 3] += v[j];
    }
    double tot = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
    if (lane == 0) {
        // at L2: in the persistent batch another SM may hold an old copy in its L1
        Acc* A = P.acc;
        const double qt = tot * P.qscale;
        __stcg(&A->q_last, qt);
        __stcg(&A->q_sum, __ldcg(&A->q_sum) + qt);
        __stcg(&A->q_sum2, __fma_rn(qt, qt, __ldcg(&A->q_sum2)));
        __stcg(&A->q_n, __ldcg(&A->q_n) + 1.0);
    }
}

// A column's term of q(t) (Sec. 3.2): q_w = -c_v chi rho(x, 0) dT/dy with
// dT/dy = (-3 T_0 + 4 T_1 - T_2) / 2; the constant factors are in P.qscale.
__device__ __forceinline__ double heat_term(float rho0, float t0, float t1, float t2) {
    // (rounded as written, so that every form of the step gives the same bits)
    return __dmul_rn((double)rho0, __fma_rn(-3.0, (double)t0, __fma_rn(4.0, (double)t1, -(double)t2)));
}

// Checked build: a shared-memory pointer whose slots q + lo .. q + hi are
// about to be used, inside the block's n slots; otherwise ERR_BOUNDS is set
// and the accesses go to the first slots instead.
__device__ __forceinline__ float2* smem_at(float2* q, int lo, int hi, float2* base, int n, Acc* acc) {
#ifdef LB_CHECKED
    if (q + lo >= base && q + hi < base + n) return q;
    atomicOr(&acc->err, ERR_BOUNDS);
    return base - lo;
#else
    return q;
#endif
}

// Wait for the work this grid depends on. Every kernel of the step is
// launched to start while its predecessor in the stream drains
// (launch_after), so it waits here before it touches memory; the first
// instruction lets its own successor do the same.
__device__ __forceinline__ void grid_start() {
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Launch on `st` with the launch latency hidden behind the predecessor's last
// blocks (programmatic dependent launch; 0.3 us of a 5 us step).
template <class... A, class... B>
cudaError_t launch_after(void (*kernel)(A...), int blocks, int threads, int smem, cudaStream_t st, B... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, A(args)...);
}

inline cudaError_t allow_smem(const void* kernel, int bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

}  // namespace

}  // namespace lbgpu
