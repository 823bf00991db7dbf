// Off-hot-path kernels: initial state, macroscopic fields, FP64 mass sum,
// and the pressure probe run after a step when probes are set (Fig. 3).
#include <algorithm>
#include <type_traits>

#include "lb_internal.h"

namespace lbgpu {

// SMs of a GB300: caps the grids of kernels whose warps loop over the work
// (any number of blocks gives the same result)
constexpr int SMS = 152;

namespace {

__constant__ float kW[9] = {4.f / 9.f, 1.f / 9.f, 1.f / 9.f, 1.f / 9.f, 1.f / 9.f,
                            1.f / 36.f, 1.f / 36.f, 1.f / 36.f, 1.f / 36.f};

// The per-cell kernels below take rows blockIdx.y, blockIdx.y + gridDim.y, ...
// (gridDim.y is capped at the 65535 limit of the launch).
__global__ void init_kernel(const StepParams P, const float* __restrict__ rho0, float* f, float* th) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= P.Lx) return;
    for (int y = blockIdx.y; y < P.Ly; y += gridDim.y) {
        const int i = y * P.pitch + x;
        const float r = rho0[i];
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a * P.plane + i] = kW[a] * r;
        float t = 0.f;
        if (P.bc != BC_PERIODIC && y == 0) t = P.thb[x];
        th[i] = t;
    }
}

// Pass 1 at one cell: the pulled populations give rho, psi and the momentum
// sums.
__device__ __forceinline__ void macro1_cell(const StepParams& P, float* scr, int x, int y) {
    const int xm = x == 0 ? P.Lx - 1 : x - 1;
    const int xp = x == P.Lx - 1 ? 0 : x + 1;
    float f[9], th;
    load_row(P, y, x, xm, xp, f, th);
    wall_fill(P, y, f);
    float rho = 0.f;
#pragma unroll
    for (int a = 0; a < 9; ++a) rho += f[a];
    const float jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
    const float jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
    bool bad = false;
    const float psi = eos_psi(rho, P.Ts + th, P, bad);
    if (bad) atomicOr(&P.acc->err, ERR_EOS);
    const int i = y * P.pitch + x;
    scr[i] = rho;
    scr[P.plane + i] = psi;
    scr[2 * P.plane + i] = jx;
    scr[3 * P.plane + i] = jy;
}

// Pass 2 at one cell.
__device__ __forceinline__ void macro2_cell(const StepParams& P, const float* __restrict__ scr, float* orho,
                                            float* oux, float* ouy, float* oT, int ostride, int x, int y) {
    const int Lx = P.Lx, Ly = P.Ly, pitch = P.pitch;
    const bool periodic = P.bc == BC_PERIODIC;
    const bool wall = !periodic && (y == 0 || y == Ly - 1);
    const float* psi = scr + P.plane;
    const int i = y * pitch + x;
    const float rho = scr[i], ps = psi[i];
    float Fmx = 0.f, Fmy = 0.f;
    if (!wall || P.ghost) {
        const int ym = periodic ? wrap(y - 1, Ly) : (y == 0 ? 0 : y - 1);
        const int yp = periodic ? wrap(y + 1, Ly) : (y == Ly - 1 ? Ly - 1 : y + 1);
        const int xm = x == 0 ? Lx - 1 : x - 1, xp = x == Lx - 1 ? 0 : x + 1;
        float pm[3] = {psi[ym * pitch + xm], psi[ym * pitch + x], psi[ym * pitch + xp]};
        float pc[3] = {psi[y * pitch + xm], ps, psi[y * pitch + xp]};
        float pn[3] = {psi[yp * pitch + xm], psi[yp * pitch + x], psi[yp * pitch + xp]};
        float sx, sy;
        psi_sum(pm + 1, pc + 1, pn + 1, sx, sy);
        Fmx = -P.G * ps * sx;
        Fmy = -P.G * ps * sy;
    }
    float Fx = Fmx, Fy = Fmy;
    if (!wall) {
        if (!periodic && y == 1) Fy += P.gw6 * ps * ps;
        Fy -= P.g * (rho - P.rho_ave);
    }
    const int o = y * ostride + x;
    if (orho) orho[o] = rho;
    if (oux) oux[o] = (scr[2 * P.plane + i] + 0.5f * Fx) / rho;
    if (ouy) ouy[o] = (scr[3 * P.plane + i] + 0.5f * Fy) / rho;
    if (oT) oT[o] = P.Ts + P.th_in[i];
}

// Pass 1: pulled populations -> rho, psi, momentum sums into scratch planes.
__global__ void macro_pass1(const StepParams P, float* scr) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= P.Lx) return;
    for (int y = blockIdx.y; y < P.Ly; y += gridDim.y) macro1_cell(P, scr, x, y);
}

// Pass 2: forces (Eqs. 7, 9, 22) and u = (j + F/2)/rho (Eq. 6).
__global__ void macro_pass2(const StepParams P, const float* __restrict__ scr, float* orho, float* oux,
                            float* ouy, float* oT, int ostride) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= P.Lx) return;
    for (int y = blockIdx.y; y < P.Ly; y += gridDim.y) macro2_cell(P, scr, orho, oux, ouy, oT, ostride, x, y);
}

// The fields of lb_fields in one pass (launch_fields): a block of FIELD_T
// threads marches up a segment of rows, one column per thread, the outer two
// halo. psi of the last rows sits in a four-row shared ring (one barrier per
// row); rho and the momentum sums of a row wait in registers for the row
// above it. Ten planes in, four out, 48 bytes per cell less than with rho, psi
// and j in scratch planes between two kernels: 57 us on 2048^2, 35 of them HBM's;
// bound by its instructions (IEEE divisions and square roots; whole waves of
// taller segments 54.5 us, a row of prefetch 60, shuffles for the ring 55.5).
constexpr int FIELD_T = 128, FIELD_COLS = FIELD_T - 2, FIELD_ROWS = 16;

__global__ void __launch_bounds__(FIELD_T) fields_kernel(const StepParams P, float* __restrict__ orho,
                                                         float* __restrict__ oux, float* __restrict__ ouy,
                                                         float* __restrict__ oT, int ostride) {
    __shared__ float ring[4][FIELD_T];
    const int Lx = P.Lx, Ly = P.Ly;
    const bool periodic = P.bc == BC_PERIODIC;
    const int lc = threadIdx.x;
    const int nstrips = (Lx + FIELD_COLS - 1) / FIELD_COLS;
    const int x0 = blockIdx.x % nstrips * FIELD_COLS;
    const int ys = blockIdx.x / nstrips * FIELD_ROWS, ye = min(ys + FIELD_ROWS, Ly);
    const int x = wrap(x0 - 1 + lc, Lx);
    const int xm = x == 0 ? Lx - 1 : x - 1, xp = x == Lx - 1 ? 0 : x + 1;
    const bool own = lc >= 1 && lc <= FIELD_COLS && x0 + lc - 1 < Lx;
    const int lo = periodic ? ys - 1 : max(ys - 1, 0), hi = periodic ? ye : min(ye, Ly - 1);  // psi rows
    bool bad = false;
    float rho = 0.f, jx = 0.f, jy = 0.f, th = 0.f;  // row r
    for (int L = lo; L <= hi + 1; ++L) {
        const float rho1 = rho, jx1 = jx, jy1 = jy, th1 = th;  // row L - 1
        if (L <= hi) {
            const int y = periodic ? wrap(L, Ly) : L;
            float f[9];
            load_row(P, y, x, xm, xp, f, th);
            wall_fill(P, y, f);
            rho = 0.f;
#pragma unroll
            for (int a = 0; a < 9; ++a) rho += f[a];
            jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]);
            jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8]);
            ring[L & 3][lc] = eos_psi(rho, P.Ts + th, P, bad);
        }
        __syncthreads();
        const int r = L - 1;
        if (r >= ys && r < ye && own) {
            const bool wall = !periodic && (r == 0 || r == Ly - 1);
            const float* pc = &ring[r & 3][lc];
            const float ps = *pc;
            float Fx = 0.f, Fy = 0.f;
            if (!wall || P.ghost) {  // the ghost row beyond a wall copies the wall row
                const float* pm = wall && r == 0 ? pc : &ring[(r - 1) & 3][lc];
                const float* pn = wall && r == Ly - 1 ? pc : &ring[(r + 1) & 3][lc];
                float sx, sy;
                psi_sum(pm, pc, pn, sx, sy);
                Fx = -P.G * ps * sx;
                Fy = -P.G * ps * sy;
            }
            if (!wall) {
                if (!periodic && r == 1) Fy += P.gw6 * ps * ps;
                Fy -= P.g * (rho1 - P.rho_ave);
            }
            const int o = r * ostride + x;
            if (orho) orho[o] = rho1;
            if (oux) oux[o] = (jx1 + 0.5f * Fx) / rho1;
            if (ouy) ouy[o] = (jy1 + 0.5f * Fy) / rho1;
            if (oT) oT[o] = P.Ts + th1;
        }
    }
    if (bad) atomicOr(&P.acc->err, ERR_EOS);
}

// Rows of lx floats between arrays of row stride sp and dp, two arrays (the
// populations' 9 Ly rows, theta's Ly) in one launch; V floats per access. A
// warp takes 4 KB runs of a row, so that short rows do not leave lanes idle
// for long and long ones keep many loads in flight. The fault flags go along
// to host memory (a read of their own costs 4 us more).
template <int V>
__global__ void __launch_bounds__(256) copy_rows(const float* __restrict__ s0, float* __restrict__ d0, int n0,
                                                 const float* __restrict__ s1, float* __restrict__ d1, int n1, int lx,
                                                 int sp, int dp, const unsigned* err, unsigned* err_out) {
    if (err_out && blockIdx.x == 0 && threadIdx.x == 0) *err_out = *err;
    using T = typename std::conditional<V == 4, float4, float>::type;
    constexpr int RUN = 1024;  // floats
    const int lane = threadIdx.x & 31;
    const int runs = (lx + RUN - 1) / RUN;
    const long long total = (long long)(n0 + n1) * runs;
    for (long long w = (long long)blockIdx.x * 8 + (threadIdx.x >> 5); w < total; w += (long long)gridDim.x * 8) {
        const int r = (int)(w / runs), x0 = (int)(w - (long long)r * runs) * RUN;
        const bool second = r >= n0;
        const float* s = (second ? s1 + (size_t)(r - n0) * sp : s0 + (size_t)r * sp) + x0;
        float* d = (second ? d1 + (size_t)(r - n0) * dp : d0 + (size_t)r * dp) + x0;
        const int n = min(RUN, lx - x0) / V;
#pragma unroll 8
        for (int i = lane; i < n; i += 32)
            reinterpret_cast<T*>(d)[i] = __ldg(reinterpret_cast<const T*>(s) + i);
    }
}

// Sums of a few dozen floats without rounding, in FP32: a value is cut into
// multiples of 2^-8, of 2^-23 and the rest by adding and subtracting a power
// of two (extraction, as in Rump, Ogita and Oishi, "Accurate floating-point
// summation", SIAM J. Sci. Comput. 31, 2008), and each part's sum stays
// within 24 bits: exact for up to 64 values with 2^-18 <= |v| < 2^9 or v = 0.
// FP64 adds only the parts' sums.
struct Parts {
    float hi, mid, lo;
    bool ok;  // every value was in that range
    __device__ __forceinline__ void clear() {
        hi = mid = lo = 0.f;
        ok = true;
    }
    __device__ __forceinline__ void add(float v) {
        constexpr float c1 = 49152.f, c2 = 1.5f;  // 1.5 x 2^15, 1.5 x 2^0
        const float h = __fadd_rn(__fadd_rn(v, c1), -c1);
        const float r = __fadd_rn(v, -h);
        const float m = __fadd_rn(__fadd_rn(r, c2), -c2);
        hi = __fadd_rn(hi, h);
        mid = __fadd_rn(mid, m);
        lo = __fadd_rn(lo, __fadd_rn(r, -m));
        const unsigned u = __float_as_uint(v) & 0x7fffffffu;
        ok &= u - 0x36800000u < 0x44000000u - 0x36800000u || u == 0u;
    }
    __device__ __forceinline__ double sum() const { return ((double)lo + (double)mid) + (double)hi; }
};

// Sum of f over the cells and directions, exact up to the FP64 sum of runs of
// 64 values. Warps take rows of the nine planes, four columns per lane and
// load. FP64 adds run at 1/64 of the FP32 rate: one per value took 154 us on
// 2048^2 (22 us from HBM), one per run of 64 takes 28.
__global__ void __launch_bounds__(256) mass_kernel(const StepParams P, const float* __restrict__ f) {
    __shared__ double red[8];
    double t = 0.0;
    const int lane = threadIdx.x & 31;
    const int rows = 9 * P.Ly;  // of pitch floats, pitch a multiple of 32: 16-byte aligned
    for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < rows; r += gridDim.x * 8) {
        const float* p = f + (size_t)r * P.pitch;
        for (int x0 = 4 * lane; x0 < P.Lx; x0 += 16 * 128) {
            const int n = min(16, (P.Lx - x0 + 127) / 128);
            Parts s;
            s.clear();
#pragma unroll 4
            for (int k = 0; k < n; ++k) {
                const int x = x0 + 128 * k;
                const float4 v = __ldg(reinterpret_cast<const float4*>(p + x));
                s.add(v.x);
                s.add(x + 1 < P.Lx ? v.y : 0.f);
                s.add(x + 2 < P.Lx ? v.z : 0.f);
                s.add(x + 3 < P.Lx ? v.w : 0.f);
            }
            if (s.ok) {
                t += s.sum();
            } else {
                for (int k = 0; k < n; ++k)
                    for (int j = 0; j < 4; ++j)
                        if (x0 + 128 * k + j < P.Lx) t += (double)p[x0 + 128 * k + j];
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < 8; ++w) m += red[w];
        atomicAdd(&P.acc->mass, m);
    }
}

}  // namespace

cudaError_t launch_init(const StepParams& P, const float* rho0, float* f, float* th, cudaStream_t st) {
    dim3 grid((P.Lx + 127) / 128, P.Ly < 65535 ? P.Ly : 65535);
    init_kernel<<<grid, 128, 0, st>>>(P, rho0, f, th);
    return cudaGetLastError();
}

cudaError_t launch_macro(const StepParams& P, float* scratch, float* rho, float* ux, float* uy, float* T,
                         int ostride, cudaStream_t st) {
    dim3 grid((P.Lx + 127) / 128, P.Ly < 65535 ? P.Ly : 65535);
    macro_pass1<<<grid, 128, 0, st>>>(P, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    macro_pass2<<<grid, 128, 0, st>>>(P, scratch, rho, ux, uy, T, ostride);
    return cudaGetLastError();
}

// A launch that returns its own status: cudaGetLastError after it would also
// report an earlier call's failure, which these read-backs may follow.
template <class... A, class... B>
static cudaError_t launch(void (*kernel)(A...), int blocks, int threads, cudaStream_t st, B... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    return cudaLaunchKernelEx(&cfg, kernel, A(args)...);
}

cudaError_t launch_copy_state(const float* f_src, float* f_dst, const float* t_src, float* t_dst, int Lx, int Ly,
                              int src_pitch, int dst_pitch, const unsigned* err, unsigned* err_out,
                              cudaStream_t st) {
    const int n0 = f_src ? 9 * Ly : 0, n1 = t_src ? Ly : 0;
    const uintptr_t all = (uintptr_t)f_src | (uintptr_t)f_dst | (uintptr_t)t_src | (uintptr_t)t_dst;
    const long long warps = (long long)(n0 + n1) * ((Lx + 1023) / 1024);
    const int blocks = (int)std::min<long long>((warps + 7) / 8, 16 * SMS);
    if (blocks == 0) return cudaSuccess;
    // (the pitch is a multiple of 32 floats: the other side's rows decide)
    auto kernel = all % 16 == 0 && Lx % 4 == 0 ? copy_rows<4> : copy_rows<1>;
    return launch(kernel, blocks, 256, st, f_src, f_dst, n0, t_src, t_dst, n1, Lx, src_pitch, dst_pitch, err, err_out);
}

// The accumulator records of a batch's instances (table) or of one simulation
// (acc) into out (host memory the device can write), one thread each; reset
// clears the heat-flux sums.
__global__ void collect_acc(const StepParams* __restrict__ table, Acc* acc, int n, Acc* out, int reset) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    Acc* a = table ? table[i].acc : acc;
    out[i] = *a;
    if (reset) a->q_sum = a->q_sum2 = a->q_n = 0.0;
}

cudaError_t launch_collect(const StepParams* table, Acc* acc, int n, Acc* out, bool reset, cudaStream_t st) {
    return launch(collect_acc, (n + 63) / 64, 64, st, table, acc, n, out, reset ? 1 : 0);
}

cudaError_t launch_fields(const StepParams& P, float* rho, float* ux, float* uy, float* T, int ostride,
                          cudaStream_t st) {
    const int nstrips = (P.Lx + FIELD_COLS - 1) / FIELD_COLS, nseg = (P.Ly + FIELD_ROWS - 1) / FIELD_ROWS;
    fields_kernel<<<nstrips * nseg, FIELD_T, 0, st>>>(P, rho, ux, uy, T, ostride);
    return cudaGetLastError();
}

cudaError_t launch_mass(const StepParams& P, const float* f, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(&P.acc->mass, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    mass_kernel<<<std::min(8 * SMS, (9 * P.Ly + 7) / 8), 256, 0, st>>>(P, f);
    return cudaGetLastError();
}

// One block: thread k < n handles probe k. rho^t is the sum of the stored
// post-collision populations (the collision conserves it), T^t = T_s +
// theta^t, and p the Peng-Robinson pressure of Eq. 21 in FP64.
__global__ void probe_kernel(const ProbeArgs A) {
    const int k = threadIdx.x;
    unsigned long long* count = reinterpret_cast<unsigned long long*>(A.ring);
    const unsigned long long s = *count;
    __syncthreads();
    if (k < A.n) {
        const int i = A.y[k] * A.pitch + A.x[k];
        float rho = 0.f;
#pragma unroll
        for (int a = 0; a < 9; ++a) rho += A.f[a * A.plane + i];
        const double r = rho, T = A.Ts + (double)A.th[i];
        const double br = A.b * r, ph = A.k0 - A.k1 * sqrt(T);
        const double p = A.R * r * T / (1.0 - br) - A.a * ph * ph * r * r / (1.0 + 2.0 * br - br * br);
        float* rec = A.ring + 64 + 4 * ((size_t)k * A.cap + (size_t)(s % (unsigned long long)A.cap));
        rec[0] = rho;
        rec[1] = (float)T;
        rec[2] = (float)p;
        rec[3] = 0.f;
    }
    __syncthreads();
    if (k == 0) *count = s + 1;
}

cudaError_t launch_probe(const ProbeArgs& A, cudaStream_t st) {
    probe_kernel<<<1, 32, 0, st>>>(A);
    return cudaGetLastError();
}

}  // namespace lbgpu
