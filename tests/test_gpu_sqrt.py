"""The square root behind psi (sqrt2 in lb_cell.cuh) against CUDA's correctly
rounded one, bit for bit: every mantissa of an odd and an even exponent, the
ends of its range [2^-96, inf) and 2^24 random values in it; the test that
guards the range; and psi of two cells (eos_psi2), which forms psi^2 times a
power of 4, against the general square root of psi^2 itself. Through the public
calls: a uniform vapour so thin that psi^2 is subnormal stays at rest."""

import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lb_cell.cuh"
using namespace lbgpu;
__global__ void go(const float* a, long long n, float* out, float* ref) {
    const long long i = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
    if (i + 1 >= n) return;
    const P2 s = sqrt2(P2(a[i], a[i + 1]));
    out[i] = s.x(), out[i + 1] = s.y();
    ref[i] = __fsqrt_rn(a[i]), ref[i + 1] = __fsqrt_rn(a[i + 1]);
}
__global__ void takes(const float* a, long long n, int* out) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i < n) out[i] = sqrt2_takes(a[i]);
}
__global__ void psi(const StepParams P, const float* rho, const float* T, long long n, float* out, float* ref, float* arg) {
    const long long i = 2 * (blockIdx.x * (long long)blockDim.x + threadIdx.x);
    if (i + 1 >= n) return;
    const P2 r(rho[i], rho[i + 1]), t(T[i], T[i + 1]);
    bool bad = false;
    const P2 s = eos_psi2(r, t, P, bad);
    out[i] = s.x(), out[i + 1] = s.y();
    // Eq. 21 with the same operations, psi^2 = 2 (p - rho / 3) / G unscaled
    P2 ph = fma2(P2::bc(-P.k1), t * rsqrt2(t), P2::bc(P.k0));
    ph = ph * ph;
    const P2 br = P.b * r, d1 = P2::bc(1.f) - br, d2 = fma2(br, P2::bc(2.f) - br, P2::bc(1.f));
    const P2 p = fma2((P.R * r) * t, d2, -(((P.a * ph) * (r * r)) * d1)) * rcp2(d1 * d2);
    const P2 q = fma2(r, P2::bc(-1.f / 3.f), p), a = P.two_over_G * q;
    arg[i] = a.x(), arg[i + 1] = a.y();
    ref[i] = __fsqrt_rn(fmaxf(a.x(), 0.f)), ref[i + 1] = __fsqrt_rn(fmaxf(a.y(), 0.f));
    if (bad != (q.x() > 0.f || q.y() > 0.f)) out[i] = -1.f;
}
extern "C" int run_psi(const float* rho, const float* T, long long n, double G, float* out, float* ref, float* arg) {
    StepParams P = {};
    const double a = 3.0 / 49.0, b = 2.0 / 21.0, omega = 0.344, Tc = 0.0778 * a / (0.45724 * b);
    const double kappa = 0.37464 + 1.54226 * omega - 0.26992 * omega * omega;
    P.a = (float)a, P.b = (float)b, P.R = 1.f;
    P.k0 = (float)(1.0 + kappa), P.k1 = (float)(kappa / sqrt(Tc));
    P.G = (float)G, P.two_over_G = (float)(2.0 / G);
    set_pairs(P);
    if (n > 0) psi<<<(unsigned)((n / 2 + 255) / 256), 256>>>(P, rho, T, n, out, ref, arg);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run(const float* a, long long n, float* out, float* ref) {
    if (n > 0) go<<<(unsigned)((n / 2 + 255) / 256), 256>>>(a, n, out, ref);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_takes(const float* a, long long n, int* out) {
    if (n > 0) takes<<<(unsigned)((n + 255) / 256), 256>>>(a, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1501_03857_gb300 import build
    d = tmp_path_factory.mktemp("sqrt")
    src, so = str(d / "roots.cu"), str(d / "roots.so")
    open(src, "w").write(SOURCE)
    subprocess.run([build.nvcc_path()] + build.ARCH + ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                   "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), src, "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def psi(rho, T, G):
        """psi, the reference and its psi^2, of the given states."""
        r, t = torch.from_numpy(rho).cuda(), torch.from_numpy(T).cuda()
        o = [torch.empty_like(r) for _ in range(3)]
        torch.cuda.synchronize()
        assert r.numel() % 2 == 0
        p = lambda x: ctypes.c_void_p(x.data_ptr())
        assert lib.run_psi(p(r), p(t), ctypes.c_longlong(r.numel()), ctypes.c_double(G), *[p(x) for x in o]) == 0
        return [x.cpu().numpy() for x in o]

    def compare(bits):
        """Mismatches over the given bit patterns (an even number of them)."""
        a = torch.from_numpy(bits.astype(np.uint32).view(np.float32)).cuda()
        out, ref = torch.empty_like(a), torch.empty_like(a)
        torch.cuda.synchronize()
        assert a.numel() % 2 == 0
        p = lambda t: ctypes.c_void_p(t.data_ptr())
        assert lib.run(p(a), ctypes.c_longlong(a.numel()), p(out), p(ref)) == 0
        return int((out.view(torch.int32) != ref.view(torch.int32)).sum())

    def takes(bits):
        a = torch.from_numpy(bits.astype(np.uint32).view(np.float32)).cuda()
        out = torch.empty(a.numel(), dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.run_takes(ctypes.c_void_p(a.data_ptr()), ctypes.c_longlong(a.numel()), ctypes.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy().astype(bool)
    return compare, takes, psi


LOW, INF = (127 - 96) << 23, 0x7f800000  # bits of 2^-96 and infinity


def test_square_roots_are_correctly_rounded(roots):
    compare, _, _ = roots
    assert compare(np.arange(127 << 23, 129 << 23)) == 0           # [1, 4)
    assert compare(np.arange(LOW, LOW + (2 << 23))) == 0           # the first two binades
    assert compare(np.arange(INF - (2 << 23), INF)) == 0           # the last two
    assert compare(np.random.default_rng(1).integers(LOW, INF, 1 << 24)) == 0


def test_range_of_the_paired_square_root(roots):
    _, takes, _ = roots
    inside = np.array([LOW, LOW + 1, 0x3f800000, INF - 1])
    outside = np.array([0, 1, 0x00800000, LOW - 1, INF, INF + 1, 0x7fffffff, 0x80000000, 0xbf800000, 0xff800000, 0xffffffff])
    assert takes(inside).all() and not takes(outside).any()


@pytest.mark.parametrize("form", [(64, 0), (128, 0), (256, 0)])
def test_vapour_with_subnormal_psi2_stays_at_rest(form):
    """rho = 1.5e-38: psi^2 = 2 (p - rho / 3) / G is about 8e-39, subnormal.
    Uniform and at rest without gravity: a step changes nothing but the last
    bits of the subnormal populations (multiples of 1.4e-45)."""
    from paper_1501_03857_gb300 import lb
    cfg = lb.Config(Lx=120, Ly=30, bc_y=lb.BC_PERIODIC, g=0.0)
    sim = lb.Simulation(cfg, rho0=np.full((30, 120), 1.5e-38, np.float32))
    sim.set_launch(*form)
    f0, th0 = sim.get_state()
    sim.step(3)
    sim.sync()
    f, th = sim.get_state()
    sim.close()
    assert np.isfinite(f).all() and np.isfinite(th).all()
    # three steps of some tens of operations, each within one unit of 2^-149
    assert np.abs(f.astype(np.float64) - f0).max() <= 300 * 2.0 ** -149
    assert np.abs(th).max() <= 1e-6


@pytest.mark.parametrize("G", [-1.0, -2.0, -4.0 ** -20, -0.3, -4096.0, -1e-30, -1e30])
def test_psi_equals_the_general_square_root(roots, G):
    """The same bits wherever psi^2 unscaled is a normal number, zero, infinite
    or NaN as the scaled one is: everywhere if 2 / G is a power of two from 1
    up to 2^41, else where it is normal or p - rho / 3 is no number or 0. psi^2 <
    0 is told by p > rho / 3."""
    _, _, psi = roots
    rng = np.random.default_rng(3)
    n = 1 << 20
    rho = (2.0 ** rng.uniform(-149, 126, n)).astype(np.float32)
    rho[::2] = (2.0 ** rng.uniform(-8, 5, n // 2)).astype(np.float32)  # the model's own range
    rho[:8] = [0.0, 10.5, 25.3492424, 25.3492432, 1e-45, np.inf, np.nan, 3e38]
    T = rng.uniform(0.02, 0.2, n).astype(np.float32)
    out, ref, arg = psi(rho, T, G)
    exact = np.ones(n, bool)
    if -G not in (1.0, 2.0, 4.0 ** -20):
        exact = (np.abs(arg) >= 2.0 ** -126) & np.isfinite(arg) | np.isnan(arg) | (rho == 0)
    assert exact.sum() > n // 2 and (ref > 0).sum() > n // 4
    assert np.array_equal(out[exact].view(np.int32), ref[exact].view(np.int32))
    assert (out[~exact] >= 0).all()
