// The fused time step of one domain: stream + collide + forces, RK4
// temperature, wall heat flux, in one kernel. It has two forms with the same
// arithmetic per cell (lb_cell.cuh) and so the same results bit for bit: a
// marching one for domains that fill the GPU (lb_march.cuh) and a tiled one
// for smaller ones (lb_tile.cuh, four tile heights); the host picks by the
// measured times of each (compute_launch in lb_host.cu).
#include "lb_forms.cuh"

namespace lbgpu {

namespace {

template <class F>
__global__ void __launch_bounds__(F::threads, F::min_blocks) lb_step_kernel(const StepParams P, const int fold) {
    grid_start();
    F::template body<false, true, true>(P, P, blockIdx.x, fold, nullptr);
}

// q(t) of the last step of a call (fold_heat): one warp.
__global__ void __launch_bounds__(32) lb_fold_kernel(const StepParams P) {
    grid_start();
    fold_heat(P, threadIdx.x);
}

}  // namespace

cudaError_t step_prepare() {
    cudaError_t e = cudaSuccess;
    for (int form = 0; form < FORM_COUNT && e == cudaSuccess; ++form)
        e = with_form(form, [](auto f) { return allow_smem((const void*)lb_step_kernel<decltype(f)>, decltype(f)::smem); });
    return e;
}

cudaError_t step_occupancy(int form, int* threads, int* blocks_per_sm) {
    return with_form(form, [&](auto f) {
        using F = decltype(f);
        *threads = F::threads;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, lb_step_kernel<F>, F::threads, F::smem);
    });
}

cudaError_t launch_step(const StepParams& P, const Launch& L, bool fold, cudaStream_t st) {
    return with_form(L.form, [&](auto f) {
        using F = decltype(f);
        return launch_after(lb_step_kernel<F>, L.nstrips * L.nseg, F::threads, F::smem, st, P, (int)fold);
    });
}

cudaError_t launch_fold(const StepParams& P, cudaStream_t st) {
    return launch_after(lb_fold_kernel, 1, 32, 0, st, P);
}

}  // namespace lbgpu
