// The fused step in the adjoint's recompute mode: it writes the forward
// intermediates of the step (RecomputeOut) and, with OUT, the step itself;
// with QF also q(t).
#include "lb_forms.cuh"

namespace lbgpu {

namespace {

template <class F, bool OUT, bool QF>
__global__ void __launch_bounds__(F::threads, F::min_blocks)
    lb_step_recompute(const StepParams P, const __grid_constant__ RecomputeOut R, const int fold) {
    grid_start();
    F::template body<true, OUT, QF>(P, P, blockIdx.x, fold, &R);
}

template <class F, bool OUT, bool QF>
cudaError_t go(const StepParams& P, const RecomputeOut& R, bool fold, int blocks, cudaStream_t st) {
    return launch_after(lb_step_recompute<F, OUT, QF>, blocks, F::threads, F::smem, st, P, R, (int)fold);
}

}  // namespace

cudaError_t recompute_prepare() {
    cudaError_t e = cudaSuccess;
    for (int form = 0; form < FORM_COUNT && e == cudaSuccess; ++form)
        e = with_form(form, [](auto f) {
            using F = decltype(f);
            cudaError_t r = allow_smem((const void*)lb_step_recompute<F, false, false>, F::smem);
            if (r == cudaSuccess) r = allow_smem((const void*)lb_step_recompute<F, true, false>, F::smem);
            if (r == cudaSuccess) r = allow_smem((const void*)lb_step_recompute<F, true, true>, F::smem);
            return r;
        });
    return e;
}

cudaError_t launch_recompute(const StepParams& P, const RecomputeOut& R, bool out, bool heat, bool fold,
                             const Launch& L, cudaStream_t st) {
    if (heat && !out) return cudaErrorInvalidValue;
    return with_form(L.form, [&](auto f) {
        using F = decltype(f);
        const int nb = L.nstrips * L.nseg;
        if (out && heat) return go<F, true, true>(P, R, fold, nb, st);
        if (out) return go<F, true, false>(P, R, false, nb, st);
        return go<F, false, false>(P, R, false, nb, st);
    });
}

}  // namespace lbgpu
