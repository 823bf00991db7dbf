// The forms of the fused step behind one interface, for the kernels that
// instantiate them (lb_step3.cu: one domain; lb_step_rec.cu: the adjoint's
// recompute mode; lb_step_batch.cu: batches).
#pragma once

#include <algorithm>

#include "lb_march.cuh"

namespace lbgpu {

namespace {

struct MarchForm {
    static constexpr int threads = MARCH_T, min_blocks = 4;
    static constexpr int smem = MarchSmem::total * (int)sizeof(float2);
    template <bool REC, bool CG, bool OUT, bool QF>
    static __device__ __forceinline__ void body(const StepParams& P, const StepParams& C, int block, int fold,
                                                const RecomputeOut* R) {
        march_body<REC, CG, OUT, QF>(P, C, block, fold, R);
    }
};

static_assert(MARCH_COLS == 2 * TILE_COLS, "the host's launch shapes use this");

template <class... A, class... B>
cudaError_t launch_after(void (*kernel)(A...), int blocks, int threads, int smem, cudaStream_t st, B... args) {
    kernel<<<blocks, threads, smem, st>>>(A(args)...);
    return cudaGetLastError();
}

inline cudaError_t allow_smem(const void* kernel, int bytes) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// f(form) for the form a launch names (Form in lb_internal.h)
template <class F>
auto with_form(int form, F f) {
    (void)form;
    return f(MarchForm{});
}

}  // namespace

}  // namespace lbgpu
