// The forms of the fused step behind one interface, for the kernels that
// instantiate them (lb_step3.cu: one domain; lb_step_rec.cu: the adjoint's
// recompute mode; lb_step_batch.cu: batches).
#pragma once

#include <algorithm>

#include "lb_march.cuh"
#include "lb_tile.cuh"

namespace lbgpu {

namespace {

template <int MINB>
struct MarchFormT {
    static constexpr int threads = MARCH_T, min_blocks = MINB;
    static constexpr int smem = MarchSmem::total * (int)sizeof(float2);
    template <bool REC, bool CG, bool OUT, bool QF>
    static __device__ __forceinline__ void body(const StepParams& P, const StepParams& C, int block, int fold,
                                                const RecomputeOut* R) {
        march_body<REC, CG, OUT, QF>(P, C, block, fold, R);
    }
};

using MarchForm = MarchFormT<4>;
// 168 registers: no faster at full load (310 us on 4096^2 against 302), but
// half as many blocks again fit, so a batch's tiles come in finer steps of
// one wave (36 domains of 600 x 150: 85 us per step against 101).
using March6 = MarchFormT<6>;

template <int NW, int K>
struct TileForm {
    static constexpr int threads = NW * 32, min_blocks = 1;
    static constexpr int smem = TileShape<NW, K>::slots * (int)sizeof(float2);
    template <bool REC, bool CG, bool OUT, bool QF>
    static __device__ __forceinline__ void body(const StepParams& P, const StepParams& C, int block, int fold,
                                                const RecomputeOut* R) {
        tile_body<NW, K, REC, CG, OUT, QF>(P, C, block, fold, R);
    }
};
using Tile16 = TileForm<16, 1>;
using Tile24 = TileForm<12, 2>;
static_assert(TileShape<16, 1>::out == TILE16_ROWS && TileShape<12, 2>::out == TILE24_ROWS && TILE_OUT == TILE_COLS &&
                  MARCH_COLS == 2 * TILE_COLS,
              "the host's launch shapes use these");

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

// f(form) for the form a launch names (Form in lb_internal.h)
template <class F>
auto with_form(int form, F f) {
    if (form == FORM_TILE16) return f(Tile16{});
    if (form == FORM_TILE24) return f(Tile24{});
    return f(MarchForm{});
}

}  // namespace

}  // namespace lbgpu
