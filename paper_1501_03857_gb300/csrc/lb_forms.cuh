// The forms of the fused step behind one interface, for the kernels that
// instantiate them (lb_step3.cu: one domain; lb_step_rec.cu: the adjoint's
// recompute mode; lb_step_batch.cu: batches).
#pragma once

#include "lb_march.cuh"
#include "lb_tile.cuh"

namespace lbgpu {

namespace {

template <int MINB, bool EARLY>
struct MarchFormT {
    static constexpr int threads = MARCH_T, min_blocks = MINB;
    static constexpr int smem = MarchSmem::total * (int)sizeof(float2);
    template <bool REC, bool OUT, bool QF>
    static __device__ __forceinline__ void body(const StepParams& P, const StepParams& C, int block, int fold,
                                                const RecomputeOut* R) {
        march_body<REC, OUT, QF, EARLY>(P, C, block, fold, R);
    }
};

using MarchForm = MarchFormT<4, true>;
using MarchBatch = MarchFormT<4, false>;
// 168 registers: no faster at full load (310 us on 4096^2 against 302 with the
// loads after the stores in both), but half as many blocks again fit, so a
// batch's tiles come in finer steps of one wave (36 domains of 600 x 150: 85
// us per step against 101).
using March6 = MarchFormT<6, false>;

template <int NW, int K>
struct TileForm {
    static constexpr int threads = NW * 32, min_blocks = 1;
    static constexpr int smem = TileShape<NW, K>::slots * (int)sizeof(float2);
    template <bool REC, bool OUT, bool QF>
    static __device__ __forceinline__ void body(const StepParams& P, const StepParams& C, int block, int fold,
                                                const RecomputeOut* R) {
        tile_body<NW, K, REC, OUT, QF>(P, C, block, fold, R);
    }
};
using Tile24 = TileForm<12, 2>;
using Tile16 = TileForm<16, 1>;
using Tile14 = TileForm<14, 1>;
using Tile12 = TileForm<12, 1>;
static_assert(TileShape<12, 2>::out == TILE24_ROWS && TileShape<16, 1>::out == TILE16_ROWS &&
                  TileShape<14, 1>::out == TILE14_ROWS && TileShape<12, 1>::out == TILE12_ROWS && TILE_OUT == TILE_COLS &&
                  MARCH_COLS == 2 * TILE_COLS,
              "the host's launch shapes use these");

// f(form) for the form a launch names (Form in lb_internal.h)
template <class F>
auto with_form(int form, F f) {
    if (form == FORM_TILE24) return f(Tile24{});
    if (form == FORM_TILE16) return f(Tile16{});
    if (form == FORM_TILE14) return f(Tile14{});
    if (form == FORM_TILE12) return f(Tile12{});
    return f(MarchForm{});
}

}  // namespace

}  // namespace lbgpu
