// Many independent simulations in one launch (the boiling-curve batch): one
// launch per step, or one cooperative launch for a run of steps. The
// marching form at four and at six blocks per SM and the taller tiles of the
// fused step (lb_march.cuh, lb_tile.cuh).
#include "lb_forms.cuh"

namespace lbgpu {

namespace {

// Copy an instance's parameter record to shared memory; the block's threads
// need a barrier before they use it.
template <int BD>
__device__ __forceinline__ void copy_params(const StepParams* __restrict__ src, StepParams& dst) {
    constexpr int NW = (int)(sizeof(StepParams) / sizeof(int));
    static_assert(sizeof(StepParams) % sizeof(int) == 0, "StepParams is copied as ints");
    for (int k = threadIdx.x; k < NW; k += BD)
        reinterpret_cast<int*>(&dst)[k] = __ldg(reinterpret_cast<const int*>(src) + k);
}

// One step of the batch: block g computes tiles[g] (instance, block index
// within it), with every model constant from the instance's record (SK
// false), or with the constants that all instances share in K, in the
// parameter bank (the table then supplies each instance's buffers, sizes,
// launch shape, wettability and rho_ave). The record is fetched before the
// block waits for the step before it: no kernel writes the table, and a copy
// into it is complete before the launch that follows it starts.
template <class F, bool SK>
__global__ void __launch_bounds__(F::threads, F::min_blocks)
    lb_step_batch(const StepParams K, const StepParams* __restrict__ table, const int2* __restrict__ tiles, const int fold) {
    __shared__ StepParams sP;
    asm volatile("griddepcontrol.launch_dependents;");
    const int2 tl = __ldg(tiles + blockIdx.x);
    copy_params<F::threads>(table + tl.x, sP);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    F::template body<false, true, true>(sP, SK ? K : sP, tl.y, fold, nullptr);
}

// q(t) of every instance's last step of a call: one warp per instance, from
// the parameters of the step that would follow.
__global__ void __launch_bounds__(32) lb_batch_fold(const StepParams* __restrict__ table) {
    grid_start();
    if (table[blockIdx.x].bc != BC_PERIODIC) fold_heat(table[blockIdx.x], threadIdx.x);
}

// ---------------------------------------------------------------------------
// The persistent batch: one launch advances every instance by `nsteps` steps.
//
// The instances' tiles (what one block of the per-step kernel computes) are
// dealt out to a fixed, co-resident grid (a cooperative launch); block g takes
// tiles tile_off[g] .. tile_off[g+1]-1 in that order, step after step, and the
// blocks meet at a barrier between steps: a tile's pulled rows and the strips
// beside it are then complete (read after write), and no tile still reads the
// buffer the step writes (write after read). The barrier counts in two levels
// (arrive: PERSIST_SUB counters, the last arrival at each adds to a root; all
// zero at launch). A wait polls the root at most `wait_limit` times; a block
// that gives up sets ERR_TIMEOUT in its first instance's fault flags and
// leaves the kernel, which lets every block waiting on it give up in turn, so
// the launch always ends. The step's loads of its input state are coherent
// (lb_ldco), so after the acquiring fence and the block's barrier they see the
// other SMs' writes; every tile runs the same step as the per-step kernel, so
// results are bit-identical to it.
//
// Waiting only for the tile's own instance, as this kernel did before, lets
// the instances drift apart, and blocks at different stages of their march
// evict each other's instructions (36 domains of 600 x 150: no-instruction
// stalls 1.8 cycles per issue against 0.4 per-step, 99 us per step against 92
// with the common barrier; 48 uneven domains 151 against 144).
// ---------------------------------------------------------------------------

template <class F, bool SK>
__global__ void __launch_bounds__(F::threads, F::min_blocks) lb_batch_persist(const StepParams K, const PersistArgs A) {
    constexpr int BD = F::threads;
    __shared__ StepParams sP;
    __shared__ bool s_go;
    const int t0 = A.tile_off[blockIdx.x], m = A.tile_off[blockIdx.x + 1] - t0;
    const unsigned G = gridDim.x, nsub = min(G, (unsigned)PERSIST_SUB), sub = blockIdx.x % nsub;
    const unsigned size = (G - sub + nsub - 1) / nsub;  // blocks that count at this block's counter
    unsigned* const root = A.arrive + PERSIST_SUB * PERSIST_PAD;
    for (int k = 0; k < A.nsteps; ++k) {
        if (k > 0) {
            if (threadIdx.x == 0) {
                bool go = false;
                for (unsigned long long it = 0;; ++it) {
                    unsigned v;
                    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(root) : "memory");
                    go = v >= (unsigned)k * nsub;
                    if (go || it >= A.wait_limit) break;
                    __nanosleep(32);
                }
                if (!go) atomicOr(&A.table[A.tiles[t0].x].acc->err, ERR_TIMEOUT);
                asm volatile("fence.acq_rel.gpu;" ::: "memory");
                s_go = go;
            }
            __syncthreads();
            if (!s_go) return;
        }
        for (int j = 0; j < m; ++j) {
            const int2 tl = A.tiles[t0 + j];
            if (m > 1 || k == 0) {
                copy_params<BD>(A.table + (k & 1) * A.n + tl.x, sP);
                __syncthreads();
            }
            F::template body<false, true, true>(sP, SK ? K : sP, tl.y, k > 0, nullptr);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            __threadfence();
            if (atomicAdd(A.arrive + sub * PERSIST_PAD, 1u) == (unsigned)(k + 1) * size - 1u) {
                __threadfence();
                atomicAdd(root, 1u);
            }
            if (m == 1) {  // the other parity's record is this one with its buffers exchanged
                const StepParams P = sP;
                sP.f_in = P.f_out;
                sP.f_out = const_cast<float*>(P.f_in);
                sP.th_in = P.th_out;
                sP.th_out = const_cast<float*>(P.th_in);
                sP.qpart = const_cast<double*>(P.qprev);
                sP.qprev = P.qpart;
            }
        }
        // (the next step's first barrier, at the wait above, orders sP)
    }
}

template <class F>
struct BatchForm {
    static cudaError_t prepare() {
        cudaError_t e = allow_smem((const void*)lb_step_batch<F, false>, F::smem);
        if (e == cudaSuccess) e = allow_smem((const void*)lb_step_batch<F, true>, F::smem);
        if (e == cudaSuccess) e = allow_smem((const void*)lb_batch_persist<F, false>, F::smem);
        if (e == cudaSuccess) e = allow_smem((const void*)lb_batch_persist<F, true>, F::smem);
        return e;
    }
    // a cooperative launch: the runtime refuses it unless every block can be
    // resident at once, which the blocks' waits on one another need
    template <bool SK>
    static cudaError_t persist(const StepParams& K, const PersistArgs& A, int nblocks, cudaStream_t st) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(nblocks);
        cfg.blockDim = dim3(F::threads);
        cfg.dynamicSmemBytes = F::smem;
        cfg.stream = st;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, lb_batch_persist<F, SK>, K, A);
    }
};

template <class F>
auto with_batch_form(int form, F f) {
    if (form == FORM_TILE24) return f(Tile24{});
    if (form == FORM_MARCH6) return f(March6{});
    return f(MarchBatch{});
}

}  // namespace

cudaError_t batch_prepare() {
    cudaError_t e = BatchForm<MarchBatch>::prepare();
    if (e == cudaSuccess) e = BatchForm<March6>::prepare();
    return e == cudaSuccess ? BatchForm<Tile24>::prepare() : e;
}

cudaError_t batch_occupancy(int form, bool shared_k, bool persistent, int* threads, int* n) {
    return with_batch_form(form, [&](auto f) {
        using F = decltype(f);
        const void* k = persistent ? (shared_k ? (const void*)lb_batch_persist<F, true> : (const void*)lb_batch_persist<F, false>)
                                   : (shared_k ? (const void*)lb_step_batch<F, true> : (const void*)lb_step_batch<F, false>);
        *threads = F::threads;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, F::threads, F::smem);
    });
}

cudaError_t batch_launch(int form, const StepParams* table, const int2* tiles, int nblocks, const StepParams* K,
                         bool fold, cudaStream_t st) {
    const StepParams k0 = K ? *K : StepParams{};
    return with_batch_form(form, [&](auto f) {
        using F = decltype(f);
        auto kernel = K ? lb_step_batch<F, true> : lb_step_batch<F, false>;
        return launch_after(kernel, nblocks, F::threads, F::smem, st, k0, table, tiles, (int)fold);
    });
}

cudaError_t batch_fold(const StepParams* table, int n, cudaStream_t st) {
    return launch_after(lb_batch_fold, n, 32, 0, st, table);
}

cudaError_t persist_launch(int form, const StepParams* K, const PersistArgs& A, int nblocks, cudaStream_t st) {
    const StepParams k0 = K ? *K : StepParams{};
    return with_batch_form(form, [&](auto f) {
        using B = BatchForm<decltype(f)>;
        return K ? B::template persist<true>(k0, A, nblocks, st) : B::template persist<false>(k0, A, nblocks, st);
    });
}

}  // namespace lbgpu
