// Many independent simulations in one launch (the boiling-curve batch): one
// launch per step, or one cooperative launch for a run of steps. The
// marching form and the taller tiles of the fused step (lb_march.cuh,
// lb_tile.cuh).
#include "lb_forms.cuh"

namespace lbgpu {

namespace {

// The blocks of instance i are [block_off[i], block_off[i+1]); each block copies its instance's parameter record to shared memory (sP) and returns the
// block's index within its instance.
template <int BD>
__device__ __forceinline__ int batch_instance(const StepParams* __restrict__ table, const int* __restrict__ block_off,
                                              int n, StepParams& sP) {
    __shared__ int s_inst;
    if (threadIdx.x == 0) {
        int lo = 0, hi = n - 1;  // largest i with block_off[i] <= blockIdx.x
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (block_off[mid] <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        s_inst = lo;
    }
    __syncthreads();
    const int inst = s_inst;
    constexpr int NW = (int)(sizeof(StepParams) / sizeof(int));
    static_assert(sizeof(StepParams) % sizeof(int) == 0, "StepParams is copied as ints");
    for (int k = threadIdx.x; k < NW; k += BD)
        reinterpret_cast<int*>(&sP)[k] = __ldg(reinterpret_cast<const int*>(table + inst) + k);
    __syncthreads();
    return (int)blockIdx.x - block_off[inst];
}

// The batch with every model constant from the instance's record (SK false),
// or with the constants that all instances share in K, in the parameter bank
// (the table then supplies each instance's buffers, sizes, launch shape,
// wettability and rho_ave).
template <class F, bool SK>
__global__ void __launch_bounds__(F::threads, F::min_blocks)
    lb_step_batch(const StepParams K, const StepParams* __restrict__ table, const int* __restrict__ block_off, const int n,
                  const int fold) {
    __shared__ StepParams sP;
    grid_start();
    const int b = batch_instance<F::threads>(table, block_off, n, sP);
    F::template body<false, false, true, true>(sP, SK ? K : sP, b, fold, nullptr);
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
// The instances' tiles (a pair of column strips x a segment of rows, the
// unit one block of the per-step kernel computes) are dealt out to a fixed,
// co-resident grid (a cooperative launch); block g takes tiles
// tile_off[g] .. tile_off[g+1]-1 in that order, step after step. A tile may
// start step k once every tile of its instance has finished step k-1:
// its pulled rows and the strips beside it are then complete (read after
// write), and no tile of the instance still reads the buffer step k writes
// (write after read). arrive[i] counts the tiles of instance i that have
// finished a step since the launch began (zeroed before each launch), so
// the wait is arrive[i] >= k * ntiles[i]. The wait spins at most
// `wait_limit` polls (with a short sleep between them); a block that gives
// up sets ERR_TIMEOUT in its instance's fault flags and leaves the kernel,
// which lets every block waiting on it give up in turn, so the launch always
// ends. The step's input state is read with plain loads, which after the
// acquiring wait and the barrier see the other SMs' writes (the read-only
// path could serve copies cached before them), and every tile runs the same
// step body as the per-step kernel, so results are bit-identical to it.
// ---------------------------------------------------------------------------

// Poll *p until it reaches `target`, at most `limit` times; true if reached.
__device__ __forceinline__ bool wait_at_least(const unsigned* p, unsigned target, unsigned long long limit) {
    for (unsigned long long it = 0;; ++it) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v >= target) return true;
        if (it >= limit) return false;
        __nanosleep(64);
    }
}

// The most tiles one block of the persistent batch schedules by readiness
// (more than this many are taken in order).
constexpr int PERSIST_MAX_TILES = 64;

template <class F, bool SK>
__global__ void __launch_bounds__(F::threads, F::min_blocks) lb_batch_persist(const StepParams K, const PersistArgs A) {
    constexpr int BD = F::threads;
    __shared__ StepParams sP;
    __shared__ int s_next[PERSIST_MAX_TILES];  // next step of each of the block's tiles
    __shared__ int s_pick;
    const int t0 = A.tile_off[blockIdx.x], t1 = A.tile_off[blockIdx.x + 1];
    const int m = t1 - t0;
    const bool by_ready = m <= PERSIST_MAX_TILES;
    for (int j = threadIdx.x; j < PERSIST_MAX_TILES; j += BD) s_next[j] = 0;
    __syncthreads();
    // whether tile j may run its next step: every tile of its instance has
    // finished the previous one
    auto ready = [&](int j, int k) {
        const int inst = A.tiles[t0 + j].x;
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(A.arrive + inst) : "memory");
        return k == 0 || v >= (unsigned)k * (unsigned)A.ntiles[inst];
    };
    int last = m - 1, done_in_order = 0;
    for (;;) {
        // thread 0 picks the next tile: with few tiles per block the first
        // ready one after the last tile run (round robin), so a block never
        // idles while one of its tiles can go on; otherwise the tiles in
        // order, step after step. -2: all done; -3: a wait ran out.
        if (threadIdx.x == 0) {
            int pick = -2;
            if (by_ready) {
                unsigned long long polls = 0;
                for (;;) {
                    bool left = false;
                    pick = -1;
                    for (int d = 1; d <= m; ++d) {
                        const int j = (last + d) % m;
                        if (s_next[j] >= A.nsteps) continue;
                        left = true;
                        if (ready(j, s_next[j])) {
                            pick = j;
                            break;
                        }
                    }
                    if (!left) {
                        pick = -2;
                        break;
                    }
                    if (pick >= 0) break;
                    if (polls++ >= A.wait_limit) {
                        pick = -3;
                        break;
                    }
                    __nanosleep(64);
                }
            } else if (done_in_order < m * A.nsteps) {
                const int j = done_in_order % m, k = done_in_order / m;
                pick = wait_at_least(A.arrive + A.tiles[t0 + j].x, (unsigned)k * (unsigned)A.ntiles[A.tiles[t0 + j].x],
                                     k == 0 ? 0ull : A.wait_limit) || k == 0 ? j : -3;
                if (pick >= 0) s_next[0] = k;  // the step to run
            }
            if (pick == -3) {  // latch the timeout on an unfinished tile's instance
                for (int j = 0; j < m; ++j)
                    if (!by_ready || s_next[j] < A.nsteps) {
                        atomicOr(&A.table[A.tiles[t0 + j].x].acc->err, ERR_TIMEOUT);
                        break;
                    }
            }
            s_pick = pick;
        }
        __syncthreads();
        const int pick = s_pick;
        if (pick < 0) return;  // all done, or given up
        const int k = by_ready ? s_next[pick] : s_next[0];
        const int2 tl = A.tiles[t0 + pick];
        const StepParams* src = A.table + (k & 1) * A.n + tl.x;
        constexpr int NW = (int)(sizeof(StepParams) / sizeof(int));
        for (int w = threadIdx.x; w < NW; w += BD)
            reinterpret_cast<int*>(&sP)[w] = __ldg(reinterpret_cast<const int*>(src) + w);
        __syncthreads();
        F::template body<false, true, true, true>(sP, SK ? K : sP, tl.y, k > 0, nullptr);
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            atomicAdd(A.arrive + tl.x, 1u);
            if (by_ready) ++s_next[pick];
            else ++done_in_order;
            last = pick;
        }
        __syncthreads();
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
    return f(MarchForm{});
}

}  // namespace

cudaError_t batch_prepare() {
    cudaError_t e = BatchForm<MarchForm>::prepare();
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

cudaError_t batch_launch(int form, const StepParams* table, const int* block_off, int n, int nblocks,
                         const StepParams* K, bool fold, cudaStream_t st) {
    const StepParams k0 = K ? *K : StepParams{};
    return with_batch_form(form, [&](auto f) {
        using F = decltype(f);
        auto kernel = K ? lb_step_batch<F, true> : lb_step_batch<F, false>;
        return launch_after(kernel, nblocks, F::threads, F::smem, st, k0, table, block_off, n, (int)fold);
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
