// Host-side declarations shared by the translation units of liblbboil.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lb_device.cuh"

namespace lbgpu {

// Forms of the fused step (lb_march.cuh, lb_tile.cuh); the last, marching with
// six blocks per SM instead of four, for batches only.
enum Form { FORM_MARCH, FORM_TILE24, FORM_TILE16, FORM_TILE14, FORM_TILE12, FORM_COUNT, FORM_MARCH6 = FORM_COUNT };

// Launch shape of the fused step: nstrips x nseg blocks of seg_rows rows
// each; block_x is the form's name to callers (lb_set_launch), with which and
// seg_rows the same shape is chosen again.
struct Launch {
    int form, block_x, seg_rows, nstrips, nseg;
};

cudaError_t step_prepare();  // opt in to the dynamic shared memory
cudaError_t step_occupancy(int form, int* threads, int* blocks_per_sm);
// One step. It leaves the columns' terms of q(t) in P.qpart; with fold it
// adds the previous step's (P.qprev) to the heat-flux statistics, and after
// the last step of a call launch_fold, given the parameters the next step
// would have, adds the last one's.
cudaError_t launch_step(const StepParams& P, const Launch& L, bool fold, cudaStream_t st);
cudaError_t launch_fold(const StepParams& P, cudaStream_t st);

// The forward intermediates of one step that the adjoint's reverse kernels
// read (lb_adjoint.cu), written by the fused step in its recompute mode
// (lb_step_rec.cu) into pitched [Ly][pitch] planes. The gradients drx, dry and
// div v carry the stencil weights; ax, ay are coefficients of K(T), Eq. 18
// (0 on the wall rows; cA, cB and F_m follow from div v, rho and psi); u2-u4
// the RK stage inputs (theta on the wall rows). With out the step itself is written too (f*, theta of the
// next level to P.f_out, P.th_out), and with heat (only with out) q(t) is
// accounted for as the plain step does (fold as there).
struct RecomputeOut {
    float *rho, *psi;
    float *drx, *dry, *divv, *ax, *ay, *u2, *u3, *u4;
};
constexpr int kRecomputePlanes = 10;  // the planes of RecomputeOut, in its order
cudaError_t recompute_prepare();
cudaError_t launch_recompute(const StepParams& P, const RecomputeOut& R, bool out, bool heat, bool fold,
                             const Launch& L, cudaStream_t st);

// The same step over a table of independent instances in one launch (the
// marching forms and the 24-row tiles): block g computes tiles[g] (instance,
// block index within the instance).
cudaError_t batch_prepare();
cudaError_t batch_occupancy(int form, bool shared_k, bool persistent, int* threads, int* blocks_per_sm);
// K non-null: every instance shares the model constants in *K and the kernel
// reads them from its parameters. fold as in launch_step, batch_fold as
// launch_fold (given the table of the step that would follow).
cudaError_t batch_launch(int form, const StepParams* table, const int2* tiles, int nblocks, const StepParams* K,
                         bool fold, cudaStream_t st);
cudaError_t batch_fold(const StepParams* table, int n, cudaStream_t st);

// The persistent batch (lb_batch_persist in lb_step_batch.cu): one cooperative
// launch of a fixed grid advances every instance by nsteps steps; block g
// takes tiles tile_off[g] .. tile_off[g+1]-1 (instance, block index within
// the instance) every step, with a barrier of all blocks between steps
// (arrive: persist_arrive_bytes, zero at launch). A wait gives up after
// wait_limit polls, sets ERR_TIMEOUT in an instance's fault flags and ends
// the block.
constexpr int PERSIST_SUB = 32, PERSIST_PAD = 8;  // first-level counters, a sector each
constexpr size_t persist_arrive_bytes = sizeof(unsigned) * (PERSIST_SUB + 1) * PERSIST_PAD;
struct PersistArgs {
    const StepParams* table;  // [2][n], by step parity
    const int2* tiles;
    const int* tile_off;
    unsigned* arrive;
    int n, nsteps;
    unsigned long long wait_limit;
};
cudaError_t persist_launch(int form, const StepParams* K, const PersistArgs& A, int nblocks, cudaStream_t st);

// Initial state: f* = w_a rho0 (rest equilibrium), theta = 0 with the wall
// rows at their Dirichlet values. rho0 is pitched [Ly][pitch].
cudaError_t launch_init(const StepParams& P, const float* rho0, float* f, float* th, cudaStream_t st);

// Macroscopic fields (rho, u with the level's forces, T; any may be null)
// into outputs with row stride ostride that overlap neither the populations
// nor theta.
cudaError_t launch_fields(const StepParams& P, float* rho, float* ux, float* uy, float* T, int ostride,
                          cudaStream_t st);

// The same in two kernels through scratch (4 pitched planes), after which the
// populations are no longer read: for callers whose outputs may overlay them.
cudaError_t launch_macro(const StepParams& P, float* scratch, float* rho, float* ux, float* uy,
                         float* T, int ostride, cudaStream_t st);

// Discrete adjoint of one step (lb_adjoint.cu): what the current device gives
// the reverse kernels (SMs, blocks per SM), opting them in to their dynamic
// shared memory there; work bytes, reset of the FP64 gradient accumulators,
// one reverse step, and the final read-out (which adds the initial wall row's
// lambda_theta to dJ/d theta_b).
struct ReverseShape {
    int nsm, occ_t, occ_f;
};
cudaError_t adjoint_prepare(ReverseShape* S);
size_t adjoint_work_bytes(const StepParams& P);
cudaError_t adjoint_grads_reset(const StepParams& P, void* work, cudaStream_t st);
// The adjoint of f* travels between reverse steps in two parts: lambda of
// f*_a at cell t is lf[a](t) + lr(t + e_a), where lr is one plane (lambda of
// rho = sum f at the cell that pulls f*_a(t); 0 outside the domain and on
// the wall rows and the outflow top, whose share is already in lf). Zero lf
// and lr are a zero adjoint. The in and out planes are distinct buffers.
// R holds the forward intermediates of the step being reversed (written by
// launch_recompute from the same state).
cudaError_t adjoint_reverse_step(const ReverseShape& S, const StepParams& P, const RecomputeOut& R, void* work,
                                 const float* fstar, const float* theta, const float* lf_in, const float* lt_in,
                                 const float* lr_in, float* lf_out, float* lt_out, float* lr_out, float lq,
                                 cudaStream_t st);
cudaError_t adjoint_grads_finish(const StepParams& P, void* work, const float* lt0, double* dTb_host,
                                 double* dGw_host, cudaStream_t st);

// Populations (9 Ly rows) and theta (Ly rows) of Lx floats between device
// arrays of different row strides; a null source is skipped (not both). With
// err_out (pinned host memory) the flags *err go there.
cudaError_t launch_copy_state(const float* f_src, float* f_dst, const float* t_src, float* t_dst, int Lx, int Ly,
                              int src_pitch, int dst_pitch, const unsigned* err, unsigned* err_out, cudaStream_t st);

// The accumulator records of a batch's instances (table[i].acc), or with no
// table the one at acc, into out, in pinned host memory; reset clears the
// heat-flux sums after reading.
cudaError_t launch_collect(const StepParams* table, Acc* acc, int n, Acc* out, bool reset, cudaStream_t st);

// Record the message lb_last_error() returns on this thread.
void set_last_error(const char* msg);

// acc->mass = sum over cells and directions of f (FP64).
cudaError_t launch_mass(const StepParams& P, const float* f, cudaStream_t st);

// Pressure probes (Fig. 3): after a step, record (rho^t, T^t, p_EOS) at up to
// kProbeMax cells into a device ring (256-byte header whose first 8 bytes
// count the probed steps, then float4 records [probe][cap]).
constexpr int kProbeMax = 8;
struct ProbeArgs {
    const float* f;   // post-collision populations written by the step (level t)
    const float* th;  // theta^t, the step's input temperature
    float* ring;
    int plane, pitch, n, cap;
    int x[kProbeMax], y[kProbeMax];
    double a, b, R, Ts, k0, k1;  // Eq. 21: phi(T) = (k0 - k1 sqrt(T))^2
};
cudaError_t launch_probe(const ProbeArgs& A, cudaStream_t st);

}  // namespace lbgpu
