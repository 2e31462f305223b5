// Internal declarations of the surrogate network's kernels (BF16 tensor-core
// GEMM, training step, inference, input transforms, the acceptance gate).
// Shared by mlp_kernels.cu and the host
// API in surrogate_api.cu.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace sg {

typedef __nv_bfloat16 bf16;

// Status bits written by the kernels.
constexpr unsigned kStatusTimeout = 1u;   // an mbarrier wait ran out of iterations
constexpr unsigned kStatusNonFinite = 2u; // the loss met NaN or Inf

// One GEMM, C = A B^T (A: M x K, B: N x K, both K contiguous; C FP32).
struct GemmArgs {
  const bf16* A;
  const bf16* B;
  int lda, ldb;
  int M, N, K;
  float* C;
  int ldc;
  unsigned* status;
};

// Requirements (checked by the host API): K, lda, ldb multiples of 8; 16-byte
// aligned base pointers.
cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t s);
size_t gemm_smem_bytes(int bn);

constexpr int kIn = 7, kInPad = 16, kOut = 4, kOutPad = 16, kHidden = 4;

// Per-feature transform: v -> ((log v if the bit is set) - mean) / scale.
struct Xform {
  float mean[kInPad];
  float scale[kInPad];
  int log_mask;
  int dim;
};

// Raw rows x [n][7] -> transformed BF16 rows X [n][16] (columns 7.. zero)
// and FP32 transformed columns Xf [7][ldx] (either may be null).
cudaError_t launch_prep_inputs(const float* x, int n, const Xform& xf, bf16* X, float* Xf, int ldx,
                               cudaStream_t s);
// Raw targets y [n][4] -> transformed FP32 T [n][4].
cudaError_t launch_prep_targets(const float* y, int n, const Xform& yf, float* T, cudaStream_t s);
// Parameter block of one member: for each layer l, Wt_l [out][in] then b_l [out].
struct Layout {
  int nin[kHidden + 1], nout[kHidden + 1];
  long long w_off[kHidden + 1], b_off[kHidden + 1];
  long long total;
};
// `steps` training steps of every member, two launches each: forward pass,
// loss and back-propagation of a minibatch; weight gradients and Adam.
//  X [n][16] BF16, T [n][4]: transformed training rows; a minibatch of `rows`
//  rows per member is drawn with replacement by a counter-based hash of (seed,
//  member, *d_step, row), or (direct) is rows 0 .. rows - 1.
//  Loss 1/(4 rows) sum w (y - t)^2; loss [members][train_loss_parts(rows)]
//  receives its parts.
//  Adam, bias-corrected, at step *d_step + 1; d_sched (may be null): {first
//  step, step count} of the current training call, over which lr decays along
//  a half cosine; *d_step advances by `steps` at the end.  grads_only: the gradients go to g and
//  nothing is updated.
//  Wb (layout of p) and WbT (layer-wise transposes): BF16 copies of p.
//  Xt [members][16][rows], Ht, dZt [members][H][rows], dYt, dYft
//  [members][16][rows]: workspace.
struct TrainArgs {
  int steps, members, rows, grads_only;
  Layout L;
  const bf16* X;
  const float* T;
  int n, direct;
  unsigned long long seed;
  const float* w;
  float *p, *g, *m, *v;
  bf16 *Wb, *WbT;
  bf16* Xt;
  bf16* Ht[kHidden];
  bf16* dZt[kHidden];
  bf16* dYt;
  float* dYft;
  double* loss;
  float lr, beta1, beta2, eps;
  long long* d_step;
  const long long* d_sched;
  unsigned* status;
};
cudaError_t launch_train_step(const TrainArgs& t, cudaStream_t s);
int train_loss_parts(int rows);
// d_sched = {*d_step, steps}: the start of a training call of `steps` steps.
cudaError_t launch_schedule_begin(const long long* d_step, long long* d_sched, long long steps,
                                  cudaStream_t s);
// BF16 copies of the parameters without an update.
cudaError_t launch_cast_params(const float* p, const Layout& L, int members, bf16* Wb, bf16* WbT,
                               cudaStream_t s);
// Allow the network's kernels (training and inference) their shared memory on
// the current device: called for each handle that is made, on its device.
cudaError_t allow_network_smem();
// Outputs of every member for n raw queries x [n][7]: Y [m][n][4] (FP32,
// transformed outcomes).  One kernel runs all five layers of a 128-row tile.
cudaError_t launch_forward(const float* x, int n, const Xform& xf, const float* p, const bf16* Wb,
                           const Layout& L, int members, float* Y, unsigned* status,
                           cudaStream_t s);

// The answers of n queries from the member outputs Y [m][n][4]: the mean
// [n][4] and standard deviation [n][4] over members of the inverse-
// transformed outcomes, and (accept not null) the acceptance gate: inside
// the per-feature box [lo, hi] of the training inputs, within nn_cut of a
// training point (transformed space; Xt [7][ldt], nt points), and relative
// ensemble spread sd/|mean| of outcome 0 at most tau and of outcome 1 at
// most tau_v.  *status_out receives *status.
struct GateArgs {
  const float* x;
  const float* Y;
  int n, members;
  Xform xin, xout;
  const float* Xt;
  int nt, ldt;
  const float* lo;
  const float* hi;
  float nn_cut, tau, tau_v;
  float* mean;
  float* sd;
  int* accept;
  const unsigned* status;
  unsigned* status_out;
};
cudaError_t launch_answer(const GateArgs& a, cudaStream_t s);

}  // namespace sg
