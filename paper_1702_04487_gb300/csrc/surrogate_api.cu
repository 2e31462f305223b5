// Host side of the surrogate: ensemble parameters, training steps, prediction
// with the acceptance gate, and the C ABI of include/surrogate.h.
#include <math.h>
#include <stdarg.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "../../include/surrogate.h"
#include "mlp.cuh"

using namespace sg;

namespace {

thread_local char g_err[512] = "";

ij_status fail(ij_status st, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return st;
}

#define CUDA_TRY(x)                                                                  \
  do {                                                                               \
    cudaError_t e_ = (x);                                                            \
    if (e_ != cudaSuccess) return fail(IJ_ERR_CUDA, "%s: %s", #x, cudaGetErrorString(e_)); \
  } while (0)

unsigned long long mix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

}  // namespace

struct sg_handle_s {
  sg_config cfg;
  int K = 1, H = 16, bm = 16;
  Layout L;
  cudaStream_t stream = nullptr;
  ij_alloc_fn alloc = nullptr;
  ij_free_fn free_fn = nullptr;
  void* ctx = nullptr;
  std::vector<void*> blocks;
  // parameters [K][P]
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
  bf16 *Wb = nullptr, *WbT = nullptr;
  // transforms and gate
  Xform xin, xout;
  float tau = 0.01f, tau_v = 0.01f, nn_cut = 0.0f;
  float lo[kIn], hi[kIn];
  float *d_lo = nullptr, *d_hi = nullptr, *d_w = nullptr;
  // training data
  int n_train = 0;
  bf16* X = nullptr;
  float *T = nullptr, *Xt = nullptr;  // Xt: transformed FP32 columns [7][ldt], for the gate
  int ldt = 0, train_cap = 0;
  // minibatch workspace (TrainArgs)
  bf16 *Xt_b = nullptr, *dYt = nullptr;
  float* dYft = nullptr;
  bf16* Ht[kHidden] = {};
  bf16* dZt[kHidden] = {};
  double* d_loss = nullptr;
  unsigned* d_status = nullptr;
  long long* d_step = nullptr;
  long long* d_sched = nullptr;  // {first step, steps} of the current sg_train call
  // inference workspace (grown on demand); the answers of a call are one
  // block, {status word, mean [n][4], sd [n][4], accept [n]}
  int q_cap = 0;
  float *q_x = nullptr, *q_y = nullptr, *q_out = nullptr;
  bf16* q_x16 = nullptr;
  // pinned staging of small calls' queries and answers
  float* h_stage = nullptr;

  void* dalloc(size_t bytes) {
    bytes = (bytes + 255) & ~(size_t)255;
    void* ptr = nullptr;
    if (alloc)
      ptr = alloc(bytes, ctx);
    else if (cudaMalloc(&ptr, bytes) != cudaSuccess) {
      cudaGetLastError();  // reported as IJ_ERR_OOM; the next launch check must not see it
      ptr = nullptr;
    }
    if (ptr) blocks.push_back(ptr);
    return ptr;
  }
  // Give back a block that no launch has used yet (null: nothing).
  void dfree(void* ptr) {
    if (!ptr) return;
    blocks.erase(std::find(blocks.begin(), blocks.end(), ptr));
    if (free_fn) free_fn(ptr, ctx); else cudaFree(ptr);
  }
  void release() {
    if (stream) cudaStreamSynchronize(stream); else cudaDeviceSynchronize();
    for (void* b : blocks) {
      if (free_fn) free_fn(b, ctx); else cudaFree(b);
    }
    blocks.clear();
    if (h_stage) cudaFreeHost(h_stage);
    h_stage = nullptr;
  }
};

namespace {

Layout make_layout(int H) {
  Layout L;
  const int nin[kHidden + 1] = {kInPad, H, H, H, H};
  const int nout[kHidden + 1] = {H, H, H, H, kOutPad};
  long long off = 0;
  for (int l = 0; l <= kHidden; l++) {
    L.nin[l] = nin[l];
    L.nout[l] = nout[l];
    L.w_off[l] = off;
    off += (long long)nin[l] * nout[l];
    L.b_off[l] = off;
    off += nout[l];
  }
  L.total = off;
  return L;
}

ij_status status_of(unsigned st) {
  if (st & kStatusTimeout)
    return fail(IJ_ERR_TIMEOUT, "a tensor-core completion wait ran out of its iteration limit");
  if (st & kStatusNonFinite) return fail(IJ_ERR_NUMERIC, "non-finite training loss");
  return IJ_OK;
}

ij_status status_check(sg_handle h) {
  unsigned st = 0;
  CUDA_TRY(cudaMemcpyAsync(&st, h->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(cudaStreamSynchronize(h->stream));
  return status_of(st);
}

// Everything a training step or a gradient pass of `rows` rows needs.
TrainArgs train_args(sg_handle h, int rows) {
  TrainArgs t;
  memset(&t, 0, sizeof(t));
  t.steps = 1;
  t.members = h->K;
  t.rows = rows;
  t.L = h->L;
  t.X = h->X;
  t.T = h->T;
  t.n = h->n_train;
  t.seed = h->cfg.seed ^ 0x5EEDull;
  t.w = h->d_w;
  t.p = h->p;
  t.g = h->g;
  t.m = h->m;
  t.v = h->v;
  t.Wb = h->Wb;
  t.WbT = h->WbT;
  t.Xt = h->Xt_b;
  t.dYt = h->dYt;
  t.dYft = h->dYft;
  for (int l = 0; l < kHidden; l++) {
    t.Ht[l] = h->Ht[l];
    t.dZt[l] = h->dZt[l];
  }
  t.loss = h->d_loss;
  t.lr = h->cfg.lr;
  t.beta1 = h->cfg.beta1;
  t.beta2 = h->cfg.beta2;
  t.eps = h->cfg.eps;
  t.d_step = h->d_step;
  t.d_sched = h->cfg.lr_cosine ? h->d_sched : nullptr;
  t.status = h->d_status;
  return t;
}

// Losses of the members from the parts a pass over `rows` rows left.
ij_status read_losses(sg_handle h, int rows, double* out) {
  const int parts = train_loss_parts(rows);
  std::vector<double> v((size_t)h->K * parts);
  CUDA_TRY(cudaMemcpyAsync(v.data(), h->d_loss, v.size() * 8, cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(cudaStreamSynchronize(h->stream));
  for (int m = 0; m < h->K; m++) {
    out[m] = 0.0;
    for (int j = 0; j < parts; j++) out[m] += v[(size_t)m * parts + j];
  }
  return IJ_OK;
}

// Transform (mean, scale) of each column of a [n][dim] host array.
void fit_xform(const float* a, int n, int dim, int log_mask, Xform& xf) {
  memset(&xf, 0, sizeof(xf));
  xf.log_mask = log_mask;
  xf.dim = dim;
  for (int d = 0; d < dim; d++) {
    double s = 0, s2 = 0;
    for (int i = 0; i < n; i++) {
      double v = a[(size_t)i * dim + d];
      if ((log_mask >> d) & 1) v = log(v);
      s += v;
      s2 += v * v;
    }
    const double mu = s / n, var = std::max(s2 / n - mu * mu, 0.0);
    xf.mean[d] = (float)mu;
    xf.scale[d] = var > 1e-24 ? (float)sqrt(var) : 1.0f;
  }
  for (int d = dim; d < kInPad; d++) xf.scale[d] = 1.0f;
}

// Words of the answer block before mean: the status word, padded to 16 bytes.
constexpr int kOutHead = 4;
// Calls of up to this many queries go through the pinned staging buffer: one
// copy in and one copy out (37 KB) instead of one in and four out of pageable
// memory, each of which the host waits for.
constexpr int kStagedQueries = 1024;

ij_status ensure_query(sg_handle h, int n) {
  if (n <= h->q_cap) return IJ_OK;
  const size_t nn = (size_t)n, K = h->K;
  void* b[4] = {h->dalloc(nn * kIn * 4), h->dalloc(nn * kInPad * 2), h->dalloc(K * nn * kOut * 4),
                h->dalloc((kOutHead + nn * (2 * kOut + 1)) * 4)};
  if (!b[0] || !b[1] || !b[2] || !b[3]) {
    for (void* p : b) h->dfree(p);  // the workspace in use stays
    return fail(IJ_ERR_OOM, "device allocation of the query workspace failed");
  }
  h->q_x = (float*)b[0];
  h->q_x16 = (bf16*)b[1];
  h->q_y = (float*)b[2];
  h->q_out = (float*)b[3];
  h->q_cap = n;
  return IJ_OK;
}

}  // namespace

extern "C" {

ij_status sg_create(const sg_config* cfg, ij_alloc_fn alloc, ij_free_fn free_fn, void* ctx,
                    void* stream, sg_handle* out) {
  if (!out) return fail(IJ_ERR_PARAM, "out is NULL");
  *out = nullptr;
  if (!cfg) return fail(IJ_ERR_PARAM, "cfg is NULL");
  if ((alloc == nullptr) != (free_fn == nullptr))
    return fail(IJ_ERR_PARAM, "alloc and free must both be set or both be NULL");
  if (cfg->members < 1 || cfg->members > 8) return fail(IJ_ERR_PARAM, "members must be in 1..8");
  if (cfg->hidden < 16 || cfg->hidden > 256 || cfg->hidden % 16)
    return fail(IJ_ERR_PARAM, "hidden must be a multiple of 16 in 16..256");
  if (cfg->batch < 16 || cfg->batch > 65536 || cfg->batch % 16)
    return fail(IJ_ERR_PARAM, "batch must be a multiple of 16 in 16..65536");
  if (!(cfg->lr > 0) || !(cfg->beta1 >= 0 && cfg->beta1 < 1) || !(cfg->beta2 >= 0 && cfg->beta2 < 1) ||
      !(cfg->eps > 0))
    return fail(IJ_ERR_PARAM, "Adam settings out of range");
  if (cfg->lr_cosine != 0 && cfg->lr_cosine != 1) return fail(IJ_ERR_PARAM, "lr_cosine must be 0 or 1");
  sg_handle h = new sg_handle_s();
  h->cfg = *cfg;
  h->K = cfg->members;
  h->H = cfg->hidden;
  h->bm = cfg->batch;
  h->L = make_layout(h->H);
  h->alloc = alloc;
  h->free_fn = free_fn;
  h->ctx = ctx;
  h->stream = (cudaStream_t)stream;
  auto bail = [&](ij_status st) {
    h->release();
    delete h;
    return st;
  };
  const size_t KP = (size_t)h->K * h->L.total, K = h->K, H = h->H, bm = h->bm;
  h->p = (float*)h->dalloc(KP * 4);
  h->g = (float*)h->dalloc(KP * 4);
  h->m = (float*)h->dalloc(KP * 4);
  h->v = (float*)h->dalloc(KP * 4);
  h->Wb = (bf16*)h->dalloc(KP * 2);
  h->WbT = (bf16*)h->dalloc(KP * 2);
  h->Xt_b = (bf16*)h->dalloc(K * bm * kInPad * 2);
  for (int l = 0; l < kHidden; l++) {
    h->Ht[l] = (bf16*)h->dalloc(K * bm * H * 2);
    h->dZt[l] = (bf16*)h->dalloc(K * bm * H * 2);
  }
  h->dYt = (bf16*)h->dalloc(K * bm * kOutPad * 2);
  h->dYft = (float*)h->dalloc(K * bm * kOutPad * 4);
  h->d_loss = (double*)h->dalloc(K * train_loss_parts(h->bm) * 8);
  h->d_status = (unsigned*)h->dalloc(4);
  h->d_step = (long long*)h->dalloc(8);
  h->d_sched = (long long*)h->dalloc(16);
  h->d_lo = (float*)h->dalloc(kIn * 4);
  h->d_hi = (float*)h->dalloc(kIn * 4);
  h->d_w = (float*)h->dalloc(kOut * 4);
  for (void* b : {(void*)h->p, (void*)h->g, (void*)h->m, (void*)h->v, (void*)h->Wb, (void*)h->WbT,
                  (void*)h->Xt_b, (void*)h->dYt, (void*)h->dYft, (void*)h->d_loss,
                  (void*)h->d_status, (void*)h->d_step, (void*)h->d_sched,
                  (void*)h->d_lo, (void*)h->d_hi, (void*)h->d_w})
    if (!b) return bail(fail(IJ_ERR_OOM, "device allocation failed"));
  for (int l = 0; l < kHidden; l++)
    if (!h->Ht[l] || !h->dZt[l]) return bail(fail(IJ_ERR_OOM, "device allocation failed"));
  const cudaError_t e = allow_network_smem();
  if (e != cudaSuccess) return bail(fail(IJ_ERR_CUDA, "allow_network_smem: %s", cudaGetErrorString(e)));
  // He-uniform initialisation on the host (once), zero biases and padding
  std::vector<float> init(KP, 0.0f);
  for (int mem = 0; mem < h->K; mem++)
    for (int l = 0; l <= kHidden; l++) {
      const int fan_in = l == 0 ? kIn : h->H;
      const double bound = sqrt(6.0 / fan_in);
      for (int r = 0; r < h->L.nout[l]; r++)
        for (int c = 0; c < h->L.nin[l]; c++) {
          if ((l == 0 && c >= kIn) || (l == kHidden && r >= kOut)) continue;
          const long long idx = h->L.w_off[l] + (long long)r * h->L.nin[l] + c;
          const unsigned long long u =
              mix64(cfg->seed ^ mix64(((unsigned long long)mem << 40) ^ (unsigned long long)idx));
          const double U = (double)(u >> 11) * (1.0 / 9007199254740992.0);
          init[(size_t)mem * h->L.total + idx] = (float)((2.0 * U - 1.0) * bound);
        }
    }
  cudaStream_t s = h->stream;
  CUDA_TRY(cudaMemcpyAsync(h->p, init.data(), KP * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemsetAsync(h->g, 0, KP * 4, s));
  CUDA_TRY(cudaMemsetAsync(h->m, 0, KP * 4, s));
  CUDA_TRY(cudaMemsetAsync(h->v, 0, KP * 4, s));
  CUDA_TRY(cudaMemsetAsync(h->d_status, 0, 4, s));
  CUDA_TRY(cudaMemsetAsync(h->d_step, 0, 8, s));
  CUDA_TRY(cudaMemsetAsync(h->d_sched, 0, 16, s));
  CUDA_TRY(cudaMemcpyAsync(h->d_w, cfg->out_weight, kOut * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(launch_cast_params(h->p, h->L, h->K, h->Wb, h->WbT, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  memset(&h->xin, 0, sizeof(Xform));
  memset(&h->xout, 0, sizeof(Xform));
  for (int d = 0; d < kInPad; d++) h->xin.scale[d] = h->xout.scale[d] = 1.0f;
  *out = h;
  return IJ_OK;
}

ij_status sg_set_data(sg_handle h, const float* x, const float* y, int n) {
  if (!h || !x || !y) return fail(IJ_ERR_PARAM, "null argument");
  if (n < 2) return fail(IJ_ERR_PARAM, "n must be >= 2");
  for (long long i = 0; i < (long long)n * kIn; i++)
    if (!isfinite(x[i]) || (((h->cfg.log_inputs >> (i % kIn)) & 1) && !(x[i] > 0)))
      return fail(IJ_ERR_PARAM, "input row %lld: non-finite or non-positive under a log", i / kIn);
  for (long long i = 0; i < (long long)n * kOut; i++)
    if (!isfinite(y[i]) || (((h->cfg.log_outputs >> (i % kOut)) & 1) && !(y[i] > 0)))
      return fail(IJ_ERR_PARAM, "outcome row %lld: non-finite or non-positive under a log",
                  i / kOut);
  Xform xin, xout;
  fit_xform(x, n, kIn, h->cfg.log_inputs, xin);
  fit_xform(y, n, kOut, h->cfg.log_outputs, xout);
  float lo[kIn], hi[kIn];
  for (int d = 0; d < kIn; d++) {
    lo[d] = hi[d] = x[d];
    for (int i = 1; i < n; i++) {
      lo[d] = std::min(lo[d], x[(size_t)i * kIn + d]);
      hi[d] = std::max(hi[d], x[(size_t)i * kIn + d]);
    }
  }
  // leave-one-out nearest-neighbour distances in transformed input space
  std::vector<double> xt((size_t)n * kIn);
  for (int i = 0; i < n; i++)
    for (int d = 0; d < kIn; d++) {
      double v = x[(size_t)i * kIn + d];
      if ((h->cfg.log_inputs >> d) & 1) v = log(v);
      xt[(size_t)i * kIn + d] = (v - xin.mean[d]) / xin.scale[d];
    }
  std::vector<double> nn(n, 1e300);
  for (int i = 0; i < n; i++)
    for (int j = i + 1; j < n; j++) {
      double d2 = 0;
      for (int d = 0; d < kIn; d++) {
        const double e = xt[(size_t)i * kIn + d] - xt[(size_t)j * kIn + d];
        d2 += e * e;
      }
      nn[i] = std::min(nn[i], d2);
      nn[j] = std::min(nn[j], d2);
    }
  std::sort(nn.begin(), nn.end());

  // Everything that can run out of memory comes before the handle changes: on
  // failure the data, transforms and gate it had stay in use.
  cudaStream_t s = h->stream;
  void *X = nullptr, *T = nullptr, *Xt = nullptr;
  const int ldt = (n + 127) / 128 * 128;  // the gate reads whole groups of 128 points
  ij_status st = IJ_OK;
  if (n > h->train_cap) {
    X = h->dalloc((size_t)n * kInPad * 2);
    T = h->dalloc((size_t)n * kOut * 4);
    Xt = h->dalloc((size_t)ldt * kIn * 4);
    if (!X || !T || !Xt) st = fail(IJ_ERR_OOM, "device allocation of the data failed");
  }
  if (st == IJ_OK) st = ensure_query(h, n);  // raw rows are staged in the query workspace
  if (st != IJ_OK) {
    for (void* p : {X, T, Xt}) h->dfree(p);
    return st;
  }
  if (n > h->train_cap) {
    h->X = (bf16*)X;
    h->T = (float*)T;
    h->Xt = (float*)Xt;
    h->ldt = ldt;
    h->train_cap = n;
  }
  h->xin = xin;
  h->xout = xout;
  memcpy(h->lo, lo, sizeof(lo));
  memcpy(h->hi, hi, sizeof(hi));
  h->nn_cut = (float)(2.0 * sqrt(nn[(size_t)((n - 1) * 0.95)]));
  CUDA_TRY(cudaMemcpyAsync(h->q_x, x, (size_t)n * kIn * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(h->q_out, y, (size_t)n * kOut * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(launch_prep_inputs(h->q_x, n, h->xin, h->X, h->Xt, h->ldt, s));
  CUDA_TRY(launch_prep_targets(h->q_out, n, h->xout, h->T, s));
  CUDA_TRY(cudaMemcpyAsync(h->d_lo, h->lo, kIn * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(h->d_hi, h->hi, kIn * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  h->n_train = n;
  return IJ_OK;
}

ij_status sg_train(sg_handle h, int steps, double* loss) {
  if (!h) return fail(IJ_ERR_PARAM, "null handle");
  if (steps < 0) return fail(IJ_ERR_PARAM, "steps < 0");
  if (h->n_train < 2) return fail(IJ_ERR_STATE, "no training data (sg_set_data)");
  if (h->cfg.lr_cosine && steps > 0)
    CUDA_TRY(launch_schedule_begin(h->d_step, h->d_sched, steps, h->stream));
  TrainArgs t = train_args(h, h->bm);
  t.steps = steps;
  CUDA_TRY(launch_train_step(t, h->stream));
  ij_status st = status_check(h);
  if (st != IJ_OK) return st;
  if (loss) {
    *loss = 0.0;
    if (steps > 0) {
      std::vector<double> l(h->K);
      st = read_losses(h, h->bm, l.data());
      if (st != IJ_OK) return st;
      for (double v : l) *loss += v / h->K;
    }
  }
  return IJ_OK;
}

ij_status sg_predict(sg_handle h, const float* x, int n, float* mean, float* sd, int* accept,
                     int on_device) {
  if (!h || !x) return fail(IJ_ERR_PARAM, "null argument");
  if (n < 0) return fail(IJ_ERR_PARAM, "n < 0");
  if (n == 0) return IJ_OK;
  if (accept && h->n_train < 2) return fail(IJ_ERR_STATE, "the gate needs training data");
  ij_status st = ensure_query(h, n);
  if (st != IJ_OK) return st;
  cudaStream_t s = h->stream;
  const size_t nn = (size_t)n;
  const bool staged = !on_device && n <= kStagedQueries;
  if (staged && !h->h_stage)
    CUDA_TRY(cudaMallocHost((void**)&h->h_stage,
                            (kOutHead + (size_t)kStagedQueries * (2 * kOut + 1)) * 4));
  const float* dx = x;
  if (!on_device) {
    const float* src = x;
    if (staged) src = (const float*)memcpy(h->h_stage, x, nn * kIn * 4);
    CUDA_TRY(cudaMemcpyAsync(h->q_x, src, nn * kIn * 4, cudaMemcpyHostToDevice, s));
    dx = h->q_x;
  }
  CUDA_TRY(launch_forward(dx, n, h->xin, h->p, h->Wb, h->L, h->K, h->q_y, h->d_status, s));
  GateArgs a;
  memset(&a, 0, sizeof(a));
  a.x = dx;
  a.Y = h->q_y;
  a.n = n;
  a.members = h->K;
  a.xin = h->xin;
  a.xout = h->xout;
  a.Xt = h->Xt;
  a.nt = h->n_train;
  a.ldt = h->ldt;
  a.lo = h->d_lo;
  a.hi = h->d_hi;
  a.nn_cut = h->nn_cut;
  a.tau = h->tau;
  a.tau_v = h->tau_v;
  a.mean = h->q_out + kOutHead;
  a.sd = a.mean + nn * kOut;
  a.accept = accept ? (int*)(a.sd + nn * kOut) : nullptr;
  a.status = h->d_status;
  a.status_out = (unsigned*)h->q_out;
  CUDA_TRY(launch_answer(a, s));
  if (staged) {
    const size_t words = kOutHead + nn * (2 * kOut + (accept ? 1 : 0));
    CUDA_TRY(cudaMemcpyAsync(h->h_stage, h->q_out, words * 4, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    const float* o = h->h_stage + kOutHead;
    if (mean) memcpy(mean, o, nn * kOut * 4);
    if (sd) memcpy(sd, o + nn * kOut, nn * kOut * 4);
    if (accept) memcpy(accept, o + 2 * nn * kOut, nn * 4);
    unsigned word;
    memcpy(&word, h->h_stage, 4);
    return status_of(word);
  }
  const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
  if (mean) CUDA_TRY(cudaMemcpyAsync(mean, a.mean, nn * kOut * 4, kind, s));
  if (sd) CUDA_TRY(cudaMemcpyAsync(sd, a.sd, nn * kOut * 4, kind, s));
  if (accept) CUDA_TRY(cudaMemcpyAsync(accept, a.accept, nn * 4, kind, s));
  return status_check(h);
}

ij_status sg_set_gate(sg_handle h, float tau, float tau_v, float nn_cut) {
  if (!h) return fail(IJ_ERR_PARAM, "null handle");
  if (!(tau > 0) || !(tau_v > 0)) return fail(IJ_ERR_PARAM, "tau and tau_v must be > 0");
  h->tau = tau;
  h->tau_v = tau_v;
  if (nn_cut > 0) h->nn_cut = nn_cut;
  return IJ_OK;
}

ij_status sg_param_count(sg_handle h, long long* count) {
  if (!h || !count) return fail(IJ_ERR_PARAM, "null argument");
  *count = h->L.total;
  return IJ_OK;
}

ij_status sg_get_params(sg_handle h, int member, float* out) {
  if (!h || !out) return fail(IJ_ERR_PARAM, "null argument");
  if (member < 0 || member >= h->K) return fail(IJ_ERR_PARAM, "member out of range");
  CUDA_TRY(cudaMemcpyAsync(out, h->p + (size_t)member * h->L.total, h->L.total * 4,
                           cudaMemcpyDeviceToHost, h->stream));
  CUDA_TRY(cudaStreamSynchronize(h->stream));
  return IJ_OK;
}

ij_status sg_set_params(sg_handle h, int member, const float* in) {
  if (!h || !in) return fail(IJ_ERR_PARAM, "null argument");
  if (member < 0 || member >= h->K) return fail(IJ_ERR_PARAM, "member out of range");
  CUDA_TRY(cudaMemcpyAsync(h->p + (size_t)member * h->L.total, in, h->L.total * 4,
                           cudaMemcpyHostToDevice, h->stream));
  CUDA_TRY(launch_cast_params(h->p, h->L, h->K, h->Wb, h->WbT, h->stream));
  CUDA_TRY(cudaStreamSynchronize(h->stream));
  return IJ_OK;
}

ij_status sg_get_transform(sg_handle h, float* in_mean, float* in_scale, float* out_mean,
                           float* out_scale) {
  if (!h) return fail(IJ_ERR_PARAM, "null handle");
  for (int d = 0; d < kIn; d++) {
    if (in_mean) in_mean[d] = h->xin.mean[d];
    if (in_scale) in_scale[d] = h->xin.scale[d];
  }
  for (int d = 0; d < kOut; d++) {
    if (out_mean) out_mean[d] = h->xout.mean[d];
    if (out_scale) out_scale[d] = h->xout.scale[d];
  }
  return IJ_OK;
}

ij_status sg_gradients(sg_handle h, const float* x, const float* y, int n, float* grads,
                       double* loss) {
  if (!h || !x || !y || !grads) return fail(IJ_ERR_PARAM, "null argument");
  if (n < 16 || n % 16 || n > h->bm) return fail(IJ_ERR_PARAM, "n must be a multiple of 16, <= batch");
  cudaStream_t s = h->stream;
  ij_status st = ensure_query(h, n);
  if (st != IJ_OK) return st;
  bf16* x16 = h->q_x16;
  float* yq = h->q_out;  // raw targets, then the transformed ones
  float* t = h->q_out + (size_t)n * kOut;
  CUDA_TRY(cudaMemcpyAsync(h->q_x, x, (size_t)n * kIn * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(yq, y, (size_t)n * kOut * 4, cudaMemcpyHostToDevice, s));
  CUDA_TRY(launch_prep_inputs(h->q_x, n, h->xin, x16, nullptr, 0, s));
  CUDA_TRY(launch_prep_targets(yq, n, h->xout, t, s));
  TrainArgs ta = train_args(h, n);
  ta.direct = 1;  // every member sees the same rows
  ta.grads_only = 1;
  ta.X = x16;
  ta.T = t;
  ta.n = n;
  CUDA_TRY(launch_train_step(ta, s));
  st = status_check(h);
  if (st != IJ_OK) return st;
  CUDA_TRY(cudaMemcpy(grads, h->g, (size_t)h->K * h->L.total * 4, cudaMemcpyDeviceToHost));
  return loss ? read_losses(h, n, loss) : IJ_OK;
}

ij_status sg_destroy(sg_handle h) {
  if (!h) return IJ_OK;
  h->release();
  delete h;
  return IJ_OK;
}

const char* sg_last_error(void) { return g_err; }

ij_status sg_gemm_bf16(const void* A, int lda, const void* B, int ldb, int M, int N, int K,
                       float* C, int ldc, void* stream) {
  if (!A || !B || !C) return fail(IJ_ERR_PARAM, "null pointer");
  if (M < 1 || N < 1 || K < 1) return fail(IJ_ERR_PARAM, "M, N, K must be >= 1");
  if (K % 8 || lda % 8 || ldb % 8 || lda < K || ldb < K || ldc < N)
    return fail(IJ_ERR_PARAM, "K, lda, ldb must be multiples of 8, lda, ldb >= K, ldc >= N");
  if (((uintptr_t)A | (uintptr_t)B) & 15) return fail(IJ_ERR_PARAM, "A and B must be 16-byte aligned");
  cudaStream_t s = (cudaStream_t)stream;
  unsigned* status = nullptr;
  CUDA_TRY(cudaMallocAsync((void**)&status, sizeof(unsigned), s));
  CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(unsigned), s));
  GemmArgs a;
  memset(&a, 0, sizeof(a));
  a.A = (const bf16*)A;
  a.B = (const bf16*)B;
  a.lda = lda;
  a.ldb = ldb;
  a.M = M;
  a.N = N;
  a.K = K;
  a.C = C;
  a.ldc = ldc;
  a.status = status;
  CUDA_TRY(launch_gemm(a, s));
  unsigned st = 0;
  CUDA_TRY(cudaMemcpyAsync(&st, status, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaFreeAsync(status, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  if (st & kStatusTimeout) return fail(IJ_ERR_TIMEOUT, "tensor-core completion wait timed out");
  return IJ_OK;
}

}  // extern "C"
