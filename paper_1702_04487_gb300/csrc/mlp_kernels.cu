// Kernels of the surrogate network on the 5th generation tensor cores
// (tcgen05.mma, accumulator in tensor memory): a plain BF16 GEMM and, built
// from the same pieces, the training step (chain_kernel, update_kernel), the
// inference kernels (chain_kernel, forward_kernel, pair_kernel) and the answer
// kernel (decoding, ensemble spread, acceptance gate).
//
// GEMM shape: C[M x N] = A[M x K] B[N x K]^T with A and B row-major (K
// contiguous, "K-major").  A CTA of 128 threads owns a 128 x BN tile of C,
// BN in {16, 32, 64, 128, 256}.  K advances in slices of 64 (128 bytes of
// BF16, one row of a 128-byte swizzle atom) through a ring of kStages
// shared-memory buffers.  One thread drives the pipeline: it loads slices of
// A and of B with the tensor memory accelerator (cp.async.bulk.tensor,
// 128-byte swizzle written by the copy itself, completion counted in bytes
// on the buffer's load mbarrier) up to kStages ahead -- every slice of the
// surrogate's K <= 256 at once -- issues the four K=16 MMAs of a slice once
// it has landed and commits them to the buffer's MMA mbarrier, and refills
// the buffer of the previous slice once its MMAs are done.  If a bounded
// wait gives up, every copy and MMA still in flight is waited for (again
// bounded) before the tensor memory is released and the CTA exits; the
// output is then left unwritten and the timeout flag set.  The epilogue reads the accumulator with
// tcgen05.ld (warp w owns tensor-memory lanes 32w..32w+31, i.e. rows
// 32w..32w+31 of the tile).
#include <cuda.h>
#include <math.h>

#include "mlp.cuh"

namespace sg {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kStages = 4;  // shared-memory buffers of K slices
constexpr int kThreads = 128;
constexpr int kWaitLimit = 1 << 22;  // try_wait rounds before giving up

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
// Wait for the completion of the barrier phase of the given parity; false
// after kWaitLimit rounds.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int i = 0; i < kWaitLimit; i++) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major tile in the 128-byte swizzle
// layout: rows of 128 bytes, 8-row atoms of 1024 bytes stacked along M/N
// (stride byte offset 1024); the leading byte offset is unused for this
// layout.  Bits: start address >> 4 [0,14), leading offset >> 4 [16,30),
// stride offset >> 4 [32,46), version 1 [46,48), swizzle mode 2 [61,64).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// The same in the 64-byte swizzle layout: rows of 64 bytes (32 values of K),
// 8-row atoms of 512 bytes; swizzle mode 4.  The copy of 16-byte chunk c of
// row r lies at chunk c ^ ((r >> 1) & 3).
__device__ __forceinline__ uint64_t sw64_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}

// Instruction descriptor of kind::f16: FP32 accumulator [4,6) = 1, A and B
// BF16 [7,10) = [10,13) = 1, both K-major, N >> 3 at [17,23), M >> 4 at
// [24,29).
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
      : "memory");
}

// 16 consecutive FP32 accumulator columns of this thread's lane (row).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; j++) v[j] = __uint_as_float(r[j]);
}

// The two halves of it: start the load, and wait for every load started (the
// values pass through the wait, so nothing reads them before it).
__device__ __forceinline__ void tmem_ld16_start(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld16_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                 "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                 "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}

// The same for 8 columns.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int j = 0; j < 8; j++) v[j] = __uint_as_float(r[j]);
}

__device__ __forceinline__ float gelu_f(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float gelu_grad_f(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) +
         x * 0.39894228040143268f * expf(-0.5f * x * x);
}

template <int BN>
__host__ __device__ constexpr int stage_bytes() {
  return BM * BK * 2 + BN * BK * 2;
}
template <int BN>
__host__ __device__ constexpr int tmem_cols() {
  return BN < 32 ? 32 : BN;
}

// Arm the load barrier for `bytes` of asynchronous copies (one arrival).
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
               : "memory");
}

// One box of a 3-D tensor map (x = K offset, y = row, z = member) into
// shared memory; completion is counted on `bar`.
__device__ __forceinline__ void tma_load3(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// Thread 0 of a CTA: the K loop of a 128 x BN tile, loads, MMAs and commits;
// returns once every MMA is done, or false after a wait that gave up.
// bars[b]: the load of buffer b landed; bars[kStages + b]: its MMAs done.
template <int BN>
__device__ bool gemm_pipeline(uint8_t* smem, uint64_t* bars, const CUtensorMap* tmA,
                              const CUtensorMap* tmB, int m0, int n0, int za, int zb, int K,
                              uint32_t tmem) {
  constexpr int kA = BM * BK * 2;
  constexpr int kStage = stage_bytes<BN>();
  constexpr uint32_t kIdesc = idesc_bf16(BM, BN);
  const int nk = (K + BK - 1) / BK;
  bool ok = true;
  // slice kt lives in buffer kt % kStages; its load completes phase
  // (kt / kStages) & 1 of bars[buffer], its MMAs the same phase of
  // bars[kStages + buffer]
  auto load = [&](int kt) {
    const int b = kt % kStages;
    const uint32_t ta = smem_u32(smem + b * kStage), tb = ta + kA;
    mbar_expect_tx(smem_u32(&bars[b]), (uint32_t)kStage);
    tma_load3(ta, tmA, kt * BK, m0, za, smem_u32(&bars[b]));
    tma_load3(tb, tmB, kt * BK, n0, zb, smem_u32(&bars[b]));
  };
  auto phase = [](int kt) { return (uint32_t)((kt / kStages) & 1); };
  int loaded = 0;     // slices whose loads were issued
  int landed = 0;     // slices whose loads were seen complete
  int committed = 0;  // slices whose MMAs were committed
  int freed = 0;      // slices whose MMAs were seen complete
  for (; loaded < nk && loaded < kStages; loaded++) load(loaded);
  for (int kt = 0; kt < nk; kt++) {
    const int b = kt % kStages;
    if (!mbar_wait(smem_u32(&bars[b]), phase(kt))) {
      ok = false;
      break;
    }
    landed = kt + 1;
    tc_fence_after();
    const uint32_t ta = smem_u32(smem + b * kStage), tb = ta + kA;
#pragma unroll
    for (int k = 0; k < BK / 16; k++)
      mma_bf16(tmem, sw128_desc(ta + 32 * k), sw128_desc(tb + 32 * k), kIdesc,
               (kt > 0 || k > 0) ? 1u : 0u);
    mma_commit(smem_u32(&bars[kStages + b]));
    committed = kt + 1;
    // refill the buffer of the previous slice once its MMAs are done
    if (kt >= 1 && loaded < nk) {
      if (!mbar_wait(smem_u32(&bars[kStages + (kt - 1) % kStages]), phase(kt - 1))) {
        ok = false;
        break;
      }
      freed = kt;
      load(loaded++);
    }
  }
  // Before the accumulator is read, the tensor memory released or the CTA
  // exits, every copy issued must have landed and every MMA committed must
  // be done -- also after a timeout above (these waits are bounded too).
  for (int kt = landed; kt < loaded; kt++)
    ok = mbar_wait(smem_u32(&bars[kt % kStages]), phase(kt)) && ok;
  for (int kt = freed > committed - kStages ? freed : committed - kStages; kt < committed; kt++)
    ok = mbar_wait(smem_u32(&bars[kStages + kt % kStages]), phase(kt)) && ok;
  return ok;
}

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr int kStage = stage_bytes<BN>();
  constexpr uint32_t kCols = tmem_cols<BN>();
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;

  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 2 * kStages; i++) mbar_init(smem_u32(&bars[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  bool ok = true;
  if (tid == 0) ok = gemm_pipeline<BN>(smem, bars, &tmA, &tmB, m0, n0, 0, 0, a.K, tmem);
  ok = __syncthreads_and(ok);
  tc_fence_after();

  if (ok) {
    // Epilogue through shared memory (the operand buffers are free once every
    // MMA is done): each warp takes its 32 rows x 16 columns from tensor
    // memory (lane = row), then works row by row -- half-warps on two rows,
    // lanes along n -- so that C is written in contiguous runs.
    float* T = reinterpret_cast<float*>(smem) + warp * (32 * 17);
    const int jj = lane & 15, rh = lane >> 4;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
      const int nb = n0 + c0;
      if (nb >= a.N) continue;  // uniform over the CTA
#pragma unroll
      for (int j = 0; j < 16; j++) T[lane * 17 + j] = v[j];
      __syncwarp();
      const int n = nb + jj;
#pragma unroll 4
      for (int i = 0; i < 16; i++) {
        const int r = 2 * i + rh, mm = m0 + warp * 32 + r;
        if (mm < a.M && n < a.N) a.C[(size_t)mm * a.ldc + n] = T[r * 17 + jj];
      }
      __syncwarp();  // the next chunk overwrites T
    }
  } else if (tid == 0) {
    atomicOr(a.status, kStatusTimeout);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols)
                 : "memory");
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once through the runtime (no
// link against the driver library).
EncodeTiledFn encode_tiled() {
  // (the initialisation of a local static is safe with several threads)
  static const EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    return nullptr;
  }();
  return fn;
}

// Dynamic shared memory beyond 48 KB has to be allowed for a kernel, on each
// device: nothing about it is kept between calls.
template <typename F>
cudaError_t allow_smem(F* kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// 3-D tensor map of a BF16 operand: K (contiguous) x rows (leading dimension
// ld) x layers (stride layer, or one layer), boxes of 64 x box_rows x 1 in
// the 128-byte swizzle; out-of-range elements read as zero.
cudaError_t make_map(CUtensorMap* m, const bf16* base, int K, int rows, int ld,
                     long long layer, int layers, int box_rows) {
  EncodeTiledFn enc = encode_tiled();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)layers};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 2,
                                 (cuuint64_t)(layers > 1 ? layer : (long long)ld * rows) * 2};
  const cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1};
  const cuuint32_t es[3] = {1, 1, 1};
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<bf16*>(base), dims,
                         strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

template <int BN>
cudaError_t launch_bn(const GemmArgs& a, cudaStream_t s) {
  const size_t smem = gemm_smem_bytes(BN);
  CUtensorMap ma, mb;
  cudaError_t e0 = make_map(&ma, a.A, a.K, a.M, a.lda, 0, 1, BM);
  if (e0 == cudaSuccess) e0 = make_map(&mb, a.B, a.K, a.N, a.ldb, 0, 1, BN);
  if (e0 == cudaSuccess) e0 = allow_smem(gemm_kernel<BN>, smem);
  if (e0 != cudaSuccess) return e0;
  dim3 grid((a.M + BM - 1) / BM, (a.N + BN - 1) / BN);
  gemm_kernel<BN><<<grid, kThreads, smem, s>>>(ma, mb, a);
  return cudaGetLastError();
}

}  // namespace

size_t gemm_smem_bytes(int bn) {
  return 1024 + kStages * (size_t)(BM * BK * 2 + bn * BK * 2) + 16 * kStages + 16;
}

cudaError_t launch_gemm(const GemmArgs& a, cudaStream_t s) {
  // the narrowest tile that covers N, halved (down to 32 columns) while the
  // grid has fewer than ~2 tiles per SM of a 152-SM part
  int bn = a.N <= 16 ? 16 : a.N <= 32 ? 32 : a.N <= 64 ? 64 : a.N <= 128 ? 128 : 256;
  const long long mt = (a.M + BM - 1) / BM;
  while (bn > 32 && mt * ((a.N + bn - 1) / bn) < 304) bn /= 2;
  switch (bn) {
    case 16: return launch_bn<16>(a, s);
    case 32: return launch_bn<32>(a, s);
    case 64: return launch_bn<64>(a, s);
    case 128: return launch_bn<128>(a, s);
    default: return launch_bn<256>(a, s);
  }
}

}  // namespace sg

// ---------------------------------------------------------------------------
// The network, training and inference.
namespace sg {
namespace {

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  // SplitMix64 finaliser (Steele, Lea & Flood 2014)
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

__device__ __forceinline__ float xform(float v, int d, const Xform& xf) {
  if ((xf.log_mask >> d) & 1) v = logf(v);
  return (v - xf.mean[d]) / xf.scale[d];
}

__global__ void prep_inputs_kernel(const float* __restrict__ x, int n, const Xform xf,
                                   bf16* __restrict__ X, float* __restrict__ Xf, int ldx) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
#pragma unroll
  for (int d = 0; d < kInPad; d++) {
    const float v = d < kIn ? xform(x[(size_t)r * kIn + d], d, xf) : 0.0f;
    if (X) X[(size_t)r * kInPad + d] = __float2bfloat16_rn(v);
    if (Xf && d < kIn) Xf[(size_t)d * ldx + r] = v;
  }
}

__global__ void prep_targets_kernel(const float* __restrict__ y, int n, const Xform yf,
                                    float* __restrict__ T) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
#pragma unroll
  for (int d = 0; d < kOut; d++) T[(size_t)r * kOut + d] = xform(y[(size_t)r * kOut + d], d, yf);
}

// Locate flat parameter index i of a member: layer, and whether a weight
// (row r, column c) or a bias.
__device__ __forceinline__ void locate(const Layout& L, long long i, int& l, int& r, int& c,
                                       bool& weight) {
  l = 0;
#pragma unroll
  for (int k = 1; k <= kHidden; k++)
    if (i >= L.w_off[k]) l = k;
  if (i < L.b_off[l]) {
    weight = true;
    const long long j = i - L.w_off[l];
    r = (int)(j / L.nin[l]);
    c = (int)(j % L.nin[l]);
  } else {
    weight = false;
    r = (int)(i - L.b_off[l]);
    c = 0;
  }
}

__global__ void cast_params_kernel(const float* __restrict__ p, const Layout L, int members,
                                   bf16* __restrict__ Wb, bf16* __restrict__ WbT) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= L.total * members) return;
  const long long mem = i / L.total, k = i % L.total;
  int l, r, c;
  bool weight;
  locate(L, k, l, r, c, weight);
  if (weight) {
    const bf16 b = __float2bfloat16_rn(p[i]);
    Wb[i] = b;
    WbT[mem * L.total + L.w_off[l] + (long long)c * L.nout[l] + r] = b;
  }
}

// ---------------------------------------------------------------------------
// Inference: all five layers of a 128-row tile of queries for one member in
// one CTA.  The tile's activations stay in shared memory (BF16, the K-major
// 128-byte-swizzled layout the tensor cores read) and the accumulator in
// tensor memory; only the queries are read and the four outcomes written, so
// nothing of a hidden layer touches HBM.  Weights stream from L2 through a
// ring of 64 (K) x 128 (output units) chunks loaded by the tensor memory
// accelerator; they do not depend on the activations, so the chunks of the
// next layer are fetched while this layer's outputs are computed.  Thread 0
// loads and issues; the output pass of a hidden layer (bias, GELU, rounding
// to BF16, swizzled 16-byte stores) is shared by every warp: warp w reads
// tensor-memory lanes 32 (w mod 4) .. + 31 and every (warps / 4)-th group of
// 16 units.
//
// Bound by latency (a tile per SM at most; many tiles take pair_kernel): five
// members of H = 256, queries and answers on the device, take 82 us a call from
// 385 to 3072 queries.
constexpr int kFwdChunk = 128 * BK * 2;  // bytes of a weight chunk, and of 64 activation columns
constexpr int kFwdRing = 9;

struct FwdMaps {
  CUtensorMap w[kHidden + 1];  // boxes of 64 (K) x 128 (units) x 1 (member)
};
struct FwdArgs {
  const float* x;
  int n, H;
  Xform xf;
  const float* p;
  long long P;
  int b_off[kHidden + 1];
  float* Y;
  unsigned* status;
};

constexpr int kFwdThreads = 512;
// activations, ring, then the barriers and the tensor-memory address (no
// static shared memory: the dynamic part then starts on a 1024-byte boundary)
constexpr int kFwdTail = 256;
size_t fwd_smem_bytes(int H, int ring) {
  return (size_t)((H + BK - 1) / BK + ring) * kFwdChunk + kFwdTail;
}

__global__ void __launch_bounds__(kFwdThreads, 1)
    forward_kernel(const __grid_constant__ FwdMaps maps, const FwdArgs a) {
  extern __shared__ __align__(1024) uint8_t fwd_smem[];
  constexpr int R = kFwdRing, NT = kFwdThreads;
  const int H = a.H, slices = (H + BK - 1) / BK;
  uint8_t* const smem = fwd_smem;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + (size_t)(slices + R) * kFwdChunk);
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * R + 1);
  static_assert((2 * R + 1) * 8 + 4 <= kFwdTail, "barriers outgrew their slot");
  const uint32_t act = smem_u32(smem);
  if (act & 1023u) {  // the swizzled layout needs the alignment asked for
    if (threadIdx.x == 0) atomicOr(a.status, kStatusTimeout);
    return;
  }
  const uint32_t ring = act + (uint32_t)slices * kFwdChunk;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * BM, z = blockIdx.y;
  const uint32_t cols = H <= 32 ? 32 : H <= 64 ? 64 : H <= 128 ? 128 : 256;
  // bars[b]: chunk landed; bars[R + b]: its MMAs done; bars[2 R]: layer done
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 2 * R + 1; i++) mbar_init(smem_u32(&bars[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }

  // Chunk c of the member's weights, in the order they are used: layer by
  // layer, K slice by K slice, 128 output units at a time.
  int ld_l = 0, ld_s = 0, ld_h = 0, loaded = 0;  // the next chunk to load
  auto units_of = [&](int l) { return l < kHidden ? H : kOutPad; };
  auto depth_of = [&](int l) { return l == 0 ? kInPad : H; };
  auto load_next = [&]() {
    if (ld_l > kHidden) return;
    const int b = loaded % R;
    const uint32_t bar = smem_u32(&bars[b]);
    mbar_expect_tx(bar, (uint32_t)kFwdChunk);
    tma_load3(ring + (uint32_t)b * kFwdChunk, &maps.w[ld_l], ld_s * BK, ld_h * 128, z, bar);
    loaded++;
    if ((++ld_h) * 128 >= units_of(ld_l)) {
      ld_h = 0;
      if ((++ld_s) * BK >= depth_of(ld_l)) {
        ld_s = 0;
        ld_l++;
      }
    }
  };
  if (tid == 0)
    for (int i = 0; i < R; i++) load_next();

  // layer 0's operand: transformed queries, BF16, columns 7..15 zero
  if (tid < BM) {
    const int row = m0 + tid;
    __align__(16) bf16 v[kInPad];
#pragma unroll
    for (int d = 0; d < kInPad; d++)
      v[d] = __float2bfloat16_rn(
          d < kIn && row < a.n ? xform(a.x[(size_t)row * kIn + d], d, a.xf) : 0.0f);
#pragma unroll
    for (int c = 0; c < 2; c++)
      *reinterpret_cast<uint4*>(smem + tid * 128 + ((c ^ (tid & 7)) << 4)) =
          reinterpret_cast<const uint4*>(v)[c];
  }
  const bool rows_in = m0 + (warp & 3) * 32 < a.n;  // any valid row of this warp's 32
  uint32_t tmem = 0;
  int used = 0, freed = 0;  // thread 0: chunks whose MMAs were issued / seen done
  bool ok = true;
  for (int l = 0; l <= kHidden; l++) {
    // the operand written by every thread is visible to the tensor cores
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (l == 0) tmem = *(volatile uint32_t*)tmem_slot;
    if (tid == 0) {
      const int K = depth_of(l), N = units_of(l);
      for (int s = 0; s * BK < K && ok; s++)
        for (int h = 0; h * 128 < N && ok; h++) {
          const int b = used % R;
          if (!mbar_wait(smem_u32(&bars[b]), (uint32_t)((used / R) & 1))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int nn = N - h * 128 < 128 ? N - h * 128 : 128;
          const int steps = K - s * BK < BK ? (K - s * BK) / 16 : BK / 16;
          const uint32_t ta = act + (uint32_t)s * kFwdChunk, tb = ring + (uint32_t)b * kFwdChunk;
          const uint32_t id = idesc_bf16(BM, nn);
          for (int k = 0; k < steps; k++)
            mma_bf16(tmem + h * 128, sw128_desc(ta + 32 * k), sw128_desc(tb + 32 * k), id,
                     (s > 0 || k > 0) ? 1u : 0u);
          mma_commit(smem_u32(&bars[R + b]));
          used++;
          // refill the buffer of the chunk before once its MMAs are done
          if (used >= 2 && ld_l <= kHidden && loaded < used - 1 + R) {
            if (!mbar_wait(smem_u32(&bars[R + (used - 2) % R]), (uint32_t)(((used - 2) / R) & 1))) {
              ok = false;
              break;
            }
            freed = used - 1;
            load_next();
          }
        }
      if (ok) {
        // an arrival once every MMA of the layer is done
        mma_commit(smem_u32(&bars[2 * R]));
        ok = mbar_wait(smem_u32(&bars[2 * R]), (uint32_t)(l & 1));
        if (ok) {
          freed = used;
          while (ld_l <= kHidden && loaded < used + R) load_next();
        }
      }
    }
    ok = __syncthreads_and(ok);
    if (!ok) break;
    tc_fence_after();
    if (l < kHidden) {
      const float* bias = a.p + z * a.P + a.b_off[l];
      if (rows_in)
#pragma unroll 1
        for (int c0 = (warp >> 2) * 16; c0 < H; c0 += NT / 128 * 16) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
          __align__(16) bf16 o[16];
#pragma unroll
          for (int j = 0; j < 16; j++) o[j] = __float2bfloat16_rn(gelu_f(v[j] + __ldg(bias + c0 + j)));
          const int r = (warp & 3) * 32 + lane, sl = c0 / BK, ch = (c0 % BK) / 8;
          uint8_t* row = smem + (size_t)sl * kFwdChunk + r * 128;
#pragma unroll
          for (int c = 0; c < 2; c++)
            *reinterpret_cast<uint4*>(row + (((ch + c) ^ (r & 7)) << 4)) =
                reinterpret_cast<const uint4*>(o)[c];
        }
    } else if (warp < 4 && rows_in) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16), v);
      const int row = m0 + warp * 32 + lane;
      const float* bias = a.p + z * a.P + a.b_off[l];
      if (row < a.n)
        *reinterpret_cast<float4*>(a.Y + ((size_t)z * a.n + row) * kOut) =
            make_float4(v[0] + __ldg(bias), v[1] + __ldg(bias + 1), v[2] + __ldg(bias + 2),
                        v[3] + __ldg(bias + 3));
    }
  }
  if (!ok) {
    // no copy may land and no MMA run after the CTA gives up its memory
    // (bounded again)
    if (tid == 0) {
      for (int c = used; c < loaded; c++) mbar_wait(smem_u32(&bars[c % R]), (uint32_t)((c / R) & 1));
      for (int c = freed > used - R ? freed : used - R; c < used; c++)
        if (c >= 0) mbar_wait(smem_u32(&bars[R + c % R]), (uint32_t)((c / R) & 1));
      atomicOr(a.status, kStatusTimeout);
    }
    if (tmem == 0) tmem = *(volatile uint32_t*)tmem_slot;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Inference of many queries: the same on two 128-row tiles per CTA, one CTA
// per SM.  16 warps do nothing but output passes, alternating between the
// tiles; a warp each issues the products and loads the weights (streamed from
// L2 once per tile and layer through a ring of 16 KB chunks).  While the
// output pass of one tile runs, the tensor cores work on the other, so that
// the instruction issue, which bounds this kernel, never waits for them.
//  ready[t]: the 16 warps have written tile t's next operand and are done with
//  its accumulator; done[t]: its products are complete.
//
// Bound by the GELUs (an erff each: 4 H per query and member, 32 instructions
// a GELU) at instruction issue.  Measured, five members of H = 256: a call of
// 65536 queries takes 534 us, 619 with a tile per CTA and two CTAs per SM (56 %
// issue: both wait for their products together), 568 without the accumulator
// loads one step ahead, and 2190 us more for a GEMM launch per layer with the
// activations through HBM.
constexpr int kPairRing = 6;
constexpr int kPairWarps = 16;
constexpr int kPairThreads = (kPairWarps + 2) * 32;
size_t pair_smem_bytes(int H) {
  return (size_t)(2 * ((H + BK - 1) / BK) + kPairRing) * kFwdChunk + kFwdTail;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(kPairThreads, 1)
    pair_kernel(const __grid_constant__ FwdMaps maps, const FwdArgs a) {
  extern __shared__ __align__(1024) uint8_t fwd_smem[];
  constexpr int R = kPairRing;
  const int H = a.H, slices = (H + BK - 1) / BK;
  const uint32_t base = smem_u32(fwd_smem), blk = (uint32_t)slices * kFwdChunk;
  const uint32_t ring = base + 2 * blk, tail = ring + R * kFwdChunk;
  const uint32_t b_full = tail, b_empty = tail + 8 * R, b_ready = tail + 16 * R,
                 b_done = b_ready + 16;
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(fwd_smem + (tail - base) + 16 * R + 32);
  static_assert(16 * R + 36 <= kFwdTail, "barriers outgrew their slot");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * 2 * BM, z = blockIdx.y;
  const uint32_t cols = H <= 32 ? 32 : H <= 64 ? 64 : H <= 128 ? 128 : 256;  // of one tile
  const int tiles = m0 + BM < a.n ? 2 : 1;
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 2 * R; i++) mbar_init(b_full + 8 * i, 1);
#pragma unroll
    for (int t = 0; t < 2; t++) {
      mbar_init(b_ready + 8 * t, kPairWarps);
      mbar_init(b_done + 8 * t, 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(2 * cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)tmem_slot;
  auto units_of = [&](int l) { return l < kHidden ? H : kOutPad; };
  auto depth_of = [&](int l) { return l == 0 ? kInPad : H; };
  bool ok = true;
  if (warp == kPairWarps + 1) {
    // the weights: every layer's chunks, K slice by K slice, 128 output units
    // at a time, once per tile
    if (lane == 0) {
      int c = 0;
      for (int l = 0; l <= kHidden && ok; l++)
        for (int t = 0; t < tiles && ok; t++)
          for (int s = 0; s * BK < depth_of(l) && ok; s++)
            for (int h = 0; h * 128 < units_of(l); h++) {
              const int b = c % R;
              if (c >= R && !mbar_wait(b_empty + 8 * b, (uint32_t)((c / R - 1) & 1))) {
                ok = false;
                break;
              }
              mbar_expect_tx(b_full + 8 * b, (uint32_t)kFwdChunk);
              tma_load3(ring + (uint32_t)b * kFwdChunk, &maps.w[l], s * BK, h * 128, z, b_full + 8 * b);
              c++;
            }
      // no copy may land after the CTA ends (bounded)
      if (!ok)
        for (int k = c > R ? c - R : 0; k < c; k++)
          mbar_wait(b_full + 8 * (k % R), (uint32_t)((k / R) & 1));
    }
    __syncwarp();
  } else if (warp == kPairWarps) {
    if (lane == 0) {
      int c = 0;
      for (int l = 0; l <= kHidden && ok; l++)
        for (int t = 0; t < tiles && ok; t++) {
          if (!mbar_wait(b_ready + 8 * t, (uint32_t)(l & 1))) {
            ok = false;
            break;
          }
          tc_fence_after();
          const int K = depth_of(l), N = units_of(l);
          for (int s = 0; s * BK < K && ok; s++)
            for (int h = 0; h * 128 < N; h++) {
              const int b = c % R;
              if (!mbar_wait(b_full + 8 * b, (uint32_t)((c / R) & 1))) {
                ok = false;
                break;
              }
              tc_fence_after();
              const int nn = N - h * 128 < 128 ? N - h * 128 : 128;
              const int steps = K - s * BK < BK ? (K - s * BK) / 16 : BK / 16;
              const uint64_t da = sw128_desc(base + t * blk + (uint32_t)s * kFwdChunk);
              const uint64_t db = sw128_desc(ring + (uint32_t)b * kFwdChunk);
              const uint32_t id = idesc_bf16(BM, nn);
              for (int k = 0; k < steps; k++)
                mma_bf16(tmem + t * cols + h * 128, da + 2u * k, db + 2u * k, id,
                         (s > 0 || k > 0) ? 1u : 0u);
              mma_commit(b_empty + 8 * b);
              c++;
            }
          mma_commit(b_done + 8 * t);
        }
      // no MMA may run after the CTA ends (bounded)
      if (!ok)
        for (int k = c > R ? c - R : 0; k < c; k++)
          mbar_wait(b_empty + 8 * (k % R), (uint32_t)((k / R) & 1));
    }
    __syncwarp();
  } else {
    // layer 0's operands: transformed queries, BF16, columns 7..15 zero
    if (tid < 2 * BM) {
      const int row = m0 + tid, r = tid & (BM - 1);
      __align__(16) bf16 v[kInPad];
#pragma unroll
      for (int d = 0; d < kInPad; d++)
        v[d] = __float2bfloat16_rn(
            d < kIn && row < a.n ? xform(a.x[(size_t)row * kIn + d], d, a.xf) : 0.0f);
#pragma unroll
      for (int c = 0; c < 2; c++)
        *reinterpret_cast<uint4*>(fwd_smem + (tid >> 7) * blk + r * 128 + ((c ^ (r & 7)) << 4)) =
            reinterpret_cast<const uint4*>(v)[c];
    }
    // this warp is done with tile t: its stores are visible to the tensor
    // cores, its reads of the accumulator complete
    auto hand_over = [&](int t) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_ready + 8 * t);
    };
    for (int t = 0; t < tiles; t++) hand_over(t);
    for (int l = 0; l <= kHidden && ok; l++)
      for (int t = 0; t < tiles; t++) {
        if (!mbar_wait(b_done + 8 * t, (uint32_t)(l & 1))) {
          ok = false;
          break;
        }
        __syncwarp();
        tc_fence_after();
        const int mt = m0 + t * BM, r = (warp & 3) * 32 + lane;
        const uint32_t acc = tmem + t * cols + ((uint32_t)((warp & 3) * 32) << 16);
        const bool rows_in = mt + (warp & 3) * 32 < a.n;  // any valid row of this warp's 32
        const float* bias = a.p + z * a.P + a.b_off[l];
        if (l < kHidden) {
          if (rows_in) {
            // the accumulator's next 16 columns are on their way while these
            // are worked on
            constexpr int kStep = kPairWarps / 4 * 16;
            auto work = [&](int c0, const uint32_t (&v)[16]) {
              __align__(16) bf16 o[16];
#pragma unroll
              for (int j = 0; j < 16; j += 4) {
                const float4 b4 = __ldg(reinterpret_cast<const float4*>(bias + c0 + j));
                o[j] = __float2bfloat16_rn(gelu_f(__uint_as_float(v[j]) + b4.x));
                o[j + 1] = __float2bfloat16_rn(gelu_f(__uint_as_float(v[j + 1]) + b4.y));
                o[j + 2] = __float2bfloat16_rn(gelu_f(__uint_as_float(v[j + 2]) + b4.z));
                o[j + 3] = __float2bfloat16_rn(gelu_f(__uint_as_float(v[j + 3]) + b4.w));
              }
              const int ch = (c0 % BK) / 8;
              uint8_t* row = fwd_smem + t * blk + (size_t)(c0 / BK) * kFwdChunk + r * 128;
#pragma unroll
              for (int c = 0; c < 2; c++)
                *reinterpret_cast<uint4*>(row + (((ch + c) ^ (r & 7)) << 4)) =
                    reinterpret_cast<const uint4*>(o)[c];
            };
            uint32_t va[16], vb[16];
            int c0 = (warp >> 2) * 16;
            if (c0 < H) tmem_ld16_start(acc + (uint32_t)c0, va);
#pragma unroll 1
            for (; c0 < H; c0 += 2 * kStep) {
              tmem_ld16_wait(va);
              if (c0 + kStep < H) tmem_ld16_start(acc + (uint32_t)(c0 + kStep), vb);
              work(c0, va);
              if (c0 + kStep >= H) break;
              tmem_ld16_wait(vb);
              if (c0 + 2 * kStep < H) tmem_ld16_start(acc + (uint32_t)(c0 + 2 * kStep), va);
              work(c0 + kStep, vb);
            }
          }
          hand_over(t);
        } else if (warp < 4 && rows_in) {
          float v[16];
          tmem_ld16(acc, v);
          const int row = mt + r;
          if (row < a.n)
            *reinterpret_cast<float4*>(a.Y + ((size_t)z * a.n + row) * kOut) =
                make_float4(v[0] + __ldg(bias), v[1] + __ldg(bias + 1), v[2] + __ldg(bias + 2),
                            v[3] + __ldg(bias + 3));
        }
      }
  }
  if (!ok && lane == 0) atomicOr(a.status, kStatusTimeout);
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(2 * cols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// The network on a thread-block cluster: a training step's forward pass, loss
// and back-propagation, or a small inference batch.  A cluster of ceil(H / 32)
// CTAs takes a 128-row tile of one member; CTA c owns units 32 c .. 32 c + 31
// of every hidden layer.  Per layer it multiplies the tile's whole activation
// block (in its shared memory) by its 32 rows of the weights, applies the
// output pass to 128 x 32 values, and sends the BF16 results, one contiguous
// 8 KB slice of the next activation block, to every other CTA of the cluster
// (bulk copies into distributed shared memory, counted on the receiver's
// barrier).  A CTA's own accumulators stay in tensor memory, so
// back-propagation finds the pre-activations there; its weight rows, forward
// and transposed, are fetched ahead of use.  The output layer (16 units) is
// computed by every CTA for itself, and so is the loss gradient.  What the
// weight gradients need later goes to global memory transposed: inputs, hidden
// activations, errors.
//
// Two activation blocks and no cluster barrier per layer are enough: a CTA
// sends slices of layer l + 1 only after it received every slice of layer l,
// which each sender sent after its own products of layer l - 1, the last to
// read the block that layer l + 1 is written to.
//
// Bound by latency: nine dependent layers, of which the exchange of the slices
// (56 KB into every CTA) and the products take 2.1 us, the GELUs 0.8 us; 29 us
// at batch 256, H = 256, five members, and a training step 47 us with the
// gradient kernel.  A launch per layer and pass (14 GEMMs and 10 small kernels,
// 7 to 20 us each) took 165 us a step.  16-byte remote stores by every thread
// instead of the bulk copies took 2.6 us a layer more than the copies.  Programmatic
// dependent launch hides the start of each kernel behind the one before.
constexpr int kUnits = 32;  // hidden units of a CTA
constexpr int kChainThreads = 512;
constexpr int kSlice = 128 * kUnits * 2;  // bytes of a CTA's slice of an activation block
constexpr uint32_t kColY = 128, kColB = 160, kChainCols = 256;  // tensor-memory columns

struct ChainMaps {
  CUtensorMap w[kHidden + 1];   // W_l: boxes of 64 (K) x 32 units (output layer: 16)
  CUtensorMap wt[kHidden + 1];  // W_l transposed (l >= 1): boxes of 64 x 32
};
struct ChainArgs {
  int rows, H;
  // inference: raw queries and their transform, outcomes [m][rows][4]
  const float* x;
  Xform xf;
  float* Y;
  // training: transformed rows and targets, drawn with replacement by a hash
  // of (seed, member, step, row), or taken in order (direct)
  const bf16* X;
  const float* T;
  int n, direct;
  unsigned long long seed;
  const long long* d_step;
  long long step_off;     // this launch is step *d_step + step_off
  const float* w;
  const float* p;
  long long P;
  int b_off[kHidden + 1];
  bf16* Xt;               // [m][16][rows]
  bf16* Ht[kHidden];      // [m][H][rows]
  bf16* dZt[kHidden];     // [m][H][rows]
  bf16* dYt;              // [m][16][rows]
  float* dYft;            // [m][16][rows]
  double* loss;           // [m][4 tiles]: one sum per warp of rows
  unsigned* status;
};

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// This CTA's stores to its shared memory are visible to its tensor cores and
// bulk copies.
__device__ __forceinline__ void proxy_fence() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
// Programmatic dependent launch: wait until the kernel before this one on the
// stream has finished and its writes are visible; let the next one start.
__device__ __forceinline__ void wait_for_previous() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void let_next_start() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

int chain_ctas(int H) { return (H + kUnits - 1) / kUnits; }
size_t chain_smem_bytes(int H) {
  const size_t slices = (H + BK - 1) / BK;
  return 2 * (size_t)chain_ctas(H) * kSlice + kSlice + slices * (3 * kUnits * 128 + 16 * 128) +
         2 * kUnits * 128 + kFwdTail + 1024;  // (blocks may end on half a kilobyte multiple)
}

template <bool TRAIN>
__global__ void __launch_bounds__(kChainThreads, 1)
    chain_kernel(const __grid_constant__ ChainMaps maps, const ChainArgs a) {
  extern __shared__ __align__(1024) uint8_t fwd_smem[];
  const int H = a.H, slices = (H + BK - 1) / BK;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t rank, nrank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(rank));
  asm volatile("mov.u32 %0, %%cluster_nctarank;\n" : "=r"(nrank));
  const int tile = blockIdx.x / nrank, m0 = tile * BM, z = blockIdx.y;
  const int u0 = rank * kUnits, nu = H - u0 < kUnits ? H - u0 : kUnits;
  // shared memory: two activation blocks, the loss gradient's operand, three
  // weight slots (W_1..3, then W_3..1 transposed), W_0, W_4 transposed, W_4
  const uint32_t base = smem_u32(fwd_smem);
  const uint32_t blk = nrank * kSlice, slot = (uint32_t)slices * kUnits * 128;
  const uint32_t s_dy = base + 2 * blk, s_w = s_dy + kSlice, s_w0 = s_w + 3 * slot;
  const uint32_t s_wt4 = s_w0 + kUnits * 128, s_w4 = s_wt4 + kUnits * 128;
  const uint32_t tail = s_w4 + (uint32_t)slices * 16 * 128;
  // barriers: W_0; the three slots; W_4 and its transpose; MMAs done; slices
  // of block 0 and 1 received
  const uint32_t b_w0 = tail, b_slot = tail + 8, b_w4 = tail + 32, b_mma = tail + 40,
                 b_in = tail + 48;
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(fwd_smem + (tail - base) + 64);
  float* const s_bias = reinterpret_cast<float*>(fwd_smem + (tail - base) + 128);  // [5][32]
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 8; i++) mbar_init(tail + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kChainCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  cluster_arrive();  // waited for before the first copy into another CTA
  // rows of units u0 .. of a weight matrix, all of K, into `dst`
  auto fetch = [&](const CUtensorMap* m, int K, int row, int box, uint32_t dst, uint32_t bar) {
    for (int s = 0; s * BK < K; s++) tma_load3(dst + s * box * 128, m, s * BK, row, z, bar);
  };
  // 16 BF16 values of a row as columns 0..15 of an operand slice at `s`
  auto put_row = [&](uint32_t s, const bf16* v) {
#pragma unroll
    for (int c = 0; c < 2; c++)
      *reinterpret_cast<uint4*>(fwd_smem + (s - base) + tid * 64 + ((c ^ ((tid >> 1) & 3)) << 4)) =
          reinterpret_cast<const uint4*>(v)[c];
  };
  // rows taken in order were prepared by the kernels just before; the training
  // rows and the step are constant during a call and need no wait
  if (TRAIN && a.direct) wait_for_previous();
  // layer 0's operand (every CTA for itself), BF16, columns 7..15 zero
  const int row = m0 + (tid & 127);
  const bool row_in = row < a.rows;
  float target[kOut] = {0.f, 0.f, 0.f, 0.f};
  __align__(16) bf16 v0[kInPad];
  if (tid < BM) {
    if (TRAIN) {
      uint4 q[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
      if (row_in) {
        int src = row;
        if (!a.direct) {
          const unsigned long long ctr =
              ((unsigned long long)z << 56) ^
              ((unsigned long long)(__ldcg(a.d_step) + a.step_off) << 24) ^ (unsigned)row;
          src = (int)(mix64(a.seed ^ mix64(ctr)) % (unsigned long long)a.n);
        }
        q[0] = __ldcg(reinterpret_cast<const uint4*>(a.X + (size_t)src * kInPad));
        q[1] = __ldcg(reinterpret_cast<const uint4*>(a.X + (size_t)src * kInPad) + 1);
        const float4 t4 = __ldcg(reinterpret_cast<const float4*>(a.T) + src);
        target[0] = t4.x;
        target[1] = t4.y;
        target[2] = t4.z;
        target[3] = t4.w;
      }
      reinterpret_cast<uint4*>(v0)[0] = q[0];
      reinterpret_cast<uint4*>(v0)[1] = q[1];
    } else {
#pragma unroll
      for (int d = 0; d < kInPad; d++)
        v0[d] = __float2bfloat16_rn(d < kIn && row_in ? xform(a.x[(size_t)row * kIn + d], d, a.xf) : 0.0f);
    }
    put_row(base, v0);
  }
  // Up to here nothing depends on the kernel before.  From here on: its
  // parameters; and it has finished reading what this one overwrites.
  if (TRAIN) {
    wait_for_previous();
    let_next_start();
  }
  if (tid == 0) {
    mbar_expect_tx(b_w0, kUnits * 128);
    fetch(&maps.w[0], kInPad, u0, kUnits, s_w0, b_w0);
    for (int l = 1; l < kHidden; l++) {
      mbar_expect_tx(b_slot + 8 * (l - 1), slot);
      fetch(&maps.w[l], H, u0, kUnits, s_w + (l - 1) * slot, b_slot + 8 * (l - 1));
    }
    mbar_expect_tx(b_w4, (uint32_t)slices * 16 * 128 + (TRAIN ? kUnits * 128 : 0));
    fetch(&maps.w[kHidden], H, 0, 16, s_w4, b_w4);
    if (TRAIN) fetch(&maps.wt[kHidden], kOutPad, u0, kUnits, s_wt4, b_w4);
  }
  if (tid < (kHidden + 1) * kUnits) {
    const int l = tid / kUnits, j = tid % kUnits;
    const int units = l < kHidden ? nu : kOutPad, first = l < kHidden ? u0 : 0;
    s_bias[tid] = j < units ? __ldcg(a.p + z * a.P + a.b_off[l] + first + j) : 0.0f;
  }
  if (TRAIN && tid < BM && rank == 0 && row_in)
#pragma unroll
    for (int d = 0; d < kInPad; d++) a.Xt[((size_t)z * kInPad + d) * a.rows + row] = v0[d];
  proxy_fence();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)tmem_slot;
  const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
  const bool rows_in = m0 + (warp & 3) * 32 < a.rows;
  const int col = (warp >> 2) * 8;  // this warp's 8 of the CTA's units
  const bool mine = rows_in && col < nu;
  bool ok = true;
  uint32_t mma_phase = 0, in_phase = 0;  // in_phase: bit b for block b
  // D[128 x N] at tensor-memory column dcol = (operand slices at sa, K deep)
  // times (weight rows at sb, `box` rows a 64-wide slice)^T, once barrier `bar`
  // says the weights are there; block >= 0: once its slices were received
  auto multiply = [&](uint32_t sa, int block, uint32_t sb, int box, int K, int N, uint32_t dcol,
                      uint32_t bar, uint32_t parity) {
    if (tid == 0) {
      if (!mbar_wait(bar, parity)) ok = false;
      if (block >= 0) {
        if (!mbar_wait(b_in + 8 * block, (in_phase >> block) & 1)) ok = false;
        in_phase ^= 1u << block;
      }
      tc_fence_after();
      // descriptors count in 16 bytes: 32 bytes a step of K inside a slice
      const uint32_t id = idesc_bf16(BM, N);
      const uint64_t da = sw64_desc(sa), db = sw128_desc(sb);
#pragma unroll 4
      for (int k = 0; k < K / 16; k++)
        mma_bf16(tmem + dcol, da + (uint32_t)((k >> 1) * (kSlice / 16) + 2 * (k & 1)),
                 db + (uint32_t)((k >> 2) * (box * 8) + 2 * (k & 3)), id, k > 0 ? 1u : 0u);
      mma_commit(b_mma);
    }
    __syncwarp();
    if (!mbar_wait(b_mma, mma_phase)) ok = false;
    mma_phase ^= 1;
    __syncwarp();
    tc_fence_after();
  };
  // this CTA's 8 BF16 values of row `row`, units u0 + col .., into block b
  auto put = [&](const bf16* o, uint32_t b) {
    const int r = (warp & 3) * 32 + lane;
    *reinterpret_cast<uint4*>(fwd_smem + b * blk + rank * kSlice + r * 64 +
                              (((col / 8) ^ ((r >> 1) & 3)) << 4)) =
        *reinterpret_cast<const uint4*>(o);
  };
  // the CTA's slice of block b to every other CTA of the cluster
  auto send = [&](uint32_t b) {
    __syncwarp();
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
      mbar_expect_tx(b_in + 8 * b, (nrank - 1) * kSlice);
      const uint32_t src = base + b * blk + rank * kSlice;
      for (uint32_t j = 1; j < nrank; j++) {
        const uint32_t to = rank + j < nrank ? rank + j : rank + j - nrank;
        uint32_t dst, bar;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(dst) : "r"(src), "r"(to));
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(bar) : "r"(b_in + 8 * b), "r"(to));
        asm volatile(
            "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2,"
            " [%3];\n" ::"r"(dst),
            "r"(src), "r"((uint32_t)kSlice), "r"(bar)
            : "memory");
      }
    }
    __syncwarp();
  };
  // the same values, transposed, to global memory (lane = row: 64-byte runs)
  auto keep = [&](const bf16* o, bf16* out) {
    if (!row_in) return;
    bf16* dst = out + ((size_t)z * H + u0 + col) * a.rows + row;
#pragma unroll
    for (int j = 0; j < 8; j++) dst[(size_t)j * a.rows] = o[j];
  };

  for (int l = 0; l < kHidden; l++) {
    if (l == 0)
      multiply(base, -1, s_w0, kUnits, kInPad, nu, 0, b_w0, 0);
    else
      multiply(base + (l & 1) * blk, l & 1, s_w + (l - 1) * slot, kUnits, H, nu, l * kUnits,
               b_slot + 8 * (l - 1), 0);
    if (TRAIN && tid == 0 && l >= 1) {
      // this layer's weights are used: the slot takes W_3 .. W_1 transposed
      mbar_expect_tx(b_slot + 8 * (l - 1), slot);
      fetch(&maps.wt[kHidden - l], H, u0, kUnits, s_w + (l - 1) * slot, b_slot + 8 * (l - 1));
    }
    __syncwarp();
    if (l == 0) cluster_wait();  // every CTA of the cluster has started
    __align__(16) bf16 o[8];
    if (mine) {
      float v[8];
      tmem_ld8(tmem + lanes + l * kUnits + col, v);
#pragma unroll
      for (int j = 0; j < 8; j++)
        o[j] = __float2bfloat16_rn(gelu_f(v[j] + s_bias[l * kUnits + col + j]));
      put(o, (l + 1) & 1);
    }
    send((l + 1) & 1);
    if (TRAIN && mine) keep(o, a.Ht[l]);
  }
  multiply(base, 0, s_w4, 16, H, 16, kColY, b_w4, 0);
  float diff[kOut] = {0.f, 0.f, 0.f, 0.f};
  const float inv = 2.0f / (float)(a.rows * kOut);
  if (tid < BM && rows_in) {
    const float* bias = s_bias + kHidden * kUnits;
    float v[16];
    tmem_ld16(tmem + lanes + kColY, v);
    if (!TRAIN) {
      if (rank == 0 && row_in)
        *reinterpret_cast<float4*>(a.Y + ((size_t)z * a.rows + row) * kOut) =
            make_float4(v[0] + bias[0], v[1] + bias[1], v[2] + bias[2], v[3] + bias[3]);
    } else {
      // gradient of the loss 1 / (4 rows) sum w (y - t)^2
      __align__(16) bf16 o[kOutPad];
#pragma unroll
      for (int d = 0; d < kOutPad; d++) {
        float g = 0.0f;
        if (d < kOut && row_in) {
          diff[d] = v[d] + bias[d] - target[d];
          g = inv * a.w[d] * diff[d];
        }
        o[d] = __float2bfloat16_rn(g);
      }
      put_row(s_dy, o);
    }
  }
  // The loss and what the output layer's gradients need, by the first CTA
  // while its slices of the next errors are on their way.
  auto store_loss = [&]() {
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < kOutPad; d++) {
      float g = 0.0f;
      if (d < kOut && row_in) {
        acc += (double)a.w[d] * diff[d] * diff[d];
        g = inv * a.w[d] * diff[d];
      }
      if (row_in) {
        const size_t at = ((size_t)z * kOutPad + d) * a.rows + row;
        a.dYt[at] = __float2bfloat16_rn(g);
        a.dYft[at] = g;
      }
    }
    for (int k = 16; k > 0; k >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, k);
    if (lane == 0) {
      a.loss[(size_t)z * 4 * (gridDim.x / nrank) + tile * 4 + warp] = acc / (double)(a.rows * kOut);
      if (!isfinite(acc)) atomicOr(a.status, kStatusNonFinite);
    }
    __syncwarp();
  };
  if (TRAIN) {
    __syncwarp();
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    for (int l = kHidden - 1; l >= 0; l--) {
      // errors of layer l: (errors of layer l + 1) W_{l+1}, times gelu'(z_l)
      if (l == kHidden - 1)
        multiply(s_dy, -1, s_wt4, kUnits, kOutPad, nu, kColB, b_w4, 0);
      else
        multiply(base + ((l + 1) & 1) * blk, (l + 1) & 1, s_w + (kHidden - 2 - l) * slot, kUnits, H,
                 nu, kColB, b_slot + 8 * (kHidden - 2 - l), 1);
      __align__(16) bf16 o[8];
      if (mine) {
        float v[8], zl[8];
        tmem_ld8(tmem + lanes + kColB + col, v);
        tmem_ld8(tmem + lanes + l * kUnits + col, zl);
#pragma unroll
        for (int j = 0; j < 8; j++)
          o[j] = __float2bfloat16_rn(v[j] * gelu_grad_f(zl[j] + s_bias[l * kUnits + col + j]));
        if (l > 0) put(o, l & 1);
      }
      if (l > 0) send(l & 1);
      if (mine) keep(o, a.dZt[l]);
      if (l == kHidden - 1 && rank == 0 && tid < BM) store_loss();
    }
  }
  if (!ok) atomicOr(a.status, kStatusTimeout);
  if (tid == 0 && !ok) {
    // a wait gave up: no copy may land and no MMA run after the CTA ends
    // (bounded again)
    mbar_wait(b_w0, 0);
    for (int i = 0; i < 3; i++) {
      mbar_wait(b_slot + 8 * i, 0);
      if (TRAIN) mbar_wait(b_slot + 8 * i, 1);
    }
    mbar_wait(b_w4, 0);
    mbar_wait(b_mma, mma_phase ^ 1);
  }
  // no CTA ends while another may still send to it or read from it
  __syncwarp();
  tc_fence_before();
  cluster_arrive();
  cluster_wait();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kChainCols)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Weight gradients and their Adam update in one launch: a CTA per 128 x 64
// tile of a layer's weights of one member.  The gradient dW = dZ^T A (A the
// layer's input; K = the minibatch) is accumulated in tensor memory, and the
// output pass updates the tile's parameters, moments and BF16 copies at once,
// so gradients never reach memory.  The bias gradients (row sums of dZ^T) of
// the tile's rows are shared by the CTAs of a row of tiles and taken by warps
// 1..15 while thread 0 drives the tensor cores.
//
// Bound by the parameter traffic, 28 bytes a parameter (29 MB for five members
// of H = 256), which stays in L2, and by Adam's divisions and roots: 9 us; a
// gradient GEMM per layer, row sums, Adam with strided writes of the transposed
// copy and a counter launch took 85 us.
constexpr int kUpdateThreads = 512;
constexpr int kUpdateBN = 64;
constexpr size_t kUpdateSmem = kStages * (size_t)stage_bytes<kUpdateBN>() + kFwdTail;

struct UpdateMaps {
  CUtensorMap a[kHidden + 1];  // dZ_l^T, boxes of 64 (rows of the minibatch) x 128
  CUtensorMap b[kHidden + 1];  // input of layer l, transposed, boxes of 64 x 64
};
struct UpdateArgs {
  int rows, grads_only;
  int first[kHidden + 2];  // first tile of each layer
  Layout L;
  float *p, *g, *m, *v;
  bf16 *Wb, *WbT;
  const bf16* dZt[kHidden];
  const float* dYft;
  float lr, beta1, beta2, eps;
  const long long* d_step;
  long long step_off;
  const long long* d_sched;
  unsigned* status;
};

// Loads that bypass L1, which may hold the line of an earlier step.
__device__ __forceinline__ float ld_l2(const float* p) { return __ldcg(p); }
__device__ __forceinline__ float ld_l2(const bf16* p) {
  const unsigned short u = __ldcg(reinterpret_cast<const unsigned short*>(p));
  return __bfloat162float(__ushort_as_bfloat16(u));
}

struct AdamStep {
  float lr, bc1, bc2, y1, y2;  // y: reciprocals of bc1, bc2, rounded to nearest
};

// a / b rounded to nearest, given y = 1 / b rounded to nearest: the quotient
// a y corrected once by its exact remainder (Markstein, "Computation of
// elementary functions on the IBM RISC System/6000", 1990, theorem on
// quotients from a correctly rounded reciprocal).  The remainder is exact
// while it does not underflow; moments below 1e-30, where it may, are far
// below eps in Adam's denominator; an infinite quotient stays infinite.  The
// general division takes a range check and a branch each, a fifth of this
// kernel's instructions.
__device__ __forceinline__ float quotient(float a, float b, float y) {
  const float q = __fmul_rn(a, y);
  return fabsf(q) < INFINITY ? fmaf(fmaf(-q, b, a), y, q) : q;
}

// One parameter: moments, update; returns the new value.
__device__ __forceinline__ float adam_update(const UpdateArgs& a, const AdamStep& s, size_t i,
                                             float gi, float m0, float v0, float p0) {
  // the rounding of each term is written out, so that results do not hang on
  // the compiler's choice of which product to fuse
  const float mi = fmaf(1.0f - a.beta1, gi, __fmul_rn(a.beta1, m0));
  const float vi = fmaf(__fmul_rn(1.0f - a.beta2, gi), gi, __fmul_rn(a.beta2, v0));
  a.m[i] = mi;
  a.v[i] = vi;
  const float pi =
      p0 - s.lr * quotient(mi, s.bc1, s.y1) / (sqrtf(quotient(vi, s.bc2, s.y2)) + a.eps);
  a.p[i] = pi;
  return pi;
}

__global__ void __launch_bounds__(kUpdateThreads, 1)
    update_kernel(const __grid_constant__ UpdateMaps maps, const UpdateArgs a) {
  extern __shared__ __align__(1024) uint8_t fwd_smem[];
  constexpr int BN = kUpdateBN;
  uint64_t* bars = reinterpret_cast<uint64_t*>(fwd_smem + kStages * stage_bytes<BN>());
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int z = blockIdx.y;
  int l = 0;
#pragma unroll
  for (int k = 1; k <= kHidden; k++)
    if ((int)blockIdx.x >= a.first[k]) l = k;
  const int nin = a.L.nin[l], nout = a.L.nout[l];
  const int nt = (nin + BN - 1) / BN, tile = blockIdx.x - a.first[l];
  const int m0 = tile / nt * BM, jt = tile % nt, n0 = jt * BN;
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < 2 * kStages; i++) mbar_init(smem_u32(&bars[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"((uint32_t)tmem_cols<BN>())
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  AdamStep s{a.lr, 1.0f, 1.0f, 1.0f, 1.0f};
  if (!a.grads_only) {
    const long long step = __ldcg(a.d_step) + a.step_off;
    const long long first = a.d_sched ? __ldcg(a.d_sched) : 0;
    const long long steps = a.d_sched ? __ldcg(a.d_sched + 1) : 0;
    if (steps > 0) {
      const float frac = (float)(step - first) / (float)steps;
      s.lr *= 0.5f * (1.0f + cospif(fminf(fmaxf(frac, 0.0f), 1.0f)));
    }
    const float t = (float)(step + 1);
    s.bc1 = 1.0f - powf(a.beta1, t);
    s.bc2 = 1.0f - powf(a.beta2, t);
    s.y1 = __frcp_rn(s.bc1);
    s.y2 = __frcp_rn(s.bc2);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *(volatile uint32_t*)tmem_slot;
  const size_t member = (size_t)z * a.L.total;
  // this warp's 32 rows x 16 columns, taken row by row, half-warps on two rows
  // (64-byte runs of p, m and v), which are fetched before the gradient is there
  const int mw = m0 + (warp & 3) * 32, jj = lane & 15, rh = lane >> 4;
  const int c0 = (warp >> 2) * 16, n = n0 + c0 + jj;  // nin is a multiple of 16
  const bool mine = mw < nout && n0 + c0 < nin;
  const size_t at = member + a.L.w_off[l] + (size_t)(mw + rh) * nin + n;
  float pm[16], pv[16], pp[16];
  if (mine && !a.grads_only) {
#pragma unroll
    for (int i = 0; i < 16; i++)
      if (mw + 2 * i + rh < nout) {
        pm[i] = __ldcg(a.m + at + (size_t)(2 * i) * nin);
        pv[i] = __ldcg(a.v + at + (size_t)(2 * i) * nin);
        pp[i] = __ldcg(a.p + at + (size_t)(2 * i) * nin);
      }
  }
  // Parameters and moments are the previous step's, finished before the
  // kernel that this one follows let it start; what follows is that kernel's.
  wait_for_previous();
  let_next_start();
  bool ok = true;
  if (tid == 0) {
    ok = gemm_pipeline<BN>(fwd_smem, bars, &maps.a[l], &maps.b[l], m0, n0, z, z, a.rows, tmem);
  } else if (warp > 0) {
    // bias gradients of rows m0 + jt, m0 + jt + nt, ..: four rows of a warp at
    // a time, lanes along the minibatch; lane j then updates row j of the four
    const int count = (min(BM, nout - m0) - jt + nt - 1) / nt;
    const bf16* src = l < kHidden ? a.dZt[l] + (size_t)z * nout * a.rows : nullptr;
    const float* src32 = a.dYft + (size_t)z * kOutPad * a.rows;
    for (int i0 = (warp - 1) * 4; i0 < count; i0 += 15 * 4) {
      float acc[4] = {0.f, 0.f, 0.f, 0.f};
      auto sum_rows = [&](auto* p) {
#pragma unroll 4
        for (int c = lane; c < a.rows; c += 32)
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const int u = m0 + jt + min(i0 + j, count - 1) * nt;
            acc[j] += (float)ld_l2(p + (size_t)u * a.rows + c);
          }
      };
      if (src)
        sum_rows(src);
      else
        sum_rows(src32);
      float mine_acc = 0.0f;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_down_sync(0xffffffffu, acc[j], o);
        const float t = __shfl_sync(0xffffffffu, acc[j], 0);
        if (lane == j) mine_acc = t;
      }
      if (lane < 4 && i0 + lane < count) {
        const size_t i = member + a.L.b_off[l] + m0 + jt + (i0 + lane) * nt;
        if (a.grads_only)
          a.g[i] = mine_acc;
        else
          adam_update(a, s, i, mine_acc, __ldcg(a.m + i), __ldcg(a.v + i), __ldcg(a.p + i));
      }
      __syncwarp();
    }
  }
  ok = __syncthreads_and(ok);
  tc_fence_after();
  if (ok) {
    if (mine) {
      // through shared memory, as the operand ring is free; the transposed
      // BF16 copy is written from the lane = row layout
      float* T = reinterpret_cast<float*>(fwd_smem) + warp * (32 * 17);
      float v[16];
      tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 16; j++) T[lane * 17 + j] = v[j];
      __syncwarp();
#pragma unroll
      for (int i = 0; i < 16; i++) {
        const int r = 2 * i + rh;
        if (mw + r >= nout) continue;
        const size_t idx = at + (size_t)(2 * i) * nin;
        const float x = T[r * 17 + jj];
        if (a.grads_only) {
          a.g[idx] = x;
          continue;
        }
        const bf16 b = __float2bfloat16_rn(adam_update(a, s, idx, x, pm[i], pv[i], pp[i]));
        a.Wb[idx] = b;
        T[r * 17 + jj] = __bfloat162float(b);
      }
      __syncwarp();
      if (!a.grads_only && mw + lane < nout) {
        bf16* dst = a.WbT + member + a.L.w_off[l] + (size_t)(n0 + c0) * nout + mw + lane;
#pragma unroll
        for (int j = 0; j < 16; j++) dst[(size_t)j * nout] = __float2bfloat16_rn(T[lane * 17 + j]);
      }
    }
  } else if (tid == 0) {
    atomicOr(a.status, kStatusTimeout);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((uint32_t)tmem_cols<BN>())
                 : "memory");
  }
}

// Answers of QB queries per block: a thread per (query, outcome) decodes and
// reduces over the members; the queries that pass the box and spread tests
// are listed, and warps look for a training point within nn_cut of them, a
// lane per training point, four points in flight per lane, stopping at the
// first hit (the gate asks whether the nearest point is within nn_cut, so any
// point within it decides).  A short list gives each query several warps.
//
// Bound by the distance search (FP32 pipe and L1 loads of the points, laid
// out by column so that a warp reads 128-byte lines).  One thread scanning
// all points for its query took 194 us for one query and 220 us for 65536
// against 4096 points (a serial chain of 4096 shared-memory reads per query),
// and decoding another 10 to 28 us; now 10 and 37 us for both.
constexpr int kAnswerThreads = 256;
constexpr int kScan = 4;  // points in flight per lane

template <int QB>
__global__ void __launch_bounds__(kAnswerThreads) answer_kernel(const GateArgs a) {
  constexpr int kWarps = kAnswerThreads / 32;
  __shared__ int list[QB];
  __shared__ int hit[QB];
  __shared__ int count;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q0 = blockIdx.x * QB;
  if (tid == 0) {
    count = 0;
    if (blockIdx.x == 0) *a.status_out = *(volatile const unsigned*)a.status;
  }
  __syncthreads();
  // decode: the four outcomes of a query on four neighbouring lanes
  constexpr int kDecode = QB * kOut < 32 ? 32 : QB * kOut;  // whole warps
  for (int k = tid; k < kDecode; k += kAnswerThreads) {
    const int q = q0 + (k >> 2), d = k & 3;
    const bool in = q < a.n && k < QB * kOut;
    bool ok = in;
    if (in) {
      double s = 0.0, s2 = 0.0;
      const float sc = a.xout.scale[d], mn = a.xout.mean[d];
      const bool lg = (a.xout.log_mask >> d) & 1;
      for (int mem = 0; mem < a.members; mem++) {
        float v = a.Y[((size_t)mem * a.n + q) * kOut + d] * sc + mn;
        if (lg) v = expf(v);
        s += v;
        s2 += (double)v * v;
      }
      const double mu = s / a.members;
      const float muf = (float)mu, sdf = (float)sqrt(fmax(s2 / a.members - mu * mu, 0.0));
      a.mean[(size_t)q * kOut + d] = muf;
      a.sd[(size_t)q * kOut + d] = sdf;
      if (d < 2) ok = isfinite(muf) && sdf <= (d == 0 ? a.tau : a.tau_v) * fabsf(muf);
      if (a.accept)
        for (int j = d; j < kIn; j += kOut) {
          const float raw = a.x[(size_t)q * kIn + j];
          ok = ok && raw >= a.lo[j] && raw <= a.hi[j];
        }
    }
    // every lane of the warp is here
    const unsigned votes = __ballot_sync(0xffffffffu, ok) >> (lane & ~3);
    if (in && a.accept && d == 0) {
      a.accept[q] = 0;
      if ((votes & 0xFu) == 0xFu) {
        const int at = atomicAdd(&count, 1);
        list[at] = q;
        hit[at] = 0;
      }
    }
  }
  if (!a.accept) return;
  __syncthreads();
  const int m = count;
  const int share = m >= 5 ? 1 : m >= 3 ? 2 : m == 2 ? 4 : kWarps;  // warps per query
  const int groups = kWarps / share, part = warp % share;
  for (int i = warp / share; i < m; i += groups) {
    const int q = list[i];
    float mine = 0.0f;
    if (lane < kIn) mine = xform(a.x[(size_t)q * kIn + lane], lane, a.xin);
    float xq[kIn];
#pragma unroll
    for (int d = 0; d < kIn; d++) xq[d] = __shfl_sync(0xffffffffu, mine, d);
    bool found = sqrtf(3.0e38f) <= a.nn_cut;  // a cut beyond any distance
    for (int t0 = part * 32 * kScan; t0 < a.nt && !found; t0 += share * 32 * kScan) {
      float best = 3.0e38f;
      float d2[kScan];
#pragma unroll
      for (int j = 0; j < kScan; j++) d2[j] = 0.0f;
#pragma unroll
      for (int d = 0; d < kIn; d++) {
        const float* col = a.Xt + (size_t)d * a.ldt + t0 + lane;  // ldt: padded to whole groups
#pragma unroll
        for (int j = 0; j < kScan; j++) {
          const float e = xq[d] - __ldg(col + 32 * j);
          d2[j] += e * e;
        }
      }
#pragma unroll
      for (int j = 0; j < kScan; j++)
        if (t0 + lane + 32 * j < a.nt) best = fminf(best, d2[j]);
      found = __any_sync(0xffffffffu, sqrtf(best) <= a.nn_cut);
      if (share > 1 && !found) found = __any_sync(0xffffffffu, *(volatile int*)&hit[i] != 0);
    }
    if (found && lane == 0) {
      hit[i] = 1;
      a.accept[q] = 1;
    }
  }
}

inline unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_prep_inputs(const float* x, int n, const Xform& xf, bf16* X, float* Xf, int ldx,
                               cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  prep_inputs_kernel<<<blocks(n, 128), 128, 0, s>>>(x, n, xf, X, Xf, ldx);
  return cudaGetLastError();
}

cudaError_t launch_prep_targets(const float* y, int n, const Xform& yf, float* T, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  prep_targets_kernel<<<blocks(n, 128), 128, 0, s>>>(y, n, yf, T);
  return cudaGetLastError();
}

__global__ void schedule_begin_kernel(const long long* __restrict__ d_step, long long* d_sched,
                                      long long steps) {
  d_sched[0] = *d_step;
  d_sched[1] = steps;
}

cudaError_t launch_schedule_begin(const long long* d_step, long long* d_sched, long long steps,
                                  cudaStream_t s) {
  schedule_begin_kernel<<<1, 1, 0, s>>>(d_step, d_sched, steps);
  return cudaGetLastError();
}

cudaError_t launch_cast_params(const float* p, const Layout& L, int members, bf16* Wb, bf16* WbT,
                               cudaStream_t s) {
  cast_params_kernel<<<blocks(L.total * members, 256), 256, 0, s>>>(p, L, members, Wb, WbT);
  return cudaGetLastError();
}

namespace {

__global__ void advance_step_kernel(long long* d_step, int by) { *d_step += by; }

template <bool TRAIN>
cudaError_t launch_chain(const ChainMaps& maps, const ChainArgs& a, int members, cudaStream_t s) {
  const int ctas = chain_ctas(a.H);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks(a.rows, BM) * ctas, members);
  cfg.blockDim = dim3(kChainThreads);
  cfg.dynamicSmemBytes = chain_smem_bytes(a.H);
  cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = TRAIN ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, chain_kernel<TRAIN>, maps, a);
}

// Tensor maps of the members' weights for chain_kernel.
cudaError_t chain_maps(ChainMaps* m, const Layout& L, int members, const bf16* Wb, const bf16* WbT) {
  cudaError_t e = cudaSuccess;
  for (int l = 0; l <= kHidden && e == cudaSuccess; l++) {
    e = make_map(&m->w[l], Wb + L.w_off[l], L.nin[l], L.nout[l], L.nin[l], L.total, members,
                 l == kHidden ? kOutPad : kUnits);
    if (e == cudaSuccess && WbT)
      e = make_map(&m->wt[l], WbT + L.w_off[l], L.nout[l], L.nin[l], L.nout[l], L.total, members,
                   kUnits);
  }
  return e;
}

}  // namespace

cudaError_t allow_network_smem() {
  cudaError_t e = allow_smem(chain_kernel<true>, chain_smem_bytes(256));
  if (e == cudaSuccess) e = allow_smem(chain_kernel<false>, chain_smem_bytes(256));
  if (e == cudaSuccess) e = allow_smem(forward_kernel, fwd_smem_bytes(256, kFwdRing));
  if (e == cudaSuccess) e = allow_smem(pair_kernel, pair_smem_bytes(256));
  if (e == cudaSuccess) e = allow_smem(update_kernel, kUpdateSmem);
  return e;
}

cudaError_t launch_forward(const float* x, int n, const Xform& xf, const float* p, const bf16* Wb,
                           const Layout& L, int members, float* Y, unsigned* status,
                           cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const dim3 grid(blocks(n, BM), members);
  if ((long long)grid.x * grid.y * chain_ctas(L.nout[0]) <= 152) {
    // few tiles: a cluster per tile splits the layers (up to 384 queries of
    // five members of H = 256; a call of one query 49 us, 74 with a CTA per
    // tile).  Up to 152 CTAs: not all of the largest clusters run at once then,
    // but two waves of them still take no longer than a CTA per tile (queries
    // on the device, H = 256: three members 67 us up to 120 CTAs, 80 with 144,
    // 82 with a CTA per tile; one member 78 with 128 and 152 CTAs, 81; eight
    // members 80 with 128, 84)
    ChainMaps cm = {};
    cudaError_t e = chain_maps(&cm, L, members, Wb, nullptr);
    if (e != cudaSuccess) return e;
    ChainArgs c = {};
    c.rows = n;
    c.H = L.nout[0];
    c.x = x;
    c.xf = xf;
    c.Y = Y;
    c.p = p;
    c.P = L.total;
    for (int l = 0; l <= kHidden; l++) c.b_off[l] = (int)L.b_off[l];
    c.status = status;
    return launch_chain<false>(cm, c, members, s);
  }
  FwdMaps maps;
  FwdArgs a;
  a.x = x;
  a.n = n;
  a.H = L.nout[0];
  a.xf = xf;
  a.p = p;
  a.P = L.total;
  a.Y = Y;
  a.status = status;
  for (int l = 0; l <= kHidden; l++) {
    a.b_off[l] = (int)L.b_off[l];
    cudaError_t e = make_map(&maps.w[l], Wb + L.w_off[l], L.nin[l], L.nout[l], L.nin[l], L.total,
                             members, 128);
    if (e != cudaSuccess) return e;
  }
  if ((long long)grid.x * grid.y <= 152)  // at most one tile per SM
    forward_kernel<<<grid, kFwdThreads, fwd_smem_bytes(a.H, kFwdRing), s>>>(maps, a);
  else
    pair_kernel<<<dim3(blocks(n, 2 * BM), members), kPairThreads, pair_smem_bytes(a.H), s>>>(maps, a);
  return cudaGetLastError();
}

cudaError_t launch_train_step(const TrainArgs& t, cudaStream_t s) {
  const Layout& L = t.L;
  ChainMaps cm;
  cudaError_t e = chain_maps(&cm, L, t.members, t.Wb, t.WbT);
  if (e != cudaSuccess) return e;
  ChainArgs c = {};
  c.rows = t.rows;
  c.H = L.nout[0];
  c.X = t.X;
  c.T = t.T;
  c.n = t.n;
  c.direct = t.direct;
  c.seed = t.seed;
  c.d_step = t.d_step;
  c.w = t.w;
  c.p = t.p;
  c.P = L.total;
  c.Xt = t.Xt;
  c.dYt = t.dYt;
  c.dYft = t.dYft;
  c.loss = t.loss;
  c.status = t.status;
  UpdateMaps um;
  UpdateArgs u = {};
  u.rows = t.rows;
  u.grads_only = t.grads_only;
  u.L = L;
  u.p = t.p;
  u.g = t.g;
  u.m = t.m;
  u.v = t.v;
  u.Wb = t.Wb;
  u.WbT = t.WbT;
  u.dYft = t.dYft;
  u.lr = t.lr;
  u.beta1 = t.beta1;
  u.beta2 = t.beta2;
  u.eps = t.eps;
  u.d_step = t.d_step;
  u.d_sched = t.d_sched;
  u.status = t.status;
  const int H = c.H;
  for (int l = 0; l <= kHidden; l++) {
    c.b_off[l] = (int)L.b_off[l];
    if (l < kHidden) {
      c.Ht[l] = t.Ht[l];
      c.dZt[l] = t.dZt[l];
      u.dZt[l] = t.dZt[l];
    }
    u.first[l + 1] =
        u.first[l] + (int)blocks(L.nout[l], BM) * (int)blocks(L.nin[l], kUpdateBN);
    const bf16* A = l < kHidden ? t.dZt[l] : t.dYt;
    const bf16* B = l > 0 ? t.Ht[l - 1] : t.Xt;
    const int na = l < kHidden ? H : kOutPad, nb = l > 0 ? H : kInPad;
    e = make_map(&um.a[l], A, t.rows, na, t.rows, (long long)na * t.rows, t.members, BM);
    if (e == cudaSuccess)
      e = make_map(&um.b[l], B, t.rows, nb, t.rows, (long long)nb * t.rows, t.members, kUpdateBN);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(u.first[kHidden + 1], t.members);
  cfg.blockDim = dim3(kUpdateThreads);
  cfg.dynamicSmemBytes = kUpdateSmem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (int k = 0; k < t.steps; k++) {
    c.step_off = u.step_off = k;
    e = launch_chain<true>(cm, c, t.members, s);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, update_kernel, um, u);
    if (e != cudaSuccess) return e;
  }
  if (!t.grads_only && t.steps > 0) {
    advance_step_kernel<<<1, 1, 0, s>>>(t.d_step, t.steps);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

int train_loss_parts(int rows) { return 4 * (int)blocks(rows, BM); }

cudaError_t launch_answer(const GateArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  // few queries per block while that still leaves SMs idle (one up to three
  // blocks per SM, 8 up to 4096 queries), so that each query gets as many
  // warps as possible
  if (a.n <= 456)
    answer_kernel<1><<<a.n, kAnswerThreads, 0, s>>>(a);
  else if (a.n <= 4096)
    answer_kernel<8><<<blocks(a.n, 8), kAnswerThreads, 0, s>>>(a);
  else
    answer_kernel<64><<<blocks(a.n, 64), kAnswerThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace sg
