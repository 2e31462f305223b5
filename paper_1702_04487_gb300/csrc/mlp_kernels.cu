// Kernels of the surrogate network: a BF16 tensor-core GEMM on the 5th
// generation tensor cores (tcgen05.mma, accumulator in tensor memory) with
// fused epilogues, and the small element-wise kernels around it (input
// transform and minibatch gather, loss, bias gradients, Adam, output
// transform, acceptance gate).
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

template <int BN>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                const GemmArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr int kA = BM * BK * 2;
  constexpr int kStage = stage_bytes<BN>();
  constexpr uint32_t kCols = tmem_cols<BN>();
  constexpr uint32_t kIdesc = idesc_bf16(BM, BN);
  // bars[b]: the load of buffer b landed; bars[kStages + b]: its MMAs done
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int z = blockIdx.z;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int za = a.sA ? z : 0, zb = a.sB ? z : 0;  // a zero stride shares one operand

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

  const int nk = (a.K + BK - 1) / BK;
  bool ok = true;
  if (tid == 0) {
    // slice kt lives in buffer kt % kStages; its load completes phase
    // (kt / kStages) & 1 of bars[buffer], its MMAs the same phase of
    // bars[kStages + buffer]
    auto load = [&](int kt) {
      const int b = kt % kStages;
      const uint32_t ta = smem_u32(smem + b * kStage), tb = ta + kA;
      mbar_expect_tx(smem_u32(&bars[b]), (uint32_t)kStage);
      tma_load3(ta, &tmA, kt * BK, m0, za, smem_u32(&bars[b]));
      tma_load3(tb, &tmB, kt * BK, n0, zb, smem_u32(&bars[b]));
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
  }
  ok = __syncthreads_and(ok);
  tc_fence_after();

  if (ok) {
    // Epilogue through shared memory (the operand buffers are free once every
    // MMA is done): each warp takes its 32 rows x 16 columns from tensor
    // memory (lane = row), then works row by row -- half-warps on two rows,
    // lanes along n -- so that bias, aux and every row-major output are read
    // and written in contiguous runs; the transposed BF16 copy is written
    // from the lane = row layout, contiguous along m.
    float* T = reinterpret_cast<float*>(smem) + warp * (32 * 17);
    const int m = m0 + warp * 32 + lane;
    const bool mrow = m < a.M;
    const float* bias = a.bias ? a.bias + z * a.sBias : nullptr;
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
        if (mm >= a.M || n >= a.N) continue;
        float x = T[r * 17 + jj];
        if (a.epi == EPI_F32) {
          a.Cf[z * a.sCf + (size_t)mm * a.ldcf + n] = x;
          continue;
        }
        if (a.epi == EPI_BIAS_F32) {
          a.Cf[z * a.sCf + (size_t)mm * a.ldcf + n] = x + bias[n];
          continue;
        }
        if (a.epi == EPI_BIAS_GELU) {
          x += bias[n];
          if (a.Zout) a.Zout[z * a.sZ + (size_t)mm * a.ldz + n] = x;
          x = gelu_f(x);
        } else {  // EPI_GELU_BWD
          x *= gelu_grad_f(a.aux[z * a.sAux + (size_t)mm * a.ldaux + n]);
        }
        const bf16 hb = __float2bfloat16_rn(x);
        if (a.Cb) a.Cb[z * a.sCb + (size_t)mm * a.ldcb + n] = hb;
        T[r * 17 + jj] = __bfloat162float(hb);  // for the transposed copy
      }
      __syncwarp();
      if (a.Ct && mrow && (a.epi == EPI_BIAS_GELU || a.epi == EPI_GELU_BWD)) {
#pragma unroll
        for (int j = 0; j < 16; j++)
          if (nb + j < a.N)
            a.Ct[z * a.sCt + (size_t)(nb + j) * a.ldct + m] = __float2bfloat16_rn(T[lane * 17 + j]);
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
  static EncodeTiledFn fn = nullptr;
  static bool looked = false;
  if (!looked) {
    looked = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
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
cudaError_t launch_bn(const GemmArgs& a, int members, cudaStream_t s) {
  const size_t smem = gemm_smem_bytes(BN);
  CUtensorMap ma, mb;
  cudaError_t e0 = make_map(&ma, a.A, a.K, a.M, a.lda, a.sA, a.sA ? members : 1, BM);
  if (e0 == cudaSuccess) e0 = make_map(&mb, a.B, a.K, a.N, a.ldb, a.sB, a.sB ? members : 1, BN);
  if (e0 != cudaSuccess) return e0;
  static bool attr = false;
  if (!attr) {
    cudaError_t e =
        cudaFuncSetAttribute(gemm_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  dim3 grid((a.M + BM - 1) / BM, (a.N + BN - 1) / BN, members);
  gemm_kernel<BN><<<grid, kThreads, smem, s>>>(ma, mb, a);
  return cudaGetLastError();
}

}  // namespace

size_t gemm_smem_bytes(int bn) {
  return 1024 + kStages * (size_t)(BM * BK * 2 + bn * BK * 2) + 16 * kStages + 16;
}

cudaError_t launch_gemm(const GemmArgs& a, int members, cudaStream_t s) {
  // the narrowest tile that covers N, halved (down to 32 columns) while the
  // grid has fewer than ~2 tiles per SM of a 152-SM part
  int bn = a.N <= 16 ? 16 : a.N <= 32 ? 32 : a.N <= 64 ? 64 : a.N <= 128 ? 128 : 256;
  const long long mt = (a.M + BM - 1) / BM;
  while (bn > 32 && mt * ((a.N + bn - 1) / bn) * members < 304) bn /= 2;
  switch (bn) {
    case 16: return launch_bn<16>(a, members, s);
    case 32: return launch_bn<32>(a, members, s);
    case 64: return launch_bn<64>(a, members, s);
    case 128: return launch_bn<128>(a, members, s);
    default: return launch_bn<256>(a, members, s);
  }
}

}  // namespace sg

// ---------------------------------------------------------------------------
// Element-wise kernels around the GEMMs.
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

__global__ void gather_kernel(const bf16* __restrict__ X, const float* __restrict__ T, int n,
                              int bm, unsigned long long seed, const long long* __restrict__ d_step,
                              bf16* __restrict__ Xb, bf16* __restrict__ Xbt,
                              float* __restrict__ Tb) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, mem = blockIdx.y;
  if (r >= bm) return;
  const unsigned long long ctr =
      ((unsigned long long)mem << 56) ^ ((unsigned long long)*d_step << 24) ^ (unsigned)r;
  const int src = (int)(mix64(seed ^ mix64(ctr)) % (unsigned long long)n);
  const size_t ob = (size_t)mem * bm;
#pragma unroll
  for (int d = 0; d < kInPad; d++) {
    const bf16 v = X[(size_t)src * kInPad + d];
    Xb[(ob + r) * kInPad + d] = v;
    Xbt[(size_t)mem * kInPad * bm + (size_t)d * bm + r] = v;
  }
#pragma unroll
  for (int d = 0; d < kOut; d++) Tb[(ob + r) * kOut + d] = T[(size_t)src * kOut + d];
}

__global__ void loss_kernel(const float* __restrict__ Y, const float* __restrict__ Tb,
                            const float* __restrict__ w, int bm, bf16* __restrict__ dY,
                            bf16* __restrict__ dYt, float* __restrict__ dYft, double* loss,
                            unsigned* status) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x, mem = blockIdx.y;
  double acc = 0.0;
  if (r < bm) {
    const size_t row = (size_t)mem * bm + r;
    const float inv = 2.0f / (float)(bm * kOut);
#pragma unroll
    for (int d = 0; d < kOutPad; d++) {
      float g = 0.0f;
      if (d < kOut) {
        const float diff = Y[row * kOutPad + d] - Tb[row * kOut + d];
        acc += (double)w[d] * diff * diff;
        g = inv * w[d] * diff;
      }
      const bf16 gb = __float2bfloat16_rn(g);
      dY[row * kOutPad + d] = gb;
      dYt[(size_t)mem * kOutPad * bm + (size_t)d * bm + r] = gb;
      dYft[(size_t)mem * kOutPad * bm + (size_t)d * bm + r] = g;
    }
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(loss + mem, acc / (double)(bm * kOut));
    if (!isfinite(acc)) atomicOr(status, kStatusNonFinite);
  }
}

template <typename T>
__device__ __forceinline__ float to_f(T v);
template <>
__device__ __forceinline__ float to_f<float>(float v) {
  return v;
}
template <>
__device__ __forceinline__ float to_f<bf16>(bf16 v) {
  return __bfloat162float(v);
}

// one warp per (member, row)
template <typename T>
__global__ void rowsum_kernel(const T* __restrict__ in, int rows, int cols, int ld, long long sin_,
                              float* __restrict__ out, long long sout) {
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int mem = blockIdx.y;
  if (row >= rows) return;
  const T* p = in + mem * sin_ + (size_t)row * ld;
  float acc = 0.0f;
  for (int c = lane; c < cols; c += 32) acc += to_f<T>(p[c]);
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
  if (lane == 0) out[mem * sout + row] = acc;
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

// d_sched (may be null): {first step, number of steps} of the current
// training call; lr then decays along a half cosine, lr (1 + cos(pi s / S)) / 2
// at its step s of S.
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, const Layout L, int members, float lr,
                            float beta1, float beta2, float eps, const long long* __restrict__ d_step,
                            const long long* __restrict__ d_sched, bf16* __restrict__ Wb,
                            bf16* __restrict__ WbT) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= L.total * members) return;
  if (d_sched && d_sched[1] > 0) {
    const float frac = (float)(*d_step - d_sched[0]) / (float)d_sched[1];
    lr *= 0.5f * (1.0f + cospif(fminf(fmaxf(frac, 0.0f), 1.0f)));
  }
  const float t = (float)(*d_step + 1);
  const float bc1 = 1.0f - powf(beta1, t), bc2 = 1.0f - powf(beta2, t);
  const float gi = g[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * gi;
  const float vi = beta2 * v[i] + (1.0f - beta2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  p[i] = pi;
  const long long mem = i / L.total, k = i % L.total;
  int l, r, c;
  bool weight;
  locate(L, k, l, r, c, weight);
  if (weight) {
    const bf16 b = __float2bfloat16_rn(pi);
    Wb[i] = b;
    WbT[mem * L.total + L.w_off[l] + (long long)c * L.nout[l] + r] = b;
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

__global__ void advance_step_kernel(long long* d_step) { *d_step += 1; }

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
// Bound by the GELUs (an erff each: 4 H per query and member) at instruction
// issue; two CTAs of 256 threads share an SM, so one's tensor-core pass and
// weight loads run beside the other's GELUs.  While the grid has at most one
// tile per SM, one CTA of 512 threads and a ring of nine chunks per SM halve
// the serial chain of a layer instead.  Measured, five members of H = 256:
// 65536 queries 500 us, against 2190 us for a GEMM launch per layer with the
// activations through HBM (the same results, bit for bit).
constexpr int kFwdChunk = 128 * BK * 2;  // bytes of a weight chunk, and of 64 activation columns
constexpr int kFwdRingMax = 9;

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

template <int NT>
__host__ __device__ constexpr int fwd_ring() {
  return NT == 256 ? 3 : kFwdRingMax;
}
// activations, ring, then the barriers and the tensor-memory address (no
// static shared memory: the dynamic part then starts on a 1024-byte boundary
// and two CTAs of H = 256 fit an SM)
constexpr int kFwdTail = 256;
size_t fwd_smem_bytes(int H, int ring) {
  return (size_t)((H + BK - 1) / BK + ring) * kFwdChunk + kFwdTail;
}

template <int NT>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1)
    forward_kernel(const __grid_constant__ FwdMaps maps, const FwdArgs a) {
  extern __shared__ __align__(1024) uint8_t fwd_smem[];
  constexpr int R = fwd_ring<NT>();
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
  for (int k = tid; k < QB * kOut; k += kAnswerThreads) {
    const int q = q0 + (k >> 2), d = k & 3;
    const bool in = q < a.n;
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
    // QB * kOut is a multiple of 32: every lane of the warp is here
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

cudaError_t launch_gather(const bf16* X, const float* T, int n, int bm, int members,
                          unsigned long long seed, const long long* d_step, bf16* Xb, bf16* Xbt,
                          float* Tb, cudaStream_t s) {
  gather_kernel<<<dim3(blocks(bm, 128), members), 128, 0, s>>>(X, T, n, bm, seed, d_step, Xb, Xbt,
                                                                Tb);
  return cudaGetLastError();
}

cudaError_t launch_loss(const float* Y, const float* Tb, const float* w, int bm, int members,
                        bf16* dY, bf16* dYt, float* dYft, double* loss, unsigned* status,
                        cudaStream_t s) {
  loss_kernel<<<dim3(blocks(bm, 128), members), 128, 0, s>>>(Y, Tb, w, bm, dY, dYt, dYft, loss,
                                                              status);
  return cudaGetLastError();
}

cudaError_t launch_rowsum_bf16(const bf16* in, int rows, int cols, int ld, long long sin_,
                               float* out, long long sout, int members, cudaStream_t s) {
  rowsum_kernel<bf16><<<dim3(blocks(rows, 8), members), 256, 0, s>>>(in, rows, cols, ld, sin_, out,
                                                                     sout);
  return cudaGetLastError();
}

cudaError_t launch_rowsum_f32(const float* in, int rows, int cols, int ld, long long sin_,
                              float* out, long long sout, int members, cudaStream_t s) {
  rowsum_kernel<float><<<dim3(blocks(rows, 8), members), 256, 0, s>>>(in, rows, cols, ld, sin_, out,
                                                                      sout);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m, float* v, const Layout& L, int members,
                        float lr, float beta1, float beta2, float eps, const long long* d_step,
                        const long long* d_sched, bf16* Wb, bf16* WbT, cudaStream_t s) {
  adam_kernel<<<blocks(L.total * members, 256), 256, 0, s>>>(p, g, m, v, L, members, lr, beta1,
                                                              beta2, eps, d_step, d_sched, Wb, WbT);
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

cudaError_t launch_advance_step(long long* d_step, cudaStream_t s) {
  advance_step_kernel<<<1, 1, 0, s>>>(d_step);
  return cudaGetLastError();
}

cudaError_t launch_forward(const float* x, int n, const Xform& xf, const float* p, const bf16* Wb,
                           const Layout& L, int members, float* Y, unsigned* status,
                           cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
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
  static bool attr = false;
  if (!attr) {
    cudaError_t e = cudaFuncSetAttribute(forward_kernel<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)fwd_smem_bytes(256, fwd_ring<256>()));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(forward_kernel<512>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)fwd_smem_bytes(256, fwd_ring<512>()));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const dim3 grid(blocks(n, BM), members);
  if ((long long)grid.x * grid.y <= 152)  // at most one tile per SM
    forward_kernel<512><<<grid, 512, fwd_smem_bytes(a.H, fwd_ring<512>()), s>>>(maps, a);
  else
    forward_kernel<256><<<grid, 256, fwd_smem_bytes(a.H, fwd_ring<256>()), s>>>(maps, a);
  return cudaGetLastError();
}

cudaError_t launch_answer(const GateArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  // few queries per block while that still leaves SMs idle (8 per block up to
  // 4096 queries), so that each query gets as many warps as possible
  if (a.n <= 4096)
    answer_kernel<8><<<blocks(a.n, 8), kAnswerThreads, 0, s>>>(a);
  else
    answer_kernel<64><<<blocks(a.n, 64), kAnswerThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace sg
