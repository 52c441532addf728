// BF16 GEMMs on the 5th-generation tensor cores (tcgen05) for the learned
// preconditioner's MLP, FP32 accumulation in tensor memory.
//
// gemm_tc_kernel:  C[m][n] = sum_k A[m][k] B[n][k]  (both operands
// K-contiguous, "TN") with fused epilogues.  Persistent and warp-specialised:
// one CTA per SM walks the 128 x 128 tiles of C (tile t, t + gridDim.x, ...;
// the N-tiles of a row block are neighbours, so A is read from HBM once):
//   * warp 0, lane 0 streams 128 x 64 tiles of A and B into a shared-memory
//     ring with TMA (128-byte swizzle, zero fill outside the tensor: ragged M
//     and K need no special case);
//   * warp 1, lane 0 issues tcgen05.mma (M = 128, N = 128, K = 16) from the
//     two shared-memory descriptors into one of two 128-column TMEM
//     accumulators, releases each stage with tcgen05.commit and signals the
//     finished accumulator;
//   * warps 2..17 drain the other accumulator meanwhile: a warp owns one
//     32 x 32 block of the tile (lane = row), applies the epilogue in
//     registers and moves its values between rows and coalesced global
//     accesses through 2 KB of shared memory.
// The kernel is bound by the epilogue's instructions (erff takes about 25 of
// the 45 per output of the GELU layers), not by the MMAs or by HBM: sixteen
// epilogue warps keep four per scheduler, and 128-wide tiles leave a shorter
// last wave than 256-wide ones (32768 rows: 1024 tiles over 152 SMs) and give
// a batch of 4096 rows 128 tiles instead of 64.
// 32768 rows: the whole forward 130 -> 94 us (GELU layers in 8 epilogue warps and
// 128 x 256 tiles, fp32 staging, and a copy of the output before).
//
// gemm_dw_kernel:  the three weight gradients dW[n][k] = sum_m dZ[m][n] H[m][k]
// in one launch, straight from the row-major activations: both operands are
// "MN-major" (contiguous along the output's rows and columns, the contraction
// runs down the rows), which tcgen05 reads as they lie, so nothing is
// transposed.  An output has only 28 tiles of 128 x 256 in all three layers
// together, so the contraction (the batch) is split over the CTAs; each
// writes its partial sums, and grad_reduce_kernel adds them in a fixed order.
// Loss and gradients of a batch of 4096: 596 -> 131 us against transposes,
// one GEMM per layer on 8 CTAs and column sums by one thread per column.
//
// Every mbarrier wait is bounded; a wait that runs out records an error code
// in *err, the CTA stops issuing work, drains what it issued (bounded) and
// frees its TMEM before returning.
// Requirements: K % 8 == 0, lda == ldb == K (row pitch 16-byte multiple),
// 16-byte aligned A and B, N % 32 == 0, ldc % 8 == 0, 16-byte aligned outputs.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace ax {
namespace mlp {

enum Epi {
  kEpiF32 = 0,    // Cf[m][n] = acc (+ bias[n])
  kEpiGelu = 1,   // z = acc + bias[n]; Cf[m][n] = z (when Cf is set); Hb[m][n] = bf16(gelu(z))
  kEpiDGelu = 2,  // Hb[m][n] = bf16(acc * gelu'(Zin[m][n])); column sums of Hb
  kEpiLoss = 3    // d = acc + bias[n] - Zin[m][n]; Hb[m][n] = bf16(d * scale); sums of d^2; column sums of Hb
};

struct GemmOut {
  float *Cf = nullptr;           // kEpiF32 output / kEpiGelu pre-activation
  __nv_bfloat16 *Hb = nullptr;   // bf16 output
  const float *Zin = nullptr;    // kEpiDGelu: pre-activation, kEpiLoss: target, of the output's shape
  const float *bias = nullptr;
  float *colsum = nullptr;       // [ceil(M / 32)][ldc]: sums of Hb over 32 rows (rows in order)
  float *sq = nullptr;           // kEpiLoss: [tiles][16] sums of d^2 per epilogue warp
  const double *skip = nullptr;  // when set and nonzero at launch, the GEMM does nothing
  float scale = 0.0f;
  int ldc = 0;
};

// gelu(z) = z Phi(z) with the normal CDF written through erf
__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * __expf(-0.5f * z * z);
}

}  // namespace mlp

namespace tc {

constexpr int kBM = 128, kBN = 128, kBK = 64, kStages = 5;
constexpr int kEpiWarps = 16, kThreads = 32 * (2 + kEpiWarps);
constexpr int kABytes = kBM * kBK * 2, kBBytes = kBN * kBK * 2, kStageBytes = kABytes + kBBytes;
constexpr int kTmemCols = 2 * kBN;  // two accumulators
// epilogue staging: 32 rows of 64 bytes per warp, their 16-byte chunks
// XOR-swizzled by ((row / 2) % 4): conflict-free row and row-segment accesses
constexpr int kStageTile = 32 * 64;
constexpr int kNumBars = 2 * kStages + 4;  // full[s], empty[s], tmem_full[2], tmem_empty[2]
// ring, epilogue staging, mbarriers, TMEM address slot; 1 KB for alignment
constexpr int kSmemBytes = kStages * kStageBytes + kEpiWarps * kStageTile + 8 * kNumBars + 16 + 1024;
constexpr long long kWaitCycles = 1ll << 32;  // SM clocks (about 2 s) before a wait gives up

enum TcError { kErrFull = 1, kErrEmpty = 2, kErrAccum = 3, kErrAccumFree = 4 };

// Instruction descriptor of tcgen05.mma kind::f16: D float32, A and B bf16,
// both K-major, N = 128, M = 128.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kBN >> 3) << 17) |
                            ((uint32_t)(kBM >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (SBO), descriptor version 1, base offset 0 (tiles are
// 1024-byte aligned).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// true once the phase with the given parity has completed; false after kWaitCycles
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  for (uint32_t it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 63u) == 63u && clock64() - t0 > kWaitCycles) return false;
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(kIdesc), "r"(accumulate));
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}

// 32 consecutive float32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float v[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int q = 0; q < 32; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void record_error(int *err, int code) {
  if (err) atomicCAS(err, 0, code);
}

// A warp's 32 rows of 64 bytes in shared memory, 16-byte chunk c of row r at
// chunk c ^ ((r / 2) % 4).  Rows are a lane's own values; the coalesced side
// serves four lanes per row, eight rows at a time.
__device__ __forceinline__ uint4 *stage_at(uint4 *tile, int row, int chunk) {
  return tile + row * 4 + (chunk ^ ((row >> 1) & 3));
}
// this lane's row (64 bytes) -> rows [m0, m0 + 32) of a row-major matrix, at
// byte column `col` of each; rows from M on are left out
__device__ __forceinline__ void rows_out(uint4 *tile, int lane, const uint4 v[4], char *base, size_t pitch, int m0,
                                         int M) {
#pragma unroll
  for (int c = 0; c < 4; ++c) *stage_at(tile, lane, c) = v[c];
  __syncwarp();
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = 8 * r + (lane >> 2);
    const uint4 x = *stage_at(tile, row, lane & 3);
    if (m0 + row < M) *reinterpret_cast<uint4 *>(base + (size_t)(m0 + row) * pitch + 16 * (lane & 3)) = x;
  }
  __syncwarp();
}
// the reverse: this lane's row (64 bytes); rows from M on read as zero
__device__ __forceinline__ void rows_in(uint4 *tile, int lane, uint4 v[4], const char *base, size_t pitch, int m0,
                                        int M) {
  uint4 x[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = 8 * r + (lane >> 2);
    x[r] = make_uint4(0u, 0u, 0u, 0u);
    if (m0 + row < M)
      x[r] = *reinterpret_cast<const uint4 *>(base + (size_t)(m0 + row) * pitch + 16 * (lane & 3));
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) *stage_at(tile, 8 * r + (lane >> 2), lane & 3) = x[r];
  __syncwarp();
#pragma unroll
  for (int c = 0; c < 4; ++c) v[c] = *stage_at(tile, lane, c);
  __syncwarp();
}
__device__ __forceinline__ void f32_out(uint4 *tile, int lane, const float v[32], float *C, int nc, int ldc, int m0,
                                        int M) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint4 u[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      u[c] = make_uint4(__float_as_uint(v[16 * h + 4 * c]), __float_as_uint(v[16 * h + 4 * c + 1]),
                        __float_as_uint(v[16 * h + 4 * c + 2]), __float_as_uint(v[16 * h + 4 * c + 3]));
    rows_out(tile, lane, u, reinterpret_cast<char *>(C + nc + 16 * h), (size_t)ldc * 4, m0, M);
  }
}
__device__ __forceinline__ uint32_t bf16x2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&h);
}
// 16 values of this lane's row of a float matrix (columns nc .. nc + 15)
__device__ __forceinline__ void f32_in(uint4 *tile, int lane, float v[16], const float *C, int nc, int ldc, int m0,
                                       int M) {
  uint4 u[4];
  rows_in(tile, lane, u, reinterpret_cast<const char *>(C + nc), (size_t)ldc * 4, m0, M);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    v[4 * c] = __uint_as_float(u[c].x);
    v[4 * c + 1] = __uint_as_float(u[c].y);
    v[4 * c + 2] = __uint_as_float(u[c].z);
    v[4 * c + 3] = __uint_as_float(u[c].w);
  }
}
// column sums of the warp's 32 x 32 block of bf16 values (lane's row in h),
// rows from M on left out; lane n returns column n, summed in row order
__device__ __forceinline__ float colsum32(uint4 *tile, int lane, const uint4 h[4], int rows) {
#pragma unroll
  for (int c = 0; c < 4; ++c) *stage_at(tile, lane, c) = h[c];
  __syncwarp();
  float s = 0.0f;
  const __nv_bfloat16 *t = reinterpret_cast<const __nv_bfloat16 *>(tile);
#pragma unroll 8
  for (int r = 0; r < rows; ++r)
    s += __bfloat162float(t[r * 32 + 8 * ((lane >> 3) ^ ((r >> 1) & 3)) + (lane & 7)]);
  __syncwarp();
  return s;
}

// Programmatic dependent launch: the CTAs of the next kernel of the stream may
// start (set up barriers and tensor memory) where this one's have left, and
// wait there until it has finished.  Every kernel of the chain waits, so each is
// ordered after all before it.  The tail of a GEMM and the setup of the next
// took about 2 us at each of a chain's boundaries: forward of 4096 rows 40.7 ->
// 34.4 us, of 32768 94.4 -> 89.6, loss and gradients of 4096 rows 131 -> 115.
// (Two groups of eight epilogue warps on alternating tiles, so that one computes
// while the other loads or stores: 94.4 -> 107, taken back.)
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... K, typename... A>
cudaError_t launch_after(void (*kernel)(K...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, K(args)...);
}

template <int EPI>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N,
                   int K, mlp::GemmOut out, int *err) {
  launch_next();
  if (out.skip) {
    wait_previous();
    if (*out.skip != 0.0) return;
  }
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // 1024-byte aligned ring (128-byte swizzle atoms)
  uint8_t *gbase = smem_raw + (base - raw);
  const uint32_t sA = base, sB = base + kStages * kABytes;
  uint4 *stage_tiles = reinterpret_cast<uint4 *>(gbase + kStages * kStageBytes);
  const uint32_t bars = base + kStages * kStageBytes + kEpiWarps * kStageTile;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(gbase + kStages * kStageBytes + kEpiWarps * kStageTile +
                                                     8 * kNumBars);
  __shared__ int abort_flag;
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (kStages + s); };
  auto acc_full = [&](int b) { return bars + 8u * (2 * kStages + b); };
  auto acc_free = [&](int b) { return bars + 8u * (2 * kStages + 2 + b); };

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nk = (K + kBK - 1) / kBK;
  const int ntn = (N + kBN - 1) / kBN, ntiles = ((M + kBM - 1) / kBM) * ntn;

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_free(b), kEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  wait_previous();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // producer: one k-block of A and B per stage, across all tiles of this CTA
      asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&ta) : "memory");
      asm volatile("prefetch.tensormap [%0];\n" ::"l"((uint64_t)&tb) : "memory");
      int g = 0;  // k-blocks issued
      for (int t = blockIdx.x; t < ntiles && !*(volatile int *)&abort_flag; t += gridDim.x) {
        const int m0 = (t / ntn) * kBM, n0 = (t % ntn) * kBN;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % kStages, round = g / kStages;
          if (round > 0 && !mbar_wait(empty(s), (uint32_t)((round - 1) & 1))) {
            record_error(err, kErrEmpty);
            atomicExch(&abort_flag, 1);
            break;
          }
          mbar_expect_tx(full(s), (uint32_t)kStageBytes);
          tma_load_2d(sA + s * kABytes, &ta, kb * kBK, m0, full(s));
          tma_load_2d(sB + s * kBBytes, &tb, kb * kBK, n0, full(s));
        }
      }
      // drain: the copies of the last stages issued have landed before teardown
      for (int q = (g > kStages ? g - kStages : 0); q < g; ++q)
        if (!mbar_wait(full(q % kStages), (uint32_t)((q / kStages) & 1))) record_error(err, kErrFull);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer
      int g = 0, i = 0;  // k-blocks consumed, tiles accumulated
      for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
        const int b = i & 1, use = i >> 1;
        if (use > 0 && !mbar_wait(acc_free(b), (uint32_t)((use - 1) & 1))) {
          record_error(err, kErrAccumFree);
          atomicExch(&abort_flag, 1);
        }
        if (*(volatile int *)&abort_flag) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t d = tmem + (uint32_t)(b * kBN);
        bool ok = true;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % kStages;
          if (!mbar_wait(full(s), (uint32_t)((g / kStages) & 1))) {
            record_error(err, kErrFull);
            atomicExch(&abort_flag, 1);
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
          for (int kk = 0; kk < kBK / 16; ++kk) {
            const uint64_t ad = sw128_desc(sA + s * kABytes + kk * 32);
            const uint64_t bd = sw128_desc(sB + s * kBBytes + kk * 32);
            umma_bf16(d, ad, bd, (kb | kk) != 0 ? 1u : 0u);
          }
          umma_commit(empty(s));
        }
        umma_commit(acc_full(b));  // arrives when every MMA issued so far has completed
        if (!ok) break;
      }
    }
  } else {
    // epilogue warps: lane quarter q = warp % 4 (TMEM lanes = tile rows), 32 columns at 32 h
    const int ew = warp - 2, q = warp & 3, h = ew >> 2;
    uint4 *tile = stage_tiles + ew * (kStageTile / 16);
    int i = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
      const int b = i & 1, use = i >> 1;
      const bool ok = mbar_wait(acc_full(b), (uint32_t)(use & 1));
      if (!ok) record_error(err, kErrAccum);
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (!__all_sync(0xffffffffu, ok && !*(volatile int *)&abort_flag)) break;
      const int m0 = (t / ntn) * kBM, n0 = (t % ntn) * kBN;
      const int mw = m0 + 32 * q;  // first row of this warp's 32-row block
      const int nc = n0 + 32 * h;
      if (nc < N) {  // N % 32 == 0: whole 32-column blocks
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * kBN + 32 * h), v);
        if constexpr (EPI != mlp::kEpiDGelu) {
          if (out.bias) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
              const float4 bv = *reinterpret_cast<const float4 *>(out.bias + nc + 4 * c);
              v[4 * c] += bv.x;
              v[4 * c + 1] += bv.y;
              v[4 * c + 2] += bv.z;
              v[4 * c + 3] += bv.w;
            }
          }
        }
        if constexpr (EPI == mlp::kEpiF32) {
          f32_out(tile, lane, v, out.Cf, nc, out.ldc, mw, M);
        } else {
          if constexpr (EPI == mlp::kEpiGelu) {
            if (out.Cf) f32_out(tile, lane, v, out.Cf, nc, out.ldc, mw, M);
#pragma unroll
            for (int c = 0; c < 32; ++c) v[c] = mlp::gelu_f(v[c]);
          } else {
            float sq = 0.0f;
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              float zin[16];
              f32_in(tile, lane, zin, out.Zin, nc + 16 * g, out.ldc, mw, M);
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                if constexpr (EPI == mlp::kEpiDGelu) {
                  v[16 * g + c] *= mlp::gelu_grad_f(zin[c]);
                } else {
                  const float d = v[16 * g + c] - zin[c];
                  sq = fmaf(d, d, sq);
                  v[16 * g + c] = d * out.scale;
                }
              }
            }
            if constexpr (EPI == mlp::kEpiLoss) {
              if (mw + lane >= M) sq = 0.0f;
              for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
              if (lane == 0) out.sq[(size_t)t * kEpiWarps + ew] = sq;
            }
          }
          uint4 hb[4];
#pragma unroll
          for (int c = 0; c < 4; ++c)
            hb[c] = make_uint4(bf16x2(v[8 * c], v[8 * c + 1]), bf16x2(v[8 * c + 2], v[8 * c + 3]),
                               bf16x2(v[8 * c + 4], v[8 * c + 5]), bf16x2(v[8 * c + 6], v[8 * c + 7]));
          rows_out(tile, lane, hb, reinterpret_cast<char *>(out.Hb + nc), (size_t)out.ldc * 2, mw, M);
          if constexpr (EPI == mlp::kEpiDGelu || EPI == mlp::kEpiLoss) {
            const int rows = M - mw < 32 ? M - mw : 32;
            if (rows > 0) {
              const float s = colsum32(tile, lane, hb, rows);
              out.colsum[(size_t)(mw / 32) * out.ldc + nc + lane] = s;
            }
          }
        }
      } else if constexpr (EPI == mlp::kEpiLoss) {
        if (lane == 0) out.sq[(size_t)t * kEpiWarps + ew] = 0.0f;
      }
      // this warp's reads of buffer b are complete: hand it back to the MMA warp
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(acc_free(b)) : "memory");
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// ---------------------------------------------------------------------------
// weight gradients:  P[s][n][k] = sum over the batch rows of split s of
// dZ[m][n] H[m][k], three problems in one launch
// ---------------------------------------------------------------------------
constexpr int kDwBN = 256, kDwStages = 4, kDwEpiWarps = 8, kDwThreads = 32 * (2 + kDwEpiWarps);
constexpr int kDwBox = kBK * 64 * 2;  // one TMA box: 64 batch rows of 64 columns
constexpr int kDwABytes = (kBM / 64) * kDwBox, kDwBBytes = (kDwBN / 64) * kDwBox;
constexpr int kDwStageBytes = kDwABytes + kDwBBytes;
constexpr int kDwNumBars = 2 * kDwStages + 1;
constexpr int kDwSmemBytes = kDwStages * kDwStageBytes + kDwEpiWarps * kStageTile + 8 * kDwNumBars + 16 + 1024;
// D float32, A and B bf16, both MN-major (bits 15, 16), N = 256, M = 128
constexpr uint32_t kDwIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                              ((uint32_t)(kDwBN >> 3) << 17) | ((uint32_t)(kBM >> 4) << 24);

// Shared-memory matrix descriptor: MN-major, 128-byte swizzle.  A TMA box is
// 64 rows (contraction) of 128 bytes (64 columns): groups of 8 contraction
// rows are 1024 bytes apart (SBO), the next 64 columns one box away (LBO).
__device__ __forceinline__ uint64_t mn128_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(kDwBox >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void umma_bf16_mn(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(kDwIdesc), "r"(accumulate));
}

struct DwArgs {
  CUtensorMap a[3], b[3];  // dZ [M][n], H [M][k] of each layer
  int n[3], k[3];          // rows and columns of dW
  int64_t off[3];          // its place in the parameter vector
  int first[4];            // first tile of each layer, total
  int M, splits;
  int64_t np;              // parameters: pitch of the partial sums
  float *part;             // [splits][np]
};

// CTA (tile, split): 128 x 256 of one dW over its share of the batch's
// 64-row blocks.  Warp 0 loads, warp 1 multiplies, warps 2..9 drain.
__global__ void __launch_bounds__(kDwThreads, 1) gemm_dw_kernel(const __grid_constant__ DwArgs g, int *err) {
  launch_next();
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t *gbase = smem_raw + (base - raw);
  const uint32_t sA = base, sB = base + kDwStages * kDwABytes;
  uint4 *stage_tiles = reinterpret_cast<uint4 *>(gbase + kDwStages * kDwStageBytes);
  const uint32_t bars = base + kDwStages * kDwStageBytes + kDwEpiWarps * kStageTile;
  uint32_t *tmem_slot =
      reinterpret_cast<uint32_t *>(gbase + kDwStages * kDwStageBytes + kDwEpiWarps * kStageTile + 8 * kDwNumBars);
  auto full = [&](int s) { return bars + 8u * s; };
  auto empty = [&](int s) { return bars + 8u * (kDwStages + s); };
  const uint32_t acc_full = bars + 8u * (2 * kDwStages);
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tile = blockIdx.x / g.splits, split = blockIdx.x % g.splits;
  const int p = tile < g.first[1] ? 0 : tile < g.first[2] ? 1 : 2;
  const int ntn = (g.k[p] + kDwBN - 1) / kDwBN, lt = tile - g.first[p];
  const int m0 = (lt / ntn) * kBM, n0 = (lt % ntn) * kDwBN;
  // this split's 64-row blocks of the batch (at least one: splits <= blocks)
  const int nkb = (g.M + kBK - 1) / kBK;
  const int kb0 = (int)((int64_t)nkb * split / g.splits), kb1 = (int)((int64_t)nkb * (split + 1) / g.splits);

  if (tid == 0) {
    abort_flag = 0;
    for (int s = 0; s < kDwStages; ++s) {
      mbar_init(full(s), 1);
      mbar_init(empty(s), 1);
    }
    mbar_init(acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                 "r"(kDwBN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  wait_previous();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      int c = 0;  // blocks issued
      for (int kb = kb0; kb < kb1; ++kb, ++c) {
        const int s = c % kDwStages, round = c / kDwStages;
        if (round > 0 && !mbar_wait(empty(s), (uint32_t)((round - 1) & 1))) {
          record_error(err, kErrEmpty);
          atomicExch(&abort_flag, 1);
          break;
        }
        mbar_expect_tx(full(s), (uint32_t)kDwStageBytes);
#pragma unroll
        for (int q = 0; q < kBM / 64; ++q)
          tma_load_2d(sA + s * kDwABytes + q * kDwBox, &g.a[p], m0 + 64 * q, kb * kBK, full(s));
#pragma unroll
        for (int q = 0; q < kDwBN / 64; ++q)
          tma_load_2d(sB + s * kDwBBytes + q * kDwBox, &g.b[p], n0 + 64 * q, kb * kBK, full(s));
      }
      // drain: the copies of the last stages issued have landed before teardown
      for (int q = (c > kDwStages ? c - kDwStages : 0); q < c; ++q)
        if (!mbar_wait(full(q % kDwStages), (uint32_t)((q / kDwStages) & 1))) record_error(err, kErrFull);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int c = 0;
      for (int kb = kb0; kb < kb1; ++kb, ++c) {
        const int s = c % kDwStages;
        if (*(volatile int *)&abort_flag) break;
        if (!mbar_wait(full(s), (uint32_t)((c / kDwStages) & 1))) {
          record_error(err, kErrFull);
          atomicExch(&abort_flag, 1);
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
        for (int kk = 0; kk < kBK / 16; ++kk)  // 16 contraction rows: two 8-row groups
          umma_bf16_mn(tmem, mn128_desc(sA + s * kDwABytes + kk * 2048), mn128_desc(sB + s * kDwBBytes + kk * 2048),
                       (c | kk) != 0 ? 1u : 0u);
        umma_commit(empty(s));
      }
      umma_commit(acc_full);  // arrives when every MMA issued has completed
    }
  } else {
    // rows 32 (warp % 4), columns 128 h .. of the tile
    const int ew = warp - 2, q = warp & 3, h = ew >> 2;
    uint4 *st = stage_tiles + ew * (kStageTile / 16);
    const bool ok = mbar_wait(acc_full, 0);
    if (!ok) record_error(err, kErrAccum);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (__all_sync(0xffffffffu, ok && !*(volatile int *)&abort_flag)) {
      float *C = g.part + (size_t)split * g.np + g.off[p];
#pragma unroll 1
      for (int c = 0; c < kDwBN / 64; ++c) {
        const int col = kDwBN / 2 * h + 32 * c;
        if (n0 + col >= g.k[p]) break;  // k % 32 == 0
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)col, v);
        f32_out(st, lane, v, C, n0 + col, g.k[p], m0 + 32 * q, g.n[p]);
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kDwBN) : "memory");
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// 2-D bf16 tensor [rows][K] (K contiguous), boxes of kBK x box_rows, 128-byte swizzle, zero fill outside
inline bool make_map(CUtensorMap *map, const void *ptr, int rows, int K, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kBK, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// the same tensor for the MN-major operands of gemm_dw_kernel: [rows][cols], boxes of 64 columns x 64 rows
inline bool make_map_mn(CUtensorMap *map, const void *ptr, int rows, int cols) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  const cuuint32_t box[2] = {64, (cuuint32_t)kBK};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline int sm_count() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms < 1) sms = 1;
  }
  return sms;
}

// once per process and device, outside any stream capture
inline cudaError_t gemm_init() {
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<mlp::kEpiF32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<mlp::kEpiGelu>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<mlp::kEpiDGelu>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_tc_kernel<mlp::kEpiLoss>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gemm_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDwSmemBytes);
  if (e == cudaSuccess && !encode_fn()) e = cudaErrorNotSupported;
  return e;
}

inline int gemm_tiles(int M, int N) { return ((M + kBM - 1) / kBM) * ((N + kBN - 1) / kBN); }

// C = A B^T with A [M][K], B [N][K] bf16 (row pitch K), epilogue EPI.
template <int EPI>
inline cudaError_t gemm(int M, int N, int K, const __nv_bfloat16 *A, const __nv_bfloat16 *B,
                        const mlp::GemmOut &out, int *err, cudaStream_t s) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K <= 0 || K % 8 || N % 32 || out.ldc % 8 || ((uintptr_t)A & 15) || ((uintptr_t)B & 15) ||
      ((uintptr_t)out.Cf & 15) || ((uintptr_t)out.Hb & 15) || ((uintptr_t)out.Zin & 15) || ((uintptr_t)out.bias & 15))
    return cudaErrorInvalidValue;
  CUtensorMap ta, tb;
  if (!make_map(&ta, A, M, K, kBM) || !make_map(&tb, B, N, K, kBN)) return cudaErrorInvalidValue;
  const int ntiles = gemm_tiles(M, N), sms = sm_count();
  const int grid = ntiles < sms ? ntiles : sms;
  return launch_after(gemm_tc_kernel<EPI>, grid, kThreads, kSmemBytes, s, ta, tb, M, N, K, out, err);
}

// Tiles of the three weight gradients and the splits of the batch: as many
// as fill the SMs once, one 64-row block each at least.
inline int dw_splits(int tiles, int M) {
  const int nkb = (M + kBK - 1) / kBK, s = sm_count() / tiles;
  return s < 1 ? 1 : (s < nkb ? s : nkb);
}
inline cudaError_t gemm_dw(const DwArgs &g, int *err, cudaStream_t s) {
  return launch_after(gemm_dw_kernel, g.first[3] * g.splits, kDwThreads, kDwSmemBytes, s, g, err);
}

}  // namespace tc
}  // namespace ax
