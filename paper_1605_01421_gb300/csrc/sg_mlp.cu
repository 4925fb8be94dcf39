// sg_mlp.cu -- the dense contractions of the learned one-day emulator on the
// fifth-generation tensor cores (tcgen05, accumulators in tensor memory), and
// the small element-wise kernels around them (loss, optimiser, features,
// sampling).  The emulator is an extension of the method, not part of the
// paper.
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "sg_common.h"
#include "sg_device.cuh"
#include "sg_mlp.h"
#include "sg_tc.cuh"

using namespace sg;

namespace {

constexpr int kBM = 128;              // rows per tile (tensor-core M)
constexpr int kBK = 64;               // K per pipeline stage
constexpr uint32_t kWaitLimit = 1u << 24;  // mbarrier polls before giving up

// Byte offset of element (row, k) of a rows x 64 BF16 stage in the
// no-swizzle K-major core-matrix layout: 8-row x 8-element (16 byte) core
// matrices, the 8 core matrices of an 8-row group consecutive along K.
__device__ __forceinline__ uint32_t stage_off(int row, int kgroup) {
  return (uint32_t)(((row >> 3) * 8 + kgroup) * 128 + (row & 7) * 16);
}

// 16-byte asynchronous global-to-shared copy; src_bytes = 0 zero-fills.
__device__ __forceinline__ void cp_async16(uint32_t saddr, const void *gsrc, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr), "l"(gsrc),
               "r"(src_bytes)
               : "memory");
}

// GELU in its tanh form, 0.5 x (1 + tanh(sqrt(2 / pi) (x + 0.044715 x^3))),
// with the hardware tanh approximation (relative error ~2^-11, below the
// BF16 rounding of the activations).
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// s GELU(x), given hs = s / 2: h (1 + tanh(u)) with h = hs x and u = x
// (sqrt(2 / pi) + 0.044715 sqrt(2 / pi) x^2), in fused multiply-adds (s
// folds an output scale into the activation).
__device__ __forceinline__ float gelu_scaled(float x, float hs) {
  const float u = x * __fmaf_rn(0.0356774081f, x * x, 0.7978845608f);
  const float h = hs * x;
  return __fmaf_rn(h, tanh_fast(u), h);
}

// 2^x with the hardware approximation (the sampler's softmax weights).
__device__ __forceinline__ float ex2_fast(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kLog2e = 1.44269504088896341f;

// 16 E4M3 bytes of y[0..15] (nearest even, saturated), y[0] in the lowest.
__device__ __forceinline__ uint4 pack_e4m3_16(const float *y) {
  uint32_t packed[4];
#pragma unroll
  for (int j = 0; j < 16; j += 4) {
    const __nv_fp8x2_storage_t lo =
        __nv_cvt_float2_to_fp8x2(make_float2(y[j], y[j + 1]), __NV_SATFINITE, __NV_E4M3);
    const __nv_fp8x2_storage_t hi =
        __nv_cvt_float2_to_fp8x2(make_float2(y[j + 2], y[j + 3]), __NV_SATFINITE, __NV_E4M3);
    packed[j / 4] = (uint32_t)lo | ((uint32_t)hi << 16);
  }
  return make_uint4(packed[0], packed[1], packed[2], packed[3]);
}

// C = act(A . Bt^T + bias) for one 128 x BN tile.  A: M x K, Bt: N x K, both
// row-major BF16 with K contiguous (K % 8 == 0, rows 16-byte aligned).
// 256 threads: all load the double-buffered K stages into shared memory
// (cp.async, overlapping the previous stage's MMAs), thread 0 issues the MMAs
// (4 per stage, K = 16 each) and commits them to the stage's mbarrier; in the
// epilogue warp w reads TMEM lane quarter w % 4 (32 tile rows), columns of
// half w / 4 of the tile.
//
// F8: A and B are FP8 E4M3 bytes instead (K = 128 per stage, the same 128
// bytes per row; tcgen05.mma kind::f8f6f4 with K = 32 per instruction, the
// same 32 bytes), and the accumulator is scaled by a_scale * b_scale[n].
// Optional outputs: FP32 before the activation, BF16 after it, FP8 E4M3
// after it (scaled by c8_inv_scale, saturated to the finite range).
//
// Up to NBUF stages are in flight (a stage's copies take longer than its
// MMAs, and with K = 8,192 rows of a training batch there are 128 of them).
// A long chain is bound by the copies an SM keeps in flight, ~24 KB a
// microsecond (more or larger stages changed nothing).
//
// Training epilogues: with bwd_pre the value is multiplied by GELU's
// derivative at bwd_pre (the gradient through an activation), and C16T takes
// a transposed copy of C16 in the tiled layout below.
constexpr int kGemmThreads = 256;
__device__ __forceinline__ float gelu_grad(float x);
__device__ __forceinline__ long long tiled_off(int row, int k, int R);

template <int BN, bool F8, int NBUF>
__device__ __forceinline__ void gemm_tile(const GemmArgs &g, int m0, int n0) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr int kStageK = F8 ? 2 * kBK : kBK;    // elements of K per stage
  constexpr uint32_t kAStage = kBM * kBK * 2;  // 16 KB (128 bytes per row)
  constexpr uint32_t kBStage = BN * kBK * 2;
  auto sA = [&](int b) { return smem + (uint32_t)b * kAStage; };
  auto sB = [&](int b) { return smem + NBUF * kAStage + (uint32_t)b * kBStage; };
  __shared__ __align__(8) uint64_t bar[NBUF];
  __shared__ uint32_t tmem_slot;
  // a wait of stage s ran out: set in s_fail[s & 1], read after the next
  // stage's barrier, so that every thread reads the same
  __shared__ int s_fail[2];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int b = 0; b < NBUF; ++b) tc::mbar_init(&bar[b], 1);
    tc::fence_mbar_init();
    s_fail[0] = s_fail[1] = 0;
  }
  if (warp == 0) tc::tmem_alloc(&tmem_slot, BN);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  constexpr uint32_t idesc = F8 ? tc::idesc_e4m3_f32(kBM, BN) : tc::idesc_bf16_f32(kBM, BN);
  const int stages = (g.K + kStageK - 1) / kStageK;
  bool ok = true;
  int issued = 0;  // stages whose MMAs are on their way

  // Stage loader: every thread issues its 16-byte asynchronous copies
  // (cp.async) for stage s into buffer s mod NBUF, rows past M / N and
  // columns past K are zero-filled.  A warp copies 8 rows x 4 chunks: whole
  // 32-byte sectors of each row, 512 consecutive bytes of shared memory.
  // Each thread's rows are fixed, so their addresses are formed once.
  constexpr int kChunk = F8 ? 16 : 8;            // elements per 16-byte chunk
  constexpr int kWarps = kGemmThreads / 32;
  constexpr int kNA = kBM / 4 / kWarps, kNB = BN / 4 / kWarps;
  const int K = g.K, rl = lane & 7, kl = lane >> 3;
  const char *pa[kNA], *pb[kNB];
  bool ia[kNA], ib[kNB];
  const char *Abase = F8 ? (const char *)g.A8 : (const char *)g.A;
  const char *Bbase = F8 ? (const char *)g.B8 : (const char *)g.Bt;
  auto row_of = [&](int i) { return ((warp + i * kWarps) >> 1) * 8 + rl; };
  auto chunk_of = [&](int i) { return ((warp + i * kWarps) & 1) * 4 + kl; };
#pragma unroll
  for (int i = 0; i < kNA; ++i) {
    const int m = m0 + row_of(i);
    ia[i] = m < g.M;
    pa[i] = Abase + ((long long)(ia[i] ? m : 0) * g.lda + chunk_of(i) * kChunk) * (F8 ? 1 : 2);
  }
#pragma unroll
  for (int i = 0; i < kNB; ++i) {
    const int n = n0 + row_of(i);
    ib[i] = n < g.N;
    pb[i] = Bbase + ((long long)(ib[i] ? n : 0) * g.ldb + chunk_of(i) * kChunk) * (F8 ? 1 : 2);
  }
  auto load_stage = [&](int s) {
    const int b = s % NBUF;
    const uint32_t a0 = tc::smem_u32(sA(b)), b0 = tc::smem_u32(sB(b));
    const long long off = (long long)s * 128;  // a stage is 128 bytes of a row
#pragma unroll
    for (int i = 0; i < kNA; ++i) {
      const bool in = ia[i] && s * kStageK + chunk_of(i) * kChunk < K;
      cp_async16(a0 + stage_off(row_of(i), chunk_of(i)), in ? pa[i] + off : Abase, in ? 16 : 0);
    }
#pragma unroll
    for (int i = 0; i < kNB; ++i) {
      const bool in = ib[i] && s * kStageK + chunk_of(i) * kChunk < K;
      cp_async16(b0 + stage_off(row_of(i), chunk_of(i)), in ? pb[i] + off : Bbase, in ? 16 : 0);
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;" ::: "memory"); };

  for (int s = 0; s < NBUF - 1; ++s) {
    if (s < stages) load_stage(s);
    commit();  // one group per stage, also where there is none
  }
  for (int s = 0; s < stages; ++s) {
    const int b = s % NBUF;
    // stage s has landed in shared memory
    asm volatile("cp.async.wait_group %0;" ::"n"(NBUF - 2) : "memory");
    tc::fence_async_smem();
    __syncthreads();
    if (s_fail[(s + 1) & 1]) {
      ok = false;
      break;
    }
    if (tid == 0) {
      tc::tc_fence_after();
      const uint32_t a0 = tc::smem_u32(sA(b)), b0 = tc::smem_u32(sB(b));
#pragma unroll
      for (int kk = 0; kk < kBK / 16; ++kk) {
        // two core matrices along K per MMA: +256 bytes per K step of 16
        const uint64_t ad = tc::smem_desc(a0 + kk * 256, 128, 1024);
        const uint64_t bd = tc::smem_desc(b0 + kk * 256, 128, 1024);
        if constexpr (F8)
          tc::mma_e4m3(tmem, ad, bd, idesc, (s > 0 || kk > 0) ? 1u : 0u);
        else
          tc::mma_bf16(tmem, ad, bd, idesc, (s > 0 || kk > 0) ? 1u : 0u);
      }
      tc::mma_commit(&bar[b]);
    }
    issued = s + 1;
    // the buffer of stage s + NBUF - 1 is free once the MMAs of stage s - 1
    // are done; its loads overlap those of the stages between
    const int nx = s + NBUF - 1;
    if (nx < stages) {
      if (s > 0 &&
          !tc::mbar_wait(&bar[(s - 1) % NBUF], ((s - 1) / NBUF) & 1, kWaitLimit))
        s_fail[s & 1] = 1;
      else
        load_stage(nx);
    }
    commit();
  }
  // all MMAs done: the last stage's commit completes after every earlier one
  if (ok && stages > 0) {
    const int l = stages - 1;
    ok = !__syncthreads_or(!tc::mbar_wait(&bar[l % NBUF], (l / NBUF) & 1, kWaitLimit));
  }
  if (!ok) {
    if (tid == 0) atomicExch(g.err, SG_ERR_TIMEOUT);
    // copies and MMAs still in flight end (bounded) before the memory is freed
    asm volatile("cp.async.wait_all;" ::: "memory");
    for (int l = max(0, issued - NBUF); l < issued; ++l)
      tc::mbar_wait(&bar[l % NBUF], (l / NBUF) & 1, 1u << 16);
  }
  if (ok) {
    // Epilogue.  Warp w reads TMEM lanes 32 (w % 4) .. + 31 (tile rows) and
    // half w / 4 of each 64 columns.  Results are staged in shared memory (the
    // stage buffers are free now) and then written row by row, each warp
    // storing whole row segments: a lane holds a tile row, so its own stores
    // would be 16 bytes each, 32 rows apart (100,000 x 392 logits: 125 us).
    tc::tc_fence_after();
    constexpr int kPitch = BN * 2 + 16;  // bytes per staged row (bank offset)
    unsigned char *stage = smem;
    const int q = warp & 3, half = warp >> 2;
    const int lr = q * 32 + lane;
    const int row = m0 + lr;
    const bool vec32 = g.C32 && (g.ldc32 % 4) == 0 && (((uintptr_t)g.C32) & 15) == 0;
    constexpr int kPitch32 = 64 + 4;     // floats per staged row of 64 columns
    constexpr int kPitch8 = BN + 16;     // bytes per staged E4M3 row
    constexpr int kStage16 = kBM * kPitch, kStage32 = kBM * kPitch32 * 4;
    constexpr int kSmem = NBUF * (kAStage + kBStage);
    // what fits beside each other (wide tiles: not FP32 or E4M3 beside BF16)
    const bool st32 = vec32 && (!g.C16 || kStage16 + kStage32 <= kSmem);
    const bool st8 = g.C8 && !g.C16 && (g.ldc8 % 16) == 0 && (((uintptr_t)g.C8) & 15) == 0 &&
                     kStage32 + kBM * kPitch8 <= kSmem;
    float *stage32 = reinterpret_cast<float *>(smem + (g.C16 ? kStage16 : 0));
    unsigned char *stage8 = smem + kStage32;
    for (int cb = 0; cb < BN; cb += 64) {
    for (int c = cb + half * 32; c < cb + half * 32 + 32; c += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c, v);
      const int nb = n0 + c;
      // pre-activation: accumulator x a_scale b_scale[n] (E4M3) + bias[n],
      // one fused multiply-add
      float bs[16], sc[16];
      if constexpr (F8) {
        if (nb + 16 <= g.N && (((uintptr_t)(g.b_scale + nb)) & 15) == 0) {
#pragma unroll
          for (int i = 0; i < 16; i += 4) {
            const float4 s4 = __ldg(reinterpret_cast<const float4 *>(g.b_scale + nb + i));
            sc[i] = s4.x;
            sc[i + 1] = s4.y;
            sc[i + 2] = s4.z;
            sc[i + 3] = s4.w;
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) sc[i] = nb + i < g.N ? __ldg(g.b_scale + nb + i) : 0.0f;
        }
      }
      if (g.bias && nb + 16 <= g.N && (((uintptr_t)(g.bias + nb)) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 b4 = __ldg(reinterpret_cast<const float4 *>(g.bias + nb + i));
          bs[i] = b4.x;
          bs[i + 1] = b4.y;
          bs[i + 2] = b4.z;
          bs[i + 3] = b4.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) bs[i] = (g.bias && nb + i < g.N) ? __ldg(g.bias + nb + i) : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        float cs = 1.0f;
        if constexpr (F8) cs = g.a_scale * sc[i];
        v[i] = __fmaf_rn(v[i], cs, bs[i]);
      }
      if (st32) {
#pragma unroll
        for (int i = 0; i < 16; i += 4)
          *reinterpret_cast<float4 *>(stage32 + lr * kPitch32 + (c - cb) + i) =
              make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
      } else if (g.C32 && row < g.M) {
        float *dst = g.C32 + (long long)row * g.ldc32 + nb;
        if (vec32 && nb + 16 <= g.N) {
#pragma unroll
          for (int i = 0; i < 16; i += 4)
            *reinterpret_cast<float4 *>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {
          for (int i = 0; i < 16 && nb + i < g.N; ++i) dst[i] = v[i];
        }
      }
      if (g.C16) {
        float y[16];
        if (g.bwd_pre) {
          const float *pre = g.bwd_pre + (long long)row * g.N + nb;
          if (row < g.M && nb + 16 <= g.N && (((uintptr_t)pre) & 15) == 0) {
#pragma unroll
            for (int i = 0; i < 16; i += 4) {
              const float4 p4 = __ldg(reinterpret_cast<const float4 *>(pre + i));
              y[i] = v[i] * gelu_grad(p4.x);
              y[i + 1] = v[i + 1] * gelu_grad(p4.y);
              y[i + 2] = v[i + 2] * gelu_grad(p4.z);
              y[i + 3] = v[i + 3] * gelu_grad(p4.w);
            }
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              y[i] = row < g.M && nb + i < g.N ? v[i] * gelu_grad(pre[i]) : 0.0f;
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i) y[i] = g.act == 1 ? gelu_scaled(v[i], 0.5f) : v[i];
        }
        if (g.C16T && row < g.M) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (nb + i < g.N)
              *reinterpret_cast<__nv_bfloat16 *>(
                  reinterpret_cast<unsigned char *>(g.C16T) + tiled_off(nb + i, row, g.N)) =
                  __float2bfloat16_rn(y[i]);
        }
        uint32_t packed[8];
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(y[i], y[i + 1]);
          packed[i / 2] = *reinterpret_cast<const uint32_t *>(&h2);
        }
        uint4 *sp = reinterpret_cast<uint4 *>(stage + lr * kPitch + c * 2);
        sp[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        sp[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
      }
      if (g.C8 && (st8 || row < g.M)) {
        // 16 E4M3 values of this row (the output scale folded into the
        // activation), one 16-byte store when it fits
        const float hs = 0.5f * g.c8_inv_scale;
        float y[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          y[i] = g.act == 1 ? gelu_scaled(v[i], hs) : v[i] * g.c8_inv_scale;
        const uint4 pk = pack_e4m3_16(y);
        const uint32_t packed[4] = {pk.x, pk.y, pk.z, pk.w};
        uint8_t *dst = g.C8 + (long long)row * g.ldc8 + nb;
        if (st8) {
          *reinterpret_cast<uint4 *>(stage8 + lr * kPitch8 + c) = pk;
        } else if (nb + 16 <= g.N && (((uintptr_t)dst) & 15) == 0) {
          *reinterpret_cast<uint4 *>(dst) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        } else {
          const uint8_t *bytes = reinterpret_cast<const uint8_t *>(packed);
          for (int i = 0; i < 16 && nb + i < g.N; ++i) dst[i] = bytes[i];
        }
      }
    }
    if (st32) {
      // 64 columns of every row: 16 lanes a row
      __syncthreads();
      for (int idx = tid; idx < kBM * 16; idx += kGemmThreads) {
        const int r = idx >> 4, j = (idx & 15) * 4;
        const int grow = m0 + r, col = n0 + cb + j;
        if (grow >= g.M || col >= g.N) continue;
        const float4 val = *reinterpret_cast<const float4 *>(stage32 + r * kPitch32 + j);
        float *dst = g.C32 + (long long)grow * g.ldc32 + col;
        if (col + 4 <= g.N) {
          *reinterpret_cast<float4 *>(dst) = val;
        } else {
          const float x[4] = {val.x, val.y, val.z, val.w};
          for (int i = 0; i < 4 && col + i < g.N; ++i) dst[i] = x[i];
        }
      }
      __syncthreads();
    }
    }
    if (st8) {
      __syncthreads();
      constexpr int kVecPerRow = BN / 16;
      for (int idx = tid; idx < kBM * kVecPerRow; idx += kGemmThreads) {
        const int r = idx / kVecPerRow, j = (idx - r * kVecPerRow) * 16;
        const int grow = m0 + r, col = n0 + j;
        if (grow >= g.M || col >= g.N) continue;
        const uint4 val = *reinterpret_cast<const uint4 *>(stage8 + r * kPitch8 + j);
        uint8_t *dst = g.C8 + (long long)grow * g.ldc8 + col;
        if (col + 16 <= g.N) {
          *reinterpret_cast<uint4 *>(dst) = val;
        } else {
          const uint8_t *x = reinterpret_cast<const uint8_t *>(&val);
          for (int i = 0; i < 16 && col + i < g.N; ++i) dst[i] = x[i];
        }
      }
    }
    if (g.C16) {
      __syncthreads();
      constexpr int kVecPerRow = BN * 2 / 16;
      const bool vec16 = (g.ldc16 % 8) == 0 && (((uintptr_t)g.C16) & 15) == 0;
      for (int idx = tid; idx < kBM * kVecPerRow; idx += kGemmThreads) {
        const int r = idx / kVecPerRow, j = idx - r * kVecPerRow;
        const int grow = m0 + r, col = n0 + j * 8;
        if (grow >= g.M || col >= g.N) continue;
        const uint4 val = *reinterpret_cast<const uint4 *>(stage + r * kPitch + j * 16);
        __nv_bfloat16 *dst = g.C16 + (long long)grow * g.ldc16 + col;
        if (vec16 && col + 8 <= g.N) {
          *reinterpret_cast<uint4 *>(dst) = val;
        } else {
          const __nv_bfloat16 *hv = reinterpret_cast<const __nv_bfloat16 *>(&val);
          for (int i = 0; i < 8 && col + i < g.N; ++i) dst[i] = hv[i];
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, BN);
}

template <int BN, bool F8, int NBUF>
__global__ void __launch_bounds__(kGemmThreads) k_gemm_tc(const __grid_constant__ GemmArgs g) {
  gemm_tile<BN, F8, NBUF>(g, blockIdx.x * kBM, blockIdx.y * BN);
}

// Operands of the weight gradients, laid out as the tensor core reads them:
// element (row, k) of an R x K matrix (R a multiple of 8, K padded to whole
// steps of 64 with zeros) at byte ((k / 64) (R / 8) + row / 8) 1024 +
// (k % 64 / 8) 128 + (row % 8) 16 + (k % 8) 2, so the rows r0 .. of one step
// are consecutive and come in with one bulk copy.
__device__ __forceinline__ long long tiled_off(int row, int k, int R) {
  return (((long long)(k >> 6) * (R >> 3) + (row >> 3)) << 10) + ((k & 63) >> 3) * 128 +
         (row & 7) * 16 + (k & 7) * 2;
}

// Up to four contractions C = A . B^T of tiled operands in one launch: the
// weight gradients of a training step, (256..392) x (16..256) outputs with K
// = the batch.  They are a few tiles each, bound by their chain of steps (128
// for 8,192 rows), so the chains run side by side.  One thread queues the
// bulk copies of the next kGroupBuf - 1 steps, another issues the MMAs; with
// per-thread 16-byte copies from row-major operands an SM kept ~24 KB a
// microsecond in flight (126 us for the four; one after the other in 128 x
// 256 tiles 1,260 us).  Each output is the same chain of additions as on its
// own (a split K would not be).
constexpr int kGroupBN = 64, kGroupBuf = 8;
struct GroupArgs {
  const unsigned char *A[4], *B[4];  // tiled, M x K and N x K
  float *C[4];                       // M x N, row-major
  int M[4], N[4], K, n, first[5];    // tiles of contraction i: first[i] .. first[i + 1] - 1
  int *err;
};
__global__ void __launch_bounds__(kGemmThreads)
k_gemm_group(const __grid_constant__ GroupArgs q) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr uint32_t kAStage = kBM * 128, kBStage = kGroupBN * 128;
  __shared__ __align__(8) uint64_t full[kGroupBuf], empty[kGroupBuf], done;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail, s_queued;  // a wait ran out; steps queued
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int i = 0;
  while (i + 1 < q.n && (int)blockIdx.x >= q.first[i + 1]) ++i;
  const int M = q.M[i], N = q.N[i];
  const int t = (int)blockIdx.x - q.first[i], nt = (N + kGroupBN - 1) / kGroupBN;
  const int m0 = (t / nt) * kBM, n0 = (t % nt) * kGroupBN;
  if (tid == 0) {
    for (int b = 0; b < kGroupBuf; ++b) {
      tc::mbar_init(&full[b], 1);
      tc::mbar_init(&empty[b], 1);
    }
    tc::mbar_init(&done, 1);
    tc::fence_mbar_init();
    s_fail = 0;
  }
  if (warp == 0) tc::tmem_alloc(&tmem_slot, kGroupBN);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int steps = (q.K + 63) >> 6;
  unsigned char *sA = smem, *sB = smem + kGroupBuf * kAStage;
  if (tid == 0) {
    // producer: rows past M or N are not copied (they only reach outputs
    // that are not written)
    const uint32_t ab = (uint32_t)min(kBM, M - m0) * 128, bb = (uint32_t)min(kGroupBN, N - n0) * 128;
    const unsigned char *A = q.A[i] + (long long)m0 * 128, *B = q.B[i] + (long long)n0 * 128;
    int k = 0;
    for (; k < steps; ++k) {
      const int b = k % kGroupBuf;
      if (k >= kGroupBuf &&
          !tc::mbar_wait(&empty[b], ((k / kGroupBuf) - 1) & 1, kWaitLimit)) {
        s_fail = 1;
        break;
      }
      tc::mbar_arrive_expect_tx(&full[b], ab + bb);
      tc::bulk_g2s(sA + b * kAStage, A + (long long)k * M * 128, ab, &full[b]);
      tc::bulk_g2s(sB + b * kBStage, B + (long long)k * N * 128, bb, &full[b]);
    }
    s_queued = k;
  } else if (tid == 32) {
    constexpr uint32_t idesc = tc::idesc_bf16_f32(kBM, kGroupBN);
    bool ok = true;
    for (int k = 0; k < steps; ++k) {
      const int b = k % kGroupBuf;
      if (!tc::mbar_wait(&full[b], (k / kGroupBuf) & 1, kWaitLimit)) {
        ok = false;
        break;
      }
      tc::tc_fence_after();
      const uint32_t a0 = tc::smem_u32(sA + b * kAStage), b0 = tc::smem_u32(sB + b * kBStage);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
        tc::mma_bf16(tmem, tc::smem_desc(a0 + kk * 256, 128, 1024),
                     tc::smem_desc(b0 + kk * 256, 128, 1024), idesc, (k > 0 || kk > 0) ? 1u : 0u);
      tc::mma_commit(&empty[b]);
    }
    tc::mma_commit(&done);
    if (!ok) s_fail = 1;
  }
  __syncwarp();
  // every MMA issued is done (bounded; also where a wait gave up)
  if (!tc::mbar_wait(&done, 0, kWaitLimit)) s_fail = 1;
  __syncthreads();
  if (s_fail) {
    if (tid == 0) {
      // bulk copies still in flight land before the block leaves
      for (int k = max(0, s_queued - kGroupBuf); k < s_queued; ++k)
        tc::mbar_wait(&full[k % kGroupBuf], (k / kGroupBuf) & 1, 1u << 16);
      atomicExch(q.err, SG_ERR_TIMEOUT);
    }
  } else {
    tc::tc_fence_after();
    const int w = warp & 3, half = warp >> 2, row = m0 + w * 32 + lane;
    for (int c = half * 32; c < half * 32 + 32; c += 16) {
      float v[16];
      tc::tmem_ld16(tmem + ((uint32_t)(w * 32) << 16) + (uint32_t)c, v);
      if (row < M) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (n0 + c + j < N) q.C[i][(long long)row * N + n0 + c + j] = v[j];
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, kGroupBN);
}

std::mutex g_err_mu;
int *g_err_buf[64] = {};

int gemm_err_buf(int **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return SG_ERR_CUDA;
  }
  std::lock_guard<std::mutex> lock(g_err_mu);
  if (!g_err_buf[dev]) {
    if (cudaMalloc(&g_err_buf[dev], sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      return SG_ERR_NOMEM;
    }
    cudaMemset(g_err_buf[dev], 0, sizeof(int));
  }
  *out = g_err_buf[dev];
  return SG_OK;
}

// Opts a kernel into `smem` bytes of dynamic shared memory, once per device.
template <typename K>
void allow_smem(K *kernel, size_t smem, unsigned long long &done) {
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 64 && !((done >> dev) & 1ull)) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    done |= 1ull << dev;
  }
}

constexpr size_t gemm_smem(int bn, int nbuf) {
  return nbuf * ((size_t)kBM * kBK * 2 + (size_t)bn * kBK * 2);
}

template <int BN, bool F8, int NBUF>
void launch_gemm(const GemmArgs &g, cudaStream_t st) {
  static unsigned long long attr_set = 0;
  allow_smem(k_gemm_tc<BN, F8, NBUF>, gemm_smem(BN, NBUF), attr_set);
  const dim3 grid((unsigned)((g.M + kBM - 1) / kBM), (unsigned)((g.N + BN - 1) / BN));
  k_gemm_tc<BN, F8, NBUF><<<grid, kGemmThreads, gemm_smem(BN, NBUF), st>>>(g);
}

// The widest tile that still gives every SM (152) one, else the narrowest:
// 8,192 x 256 x 256 took 20-28 us as 64 tiles of 256 columns, with 88 SMs idle.
constexpr int kGemmSms = 152;
template <bool F8>
void launch_gemm_tiles(const GemmArgs &g, cudaStream_t st) {
  const long long mt = (g.M + kBM - 1) / kBM;
  auto tiles = [&](int bn) { return mt * ((g.N + bn - 1) / bn); };
  if (g.N > 128 && tiles(256) >= kGemmSms)
    launch_gemm<256, F8, 2>(g, st);
  else if (g.N > 64 && tiles(128) >= kGemmSms)
    launch_gemm<128, F8, 3>(g, st);
  else
    launch_gemm<64, F8, 4>(g, st);
}

void launch_gemm_group(GroupArgs &q, cudaStream_t st) {
  q.first[0] = 0;
  for (int i = 0; i < q.n; ++i)
    q.first[i + 1] =
        q.first[i] + (q.M[i] + kBM - 1) / kBM * ((q.N[i] + kGroupBN - 1) / kGroupBN);
  static unsigned long long attr_set = 0;
  allow_smem(k_gemm_group, gemm_smem(kGroupBN, kGroupBuf), attr_set);
  k_gemm_group<<<q.first[q.n], kGemmThreads, gemm_smem(kGroupBN, kGroupBuf), st>>>(q);
}

}  // namespace

namespace sg {

int gemm_bf16(const GemmArgs &g0, cudaStream_t st) {
  GemmArgs g = g0;
  const bool f8 = g.f8 != 0;
  const int align = f8 ? 16 : 8;  // elements per 16 bytes
  const void *A = f8 ? (const void *)g.A8 : (const void *)g.A;
  const void *B = f8 ? (const void *)g.B8 : (const void *)g.Bt;
  if (g.M < 0 || g.N < 0 || g.K < 0 || (g.K % align) != 0 || g.lda < g.K || g.ldb < g.K ||
      (g.lda % align) != 0 || (g.ldb % align) != 0 || !A || !B ||
      (!g.C32 && !g.C16 && !g.C8) || (((uintptr_t)A | (uintptr_t)B) & 15) != 0 ||
      (f8 && !g.b_scale) || (g.C8 && g.ldc8 < g.N))
    return SG_ERR_ARG;
  if (g.M == 0 || g.N == 0) return SG_OK;
  if (!g.err) {
    int rc = gemm_err_buf(&g.err);
    if (rc) return rc;
  }
  if (f8)
    launch_gemm_tiles<true>(g, st);
  else
    launch_gemm_tiles<false>(g, st);
  return SG_OK;
}

int gemm_prepare() {
  int *e = nullptr;
  return gemm_err_buf(&e);
}

int gemm_check(cudaStream_t st) {
  int *e = nullptr;
  int rc = gemm_err_buf(&e);
  if (rc) return rc;
  int h = 0;
  if (cudaMemcpyAsync(&h, e, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    cudaGetLastError();
    return SG_ERR_CUDA;
  }
  if (h) {
    cudaMemsetAsync(e, 0, sizeof(int), st);
    return h;
  }
  return SG_OK;
}

}  // namespace sg

extern "C" int sg_gemm_bf16(const void *A, int32_t lda, const void *Bt, int32_t ldb, int32_t M,
                            int32_t N, int32_t K, const float *bias, int32_t act, float *C32,
                            int32_t ldc32, void *C16, int32_t ldc16, void *stream) {
  GemmArgs g{};
  g.A = (const __nv_bfloat16 *)A;
  g.lda = lda;
  g.Bt = (const __nv_bfloat16 *)Bt;
  g.ldb = ldb;
  g.M = M;
  g.N = N;
  g.K = K;
  g.bias = bias;
  g.act = act;
  g.C32 = C32;
  g.ldc32 = ldc32;
  g.C16 = (__nv_bfloat16 *)C16;
  g.ldc16 = ldc16;
  g.err = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = sg::gemm_bf16(g, st);
  if (rc) return rc;
  return sg::gemm_check(st);
}

extern "C" int sg_gemm_bf16_to_fp8(const void *A, int32_t lda, const void *Bt, int32_t ldb,
                                   int32_t M, int32_t N, int32_t K, const float *bias,
                                   int32_t act, void *C8, int32_t ldc8, float c8_inv_scale,
                                   void *stream) {
  GemmArgs g{};
  g.A = (const __nv_bfloat16 *)A;
  g.lda = lda;
  g.Bt = (const __nv_bfloat16 *)Bt;
  g.ldb = ldb;
  g.M = M;
  g.N = N;
  g.K = K;
  g.bias = bias;
  g.act = act;
  g.C8 = (uint8_t *)C8;
  g.ldc8 = ldc8;
  g.c8_inv_scale = c8_inv_scale;
  g.err = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = sg::gemm_bf16(g, st);
  if (rc) return rc;
  return sg::gemm_check(st);
}

extern "C" int sg_gemm_fp8(const void *A8, int32_t lda, const void *B8, int32_t ldb, int32_t M,
                           int32_t N, int32_t K, float a_scale, const float *b_scale,
                           const float *bias, int32_t act, float *C32, int32_t ldc32,
                           void *C16, int32_t ldc16, void *C8, int32_t ldc8,
                           float c8_inv_scale, void *stream) {
  GemmArgs g{};
  g.f8 = 1;
  g.A8 = (const uint8_t *)A8;
  g.lda = lda;
  g.B8 = (const uint8_t *)B8;
  g.ldb = ldb;
  g.M = M;
  g.N = N;
  g.K = K;
  g.a_scale = a_scale;
  g.b_scale = b_scale;
  g.bias = bias;
  g.act = act;
  g.C32 = C32;
  g.ldc32 = ldc32;
  g.C16 = (__nv_bfloat16 *)C16;
  g.ldc16 = ldc16;
  g.C8 = (uint8_t *)C8;
  g.ldc8 = ldc8;
  g.c8_inv_scale = c8_inv_scale;
  g.err = nullptr;
  cudaStream_t st = (cudaStream_t)stream;
  const int rc = sg::gemm_bf16(g, st);
  if (rc) return rc;
  return sg::gemm_check(st);
}

// ---------------------------------------------------------------------------
// Element-wise kernels of the emulator: training loss, GELU backward,
// transposes, bias gradients, Adam, input features, output sampling.
// ---------------------------------------------------------------------------

namespace {

constexpr int kHeads = 3;    // one head per age class
constexpr int kBins = 129;   // increments -64 .. 64
constexpr int kHalf = 64;

// d/dx of the tanh-form GELU: 0.5 (1 + t) + 0.5 x (1 - t^2) c (1 + 3 a x^2)
__device__ __forceinline__ float gelu_grad(float x) {
  const float c = 0.7978845608028654f, a = 0.044715f;
  const float t = tanh_fast(c * (x + a * x * x * x));
  return 0.5f * (1.0f + t) + 0.5f * x * (1.0f - t * t) * c * (1.0f + 3.0f * a * x * x);
}

// Cross-entropy over the three 129-way heads, one warp per row: loss and
// d loss / d logits (scaled by 1 / B, BF16; padding columns get 0).  Each
// head's logits are read once into registers; the block's losses go out in
// one atomic (8,192 rows x 392: one atomic per row took most of 24 us).
__global__ void __launch_bounds__(256)
k_ce_loss(const float *__restrict__ logits, int ldl, const int32_t *__restrict__ tgt, int B,
          __nv_bfloat16 *dlog, int ldd, int ncols_grad, double *loss_sum) {
  __shared__ double s_loss[8];
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  constexpr int kPer = (kBins + 31) / 32;
  float loss = 0.0f;
  if (warp < B) {
    const float *row = logits + (long long)warp * ldl;
    __nv_bfloat16 *grow = dlog + (long long)warp * ldd;
    const float invB = 1.0f / (float)B;
    float x[kHeads][kPer];
#pragma unroll
    for (int h = 0; h < kHeads; ++h)
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        x[h][i] = lane + 32 * i < kBins ? row[h * kBins + lane + 32 * i] : -INFINITY;
#pragma unroll
    for (int h = 0; h < kHeads; ++h) {
      float mx = -INFINITY;
#pragma unroll
      for (int i = 0; i < kPer; ++i) mx = fmaxf(mx, x[h][i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      float se = 0.0f;
#pragma unroll
      for (int i = 0; i < kPer; ++i)
        if (lane + 32 * i < kBins) se += expf(x[h][i] - mx);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
      const float lz = mx + logf(se);
      const int t = tgt[(long long)warp * kHeads + h];
      if (lane == 0) loss += lz - row[h * kBins + t];
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int c = lane + 32 * i;
        if (c >= kBins) continue;
        const float p = expf(x[h][i] - lz) - (c == t ? 1.0f : 0.0f);
        grow[h * kBins + c] = __float2bfloat16_rn(p * invB);
      }
    }
    for (int c = kHeads * kBins + lane; c < ncols_grad; c += 32)
      grow[c] = __float2bfloat16_rn(0.0f);
  }
  if (lane == 0) s_loss[threadIdx.x >> 5] = (double)loss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) sum += s_loss[i];
    atomicAdd(loss_sum, sum);
  }
}

__global__ void k_gelu_bwd(const float *__restrict__ dpost, const float *__restrict__ pre,
                           long long n, __nv_bfloat16 *dpre) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dpre[i] = __float2bfloat16_rn(dpost[i] * gelu_grad(pre[i]));
}

// dst[c][r] = src[r][c] through 32 x 32 shared-memory tiles.
__global__ void k_transpose(const __nv_bfloat16 *__restrict__ src, int rows, int cols,
                            __nv_bfloat16 *dst) {
  __shared__ __nv_bfloat16 tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < rows && c < cols) tile[i][threadIdx.x] = src[(long long)r * cols + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < rows && c < cols) dst[(long long)c * rows + r] = tile[threadIdx.x][i];
  }
}

// FP8 quantisation.  Per row of W (rows x cols, FP32): scale = max |w| /
// 448 (the largest finite E4M3 value; 1 for a zero row), W8 = e4m3(w /
// scale) rounded to nearest even and saturated.  One block per row.
__global__ void k_quant_rows_fp8(const float *__restrict__ W, int rows, int cols, uint8_t *W8,
                                 float *scale) {
  __shared__ float s_max[8];
  const int r = blockIdx.x;
  const float *w = W + (long long)r * cols;
  float m = 0.0f;
  for (int k = threadIdx.x; k < cols; k += blockDim.x) m = fmaxf(m, fabsf(w[k]));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
  __syncthreads();
  float mx = 0.0f;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) mx = fmaxf(mx, s_max[i]);
  const float sc = mx > 0.0f ? mx / 448.0f : 1.0f;
  if (threadIdx.x == 0) scale[r] = sc;
  for (int k = threadIdx.x; k < cols; k += blockDim.x)
    W8[(long long)r * cols + k] =
        (uint8_t)__nv_cvt_float_to_fp8(w[k] / sc, __NV_SATFINITE, __NV_E4M3);
}

// x8 = e4m3(x * inv_scale) for BF16 x, saturated.
__global__ void k_quant_bf16_fp8(const __nv_bfloat16 *__restrict__ x, long long n, float inv_scale,
                                 uint8_t *out) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = (uint8_t)__nv_cvt_float_to_fp8(__bfloat162float(x[i]) * inv_scale, __NV_SATFINITE,
                                            __NV_E4M3);
}

// *out = max |x_i| over BF16 x (out starts at 0; non-negative floats order
// like their bit patterns).
__global__ void k_absmax_bf16(const __nv_bfloat16 *__restrict__ x, long long n, float *out) {
  float m = 0.0f;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(__bfloat162float(x[i])));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(out), __float_as_int(m));
}

__global__ void k_colsum(const __nv_bfloat16 *__restrict__ src, int rows, int cols, float *out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  float s = 0.0f;
  for (int r = 0; r < rows; ++r) s += __bfloat162float(src[(long long)r * cols + c]);
  out[c] = s;
}

__global__ void k_adam(float *p, const float *__restrict__ g, float *m, float *v, long long n,
                       float lr, float b1, float b2, float eps, float c1, float c2,
                       __nv_bfloat16 *p16) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (p16) p16[i] = __float2bfloat16_rn(pi);
  }
}

}  // namespace

namespace sg {

// Input features of one SISe3 node for the emulator (the BF16 values of the
// 16 inputs), and whether the node is in the emulator's range (herd <=
// max_herd, phi_lo <= phi <= phi_hi, total transition rate >= min_rate).
__device__ __forceinline__ bool emu_feature_row(const int32_t *un, double phi,
                                                const EmuParams &ep, __nv_bfloat16 *row) {
  int herd = 0;
#pragma unroll
  for (int p = 0; p < 6; ++p) herd += un[p];
  // total transition rate: S_a -> I_a at upsilon_a phi S_a, I_a -> S_a at
  // gamma_a I_a
  double a0 = 0.0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    a0 += ep.gdata[a] * phi * (double)un[2 * a] + ep.gdata[3 + a] * (double)un[2 * a + 1];
  const bool in = herd <= ep.max_herd && phi >= ep.phi_lo && phi <= ep.phi_hi &&
                  a0 >= ep.min_rate;
  float f[16];
#pragma unroll
  for (int p = 0; p < 6; ++p) f[p] = log1pf((float)max(un[p], 0));
  f[6] = (float)phi;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f[7 + a] = 50.0f * (float)ep.gdata[a];
    f[10 + a] = 10.0f * (float)ep.gdata[3 + a];
  }
  f[13] = f[14] = f[15] = 0.0f;
#pragma unroll
  for (int k = 0; k < 16; ++k) row[k] = __float2bfloat16_rn(f[k]);
  return in;
}

__global__ void k_emu_features(const int32_t *__restrict__ u, const double *__restrict__ v,
                               long long units, EmuParams ep, __nv_bfloat16 *feat,
                               int32_t *flag) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < units;
       i += (long long)gridDim.x * blockDim.x)
    flag[i] = emu_feature_row(u + i * 6, v[i], ep, feat + i * 16) ? 1 : 0;
}

// Sample each in-range node's increments from the emulator's three heads:
// softmax over the 129 bins (weights 2^(z - max z) with z = logit log2 e, the
// hardware 2^x), inverse CDF at a uniform from the emulator's
// Philox stream (seed, replicate, node, day), and clamp so that neither S_a
// nor I_a becomes negative (each age class keeps its size within the day).
// One warp per node; lane l holds bins 5 l .. 5 l + 4.
__global__ void k_emu_sample(const float *__restrict__ logits, int ldl,
                             const int32_t *__restrict__ u, const int32_t *__restrict__ flag,
                             long long units, int n_nodes, uint32_t k0, uint32_t k1, int T,
                             int32_t *delta) {
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= units) return;
  int32_t *out = delta + w * 4;
  if (!flag[w]) {
    if (lane == 0) out[3] = 0;
    return;
  }
  const int rep = (int)(w / n_nodes), node = (int)(w - (long long)rep * n_nodes);
  const U4 x = philox10(U4{0u, (uint32_t)node, (uint32_t)T, (SG_STREAM_EMU << 24) | (uint32_t)rep},
                        k0, k1);
  const uint32_t words[3] = {x.x, x.y, x.z};
  const float *row = logits + w * ldl;
  for (int h = 0; h < kHeads; ++h) {
    const float *lg = row + h * kBins;
    float vals[5];
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const int c = lane * 5 + j;
      vals[j] = c < kBins ? lg[c] * kLog2e : -INFINITY;
      mx = fmaxf(mx, vals[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float part = 0.0f;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      vals[j] = lane * 5 + j < kBins ? ex2_fast(vals[j] - mx) : 0.0f;
      part += vals[j];
    }
    // inclusive scan of the lane sums
    float incl = part;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const float total = __shfl_sync(0xffffffffu, incl, 31);
    const float target = ((float)(words[h] >> 8) + 0.5f) * (1.0f / 16777216.0f) * total;
    // the lane whose range holds the target, then the bin inside it
    const unsigned ge = __ballot_sync(0xffffffffu, incl >= target);
    const int owner = ge ? __ffs(ge) - 1 : 31;
    int bin = kBins - 1;
    if (lane == owner) {
      float acc = incl - part;
      bin = min(lane * 5 + 4, kBins - 1);
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        acc += vals[j];
        if (acc >= target && lane * 5 + j < kBins) {
          bin = lane * 5 + j;
          break;
        }
      }
    }
    bin = __shfl_sync(0xffffffffu, bin, owner);
    if (lane == 0) {
      const int S = u[w * 6 + 2 * h], I = u[w * 6 + 2 * h + 1];
      int d = bin - kHalf;
      d = max(d, -I);
      d = min(d, S);
      out[h] = d;
    }
  }
  if (lane == 0) out[3] = 1;
}

// Training targets: the one-day increment of I_a, as a bin index in 0..128
// (clamped to the edge bins).
__global__ void k_emu_targets(const int32_t *__restrict__ u0, const int32_t *__restrict__ u1,
                              long long units, int32_t *tgt) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < units;
       i += (long long)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int d = u1[i * 6 + 2 * a + 1] - u0[i * 6 + 2 * a + 1];
      tgt[i * 3 + a] = min(max(d + kHalf, 0), kBins - 1);
    }
  }
}

// ---------------------------------------------------------------------------
// The engine's FP8 inference chain: one persistent kernel per layer (one CTA
// per SM), the layer's weights resident in shared memory, activations in a
// tiled layout that one bulk copy moves, and (hidden layers) two tensor-memory
// accumulators, so that the epilogue of one 128-row tile overlaps the MMAs of
// the next.  Warp roles: producer warps (bulk copies, or the input features
// computed in place), one MMA warp (one elected thread issues tcgen05.mma),
// epilogue warps (tcgen05.ld, scale, bias, activation, store).
//
// Tiled layout of a matrix with rows padded to a multiple of 128 and Kb bytes
// per row: tile t (rows 128 t .. 128 t + 127) occupies bytes [128 Kb t,
// 128 Kb (t + 1)), as Kb / 16 chunks of 128 rows x 16 bytes (chunk c at
// 2048 c, row r of it at 16 r).  Copied to shared memory this is the
// no-swizzle K-major operand layout with 8-row core matrices 128 bytes apart
// along M and 2048 bytes apart along K.  A weight image uses the same layout
// with all of its N rows in one tile (chunk c at 16 N c).
//
// Layer kinds: 0, the input layer: features computed from the node states in
// the kernel (BF16, K = 16), 256 outputs, GELU, E4M3 out; 1, a hidden layer:
// E4M3 in (K = 256), 256 outputs, GELU, E4M3 out; 2, the output layer fused
// with the sampler: E4M3 in, head h's 129 logits at accumulator columns
// 144 h .. 144 h + 128, sampled as k_emu_sample samples them, bit for bit.
// Every layer's arithmetic is that of k_gemm_tc on the same operands.
// ---------------------------------------------------------------------------
constexpr int kEmuHeadPitch = 144;               // accumulator columns per head
constexpr int kEmuHeadCols = 3 * kEmuHeadPitch;  // 432 (MMAs of N = 256 and 176)
constexpr uint32_t kEmuTmemCols = 512;
constexpr uint32_t kEmuMinSmem = 120u * 1024u;   // one CTA per SM (its TMEM is 512 columns)

template <int L>
struct EmuLayerCfg;
template <>
struct EmuLayerCfg<0> {
  static constexpr bool kF8 = false;
  static constexpr int kKb = 32, kN = 256, kStages = 4, kAcc = 2, kProdWarps = 4,
                       kEpiWarps = 16;
};
template <>
struct EmuLayerCfg<1> {
  static constexpr bool kF8 = true;
  static constexpr int kKb = 256, kN = 256, kStages = 2, kAcc = 2, kProdWarps = 1,
                       kEpiWarps = 16;
};
template <>
struct EmuLayerCfg<2> {
  static constexpr bool kF8 = true;
  static constexpr int kKb = 256, kN = kEmuHeadCols, kStages = 2, kAcc = 1, kProdWarps = 1,
                       kEpiWarps = 12;
};

template <int L>
constexpr int emu_layer_threads() {
  return (EmuLayerCfg<L>::kProdWarps + 1 + EmuLayerCfg<L>::kEpiWarps) * 32;
}

// weight image, A stages, per-column accumulator factor and bias
template <int L>
constexpr uint32_t emu_layer_smem() {
  using C = EmuLayerCfg<L>;
  return (uint32_t)C::kN * C::kKb + (uint32_t)C::kStages * 128u * C::kKb + 8u * C::kN;
}

__device__ __forceinline__ void emu_fail(volatile int *s_fail, int *err) {
  *s_fail = 1;
  atomicExch(err, SG_ERR_TIMEOUT);
}

template <int L>
__global__ void __launch_bounds__(emu_layer_threads<L>(), 1) k_emu_layer(const EmuChainArgs a) {
  using C = EmuLayerCfg<L>;
  constexpr uint32_t kATile = 128u * C::kKb;
  constexpr uint32_t kWBytes = (uint32_t)C::kN * C::kKb;
  constexpr int kKSteps = C::kKb / 32;  // 32 bytes of K per MMA
  constexpr int kMmaWarp = C::kProdWarps, kEpi0 = C::kProdWarps + 1;
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char *sW = smem;
  unsigned char *sA = smem + kWBytes;
  float *sScale = reinterpret_cast<float *>(sA + C::kStages * kATile);
  float *sBias = sScale + C::kN;
  __shared__ __align__(8) uint64_t bar_w, bar_full[C::kStages], bar_empty[C::kStages],
      bar_tfull[C::kAcc], bar_tempty[C::kAcc];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bar_w, 1);
    for (int s = 0; s < C::kStages; ++s) {
      tc::mbar_init(&bar_full[s], L == 0 ? 128 : 1);
      tc::mbar_init(&bar_empty[s], 1);
    }
    for (int b = 0; b < C::kAcc; ++b) {
      tc::mbar_init(&bar_tfull[b], 1);
      tc::mbar_init(&bar_tempty[b], C::kEpiWarps);
    }
    tc::fence_mbar_init();
    s_fail = 0;
  }
  // the accumulator's factor a_scale * w_scale[n] (E4M3 layers), the bias
  for (int n = threadIdx.x; n < C::kN; n += blockDim.x) {
    sScale[n] = C::kF8 ? a.a_scale * a.wscale[n] : 1.0f;
    sBias[n] = a.bias[n];
  }
  if (warp == kMmaWarp) tc::tmem_alloc(&tmem_slot, kEmuTmemCols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  const int my_tiles = (a.n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;

  if (warp < C::kProdWarps) {
    // ---- producer ----
    if (threadIdx.x == 0) {
      tc::mbar_arrive_expect_tx(&bar_w, kWBytes);
      for (uint32_t off = 0; off < kWBytes; off += 16384u)
        tc::bulk_g2s(sW + off, a.W + off, kWBytes - off < 16384u ? kWBytes - off : 16384u, &bar_w);
    }
    if constexpr (L == 0) {
      // four warps, thread p writes row p of each tile: its 16 BF16
      // features as two 16-byte pieces (chunks 0 and 1)
      const int p = threadIdx.x;
      for (int i = 0; i < my_tiles; ++i) {
        const int s = i % C::kStages, k = i / C::kStages;
        if (k > 0 && !tc::mbar_wait(&bar_empty[s], (k - 1) & 1, kWaitLimit)) {
          emu_fail(&s_fail, a.err);
          break;
        }
        if (s_fail) break;
        const long long w = ((long long)blockIdx.x + (long long)i * gridDim.x) * 128 + p;
        __align__(16) __nv_bfloat16 row[16];
        if (w < a.units) {
          a.flag[w] = emu_feature_row(a.u + w * 6, a.v[w], a.ep, row) ? 1 : 0;
        } else {
#pragma unroll
          for (int k2 = 0; k2 < 16; ++k2) row[k2] = __float2bfloat16_rn(0.0f);
        }
        const uint4 *r4 = reinterpret_cast<const uint4 *>(row);
        unsigned char *stage = sA + s * kATile;
        *reinterpret_cast<uint4 *>(stage + p * 16) = r4[0];
        *reinterpret_cast<uint4 *>(stage + 2048 + p * 16) = r4[1];
        tc::fence_async_smem();
        tc::mbar_arrive(&bar_full[s]);
      }
      if (threadIdx.x == 0) tc::mbar_wait(&bar_w, 0, kWaitLimit);
    } else {
      if (lane == 0) {
        int last[C::kStages];
#pragma unroll
        for (int s = 0; s < C::kStages; ++s) last[s] = -1;
        for (int i = 0; i < my_tiles; ++i) {
          const int s = i % C::kStages, k = i / C::kStages;
          if (k > 0 && !tc::mbar_wait(&bar_empty[s], (k - 1) & 1, kWaitLimit)) {
            emu_fail(&s_fail, a.err);
            break;
          }
          if (s_fail) break;
          const long long t = (long long)blockIdx.x + (long long)i * gridDim.x;
          tc::mbar_arrive_expect_tx(&bar_full[s], kATile);
          tc::bulk_g2s(sA + s * kATile, a.A + t * kATile, kATile, &bar_full[s]);
          last[s] = k;
        }
        // no copy of ours may still be landing in shared memory at exit
        tc::mbar_wait(&bar_w, 0, kWaitLimit);
#pragma unroll
        for (int s = 0; s < C::kStages; ++s)
          if (last[s] >= 0) tc::mbar_wait(&bar_full[s], last[s] & 1, kWaitLimit);
      }
      __syncwarp();
    }
  } else if (warp == kMmaWarp) {
    // ---- MMA issue ----
    if (lane == 0) {
      int last_b = -1, last_kb = 0;
      bool ok = tc::mbar_wait(&bar_w, 0, kWaitLimit);
      const uint32_t a0 = tc::smem_u32(sA), w0 = tc::smem_u32(sW);
      for (int i = 0; ok && i < my_tiles; ++i) {
        const int s = i % C::kStages, k = i / C::kStages;
        const int b = i % C::kAcc, kb = i / C::kAcc;
        if (!tc::mbar_wait(&bar_full[s], k & 1, kWaitLimit) ||
            (kb > 0 && !tc::mbar_wait(&bar_tempty[b], (kb - 1) & 1, kWaitLimit))) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * 256);
        const uint32_t as = a0 + (uint32_t)s * kATile;
#pragma unroll
        for (int ks = 0; ks < kKSteps; ++ks) {
          const uint64_t ad = tc::smem_desc(as + ks * 4096, 2048, 128);
          const uint64_t bd = tc::smem_desc(w0 + ks * 32 * C::kN, 16 * C::kN, 128);
          if constexpr (L == 0) {
            tc::mma_bf16(d, ad, bd, tc::idesc_bf16_f32(128, 256), ks > 0 ? 1u : 0u);
          } else {
            tc::mma_e4m3(d, ad, bd, tc::idesc_e4m3_f32(128, 256), ks > 0 ? 1u : 0u);
            if constexpr (L == 2) {
              const uint64_t bd2 = tc::smem_desc(w0 + 256 * 16 + ks * 32 * C::kN, 16 * C::kN, 128);
              tc::mma_e4m3(d + 256, ad, bd2, tc::idesc_e4m3_f32(128, C::kN - 256),
                           ks > 0 ? 1u : 0u);
            }
          }
        }
        tc::mma_commit(&bar_empty[s]);
        tc::mma_commit(&bar_tfull[b]);
        last_b = b;
        last_kb = kb;
      }
      if (!ok) emu_fail(&s_fail, a.err);
      // the tensor memory is freed only after our MMAs are done
      if (last_b >= 0) tc::mbar_wait(&bar_tfull[last_b], last_kb & 1, kWaitLimit);
    }
    __syncwarp();
  } else {
    // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 ----
    const int ew = warp - kEpi0;
    const int q = warp & 3;
    const int r = q * 32 + lane;  // tile row of this thread
    if constexpr (L < 2) {
      const int c0 = (ew >> 2) * 64;  // column quarter
      const float hs = 0.5f * a.inv_out;
      for (int i = 0; i < my_tiles; ++i) {
        const int b = i % C::kAcc, kb = i / C::kAcc;
        if (!tc::mbar_wait(&bar_tfull[b], kb & 1, kWaitLimit)) {
          emu_fail(&s_fail, a.err);
          break;
        }
        tc::tc_fence_after();
        const long long t = (long long)blockIdx.x + (long long)i * gridDim.x;
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * 256);
        unsigned char *orow = a.out + t * (128 * 256) + r * 16;
        tc::tmem_stream16<4>(tb + (uint32_t)c0, [&](int k, float *v) {
          const int c = c0 + 16 * k;
          const float4 *s4 = reinterpret_cast<const float4 *>(sScale + c);
          const float4 *b4 = reinterpret_cast<const float4 *>(sBias + c);
#pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) {
            const float4 sc = s4[j4], bi = b4[j4];
            float *x = v + 4 * j4;
            x[0] = __fmaf_rn(x[0], sc.x, bi.x);
            x[1] = __fmaf_rn(x[1], sc.y, bi.y);
            x[2] = __fmaf_rn(x[2], sc.z, bi.z);
            x[3] = __fmaf_rn(x[3], sc.w, bi.w);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = gelu_scaled(v[j], hs);
          *reinterpret_cast<uint4 *>(orow + (c / 16) * 2048) = pack_e4m3_16(v);
        });
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_tempty[b]);
      }
    } else {
      const int h = ew >> 2;  // head (age class) of this warp
      const int col0 = h * kEmuHeadPitch;
      for (int i = 0; i < my_tiles; ++i) {
        if (!tc::mbar_wait(&bar_tfull[0], i & 1, kWaitLimit)) {
          emu_fail(&s_fail, a.err);
          break;
        }
        tc::tc_fence_after();
        const long long w = ((long long)blockIdx.x + (long long)i * gridDim.x) * 128 + r;
        const bool live = w < a.units;
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)col0;
        // pass 1: the logits (accumulator x a_scale w_scale + bias) times
        // log2 e, written back to the tensor memory, and their maximum
        float mx = -INFINITY;
        tc::tmem_stream16<kEmuHeadPitch / 16>(tb, [&](int k, float *x) {
          const int c = 16 * k;
          const float4 *s4 = reinterpret_cast<const float4 *>(sScale + col0 + c);
          const float4 *b4 = reinterpret_cast<const float4 *>(sBias + col0 + c);
#pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) {
            const float4 sc = s4[j4], bi = b4[j4];
            float *y = x + 4 * j4;
            y[0] = __fmaf_rn(y[0], sc.x, bi.x) * kLog2e;
            y[1] = __fmaf_rn(y[1], sc.y, bi.y) * kLog2e;
            y[2] = __fmaf_rn(y[2], sc.z, bi.z) * kLog2e;
            y[3] = __fmaf_rn(y[3], sc.w, bi.w) * kLog2e;
          }
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c + j < kBins) mx = fmaxf(mx, x[j]);
          tc::tmem_st16(tb + (uint32_t)c, x);
        });
        tc::tmem_wait_st();
        // pass 2: the 32 partial sums of 5 bins' softmax weights 2^(z - max z)
        float p[32];
#pragma unroll
        for (int l = 0; l < 32; ++l) p[l] = 0.0f;
        tc::tmem_stream16<kEmuHeadPitch / 16>(tb, [&](int k, float *x) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (16 * k + j < kBins) p[(16 * k + j) / 5] += ex2_fast(x[j] - mx);
        });
        // inclusive scan of the partial sums in the order of the warp's
        // shuffle scan in k_emu_sample (steps 1, 2, 4, 8, 16)
#pragma unroll
        for (int o = 1; o < 32; o <<= 1)
#pragma unroll
          for (int l = 31; l >= o; --l) p[l] += p[l - o];
        const float total = p[31];
        const long long rep = live ? w / a.n_nodes : 0;
        const long long node = live ? w - rep * a.n_nodes : 0;
        const U4 x4 = philox10(
            U4{0u, (uint32_t)node, (uint32_t)a.T, (SG_STREAM_EMU << 24) | (uint32_t)rep}, a.k0,
            a.k1);
        const uint32_t word = h == 0 ? x4.x : (h == 1 ? x4.y : x4.z);
        const float target = ((float)(word >> 8) + 0.5f) * (1.0f / 16777216.0f) * total;
        // the first partial range that reaches the target, then the bin in it
        int owner = 31;
        float incl_o = p[31];
#pragma unroll
        for (int l = 30; l >= 0; --l)
          if (p[l] >= target) {
            owner = l;
            incl_o = p[l];
          }
        // pass 3: the five values of that range, then their weights
        float xo[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        tc::tmem_stream16<kEmuHeadPitch / 16>(tb, [&](int k, float *x) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (16 * k + j < kBins && (16 * k + j) / 5 == owner) xo[(16 * k + j) % 5] = x[j];
        });
        // the range's own partial sum, added in the same order as in pass 2
        float e[5], part_o = 0.0f;
#pragma unroll
        for (int j = 0; j < 5; ++j) {
          e[j] = owner * 5 + j < kBins ? ex2_fast(xo[j] - mx) : 0.0f;
          part_o += e[j];
        }
        float acc = incl_o - part_o;
        int bin = min(owner * 5 + 4, kBins - 1);
#pragma unroll
        for (int j = 0; j < 5; ++j) {
          acc += e[j];
          if (acc >= target && owner * 5 + j < kBins) {
            bin = owner * 5 + j;
            break;
          }
        }
        if (live) {
          int32_t *o = a.delta + w * 4;
          if (a.flag[w]) {
            const int S = a.u[w * 6 + 2 * h], I = a.u[w * 6 + 2 * h + 1];
            int d = bin - kHalf;
            d = max(d, -I);
            d = min(d, S);
            o[h] = d;
            if (h == 0) o[3] = 1;
          } else if (h == 0) {
            o[3] = 0;
          }
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_tempty[0]);
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tc::tmem_dealloc(tmem, kEmuTmemCols);
}

// Weight image of the chain: row n of the image is row n of W (src_rows x
// Kb bytes, row-major), or with head_pad row 129 h + j for image row 144 h + j
// (j < 129); other image rows are zero.
__global__ void k_emu_image(const uint8_t *__restrict__ W, int src_rows, int Kb, int n_img,
                            int head_pad, uint8_t *img) {
  const int chunks = Kb / 16;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n_img * chunks;
       idx += gridDim.x * blockDim.x) {
    const int c = idx / n_img, n = idx - c * n_img;
    int src = n;
    if (head_pad) {
      const int h = n / kEmuHeadPitch, j = n - h * kEmuHeadPitch;
      src = j < kBins ? h * kBins + j : -1;
    }
    uint4 val = make_uint4(0u, 0u, 0u, 0u);
    if (src >= 0 && src < src_rows)
      val = *reinterpret_cast<const uint4 *>(W + (size_t)src * Kb + c * 16);
    *reinterpret_cast<uint4 *>(img + (size_t)idx * 16) = val;
  }
}

// Bias and weight scales of the output layer in the head-padded order.
__global__ void k_emu_head_vec(const float *__restrict__ b, const float *__restrict__ ws,
                               float *bimg, float *wimg) {
  for (int n = blockIdx.x * blockDim.x + threadIdx.x; n < kEmuHeadCols;
       n += gridDim.x * blockDim.x) {
    const int h = n / kEmuHeadPitch, j = n - h * kEmuHeadPitch;
    const bool in = j < kBins;
    bimg[n] = in ? b[h * kBins + j] : 0.0f;
    wimg[n] = in ? ws[h * kBins + j] : 0.0f;
  }
}

template <int L>
static void launch_emu_layer(const EmuChainArgs &a, int grid, cudaStream_t st) {
  const uint32_t smem = std::max(emu_layer_smem<L>(), kEmuMinSmem);
  static bool attr_set = false;  // guarded by the caller's lock
  if (!attr_set) {
    cudaFuncSetAttribute(k_emu_layer<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    attr_set = true;
  }
  k_emu_layer<L><<<grid, emu_layer_threads<L>(), smem, st>>>(a);
}

int emu_chain_images(const EmuChainWeights &cw, uint8_t *img, float *hvec, cudaStream_t st) {
  k_emu_image<<<16, 256, 0, st>>>(reinterpret_cast<const uint8_t *>(cw.W0), kEmuHidden, 32,
                                  kEmuHidden, 0, img + kEmuImgOff[0]);
  k_emu_image<<<64, 256, 0, st>>>(cw.W8[0], kEmuHidden, 256, kEmuHidden, 0, img + kEmuImgOff[1]);
  k_emu_image<<<64, 256, 0, st>>>(cw.W8[1], kEmuHidden, 256, kEmuHidden, 0, img + kEmuImgOff[2]);
  k_emu_image<<<64, 256, 0, st>>>(cw.W8[2], kEmuOut, 256, kEmuHeadCols, 1, img + kEmuImgOff[3]);
  k_emu_head_vec<<<2, 256, 0, st>>>(cw.b[3], cw.wscale[2], hvec, hvec + kEmuHeadCols);
  return cudaPeekAtLastError() == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

int emu_chain_day(const EmuChainWeights &cw, const uint8_t *img, const float *hvec,
                  uint8_t *act0, uint8_t *act1, const int32_t *u, const double *v,
                  const EmuParams &ep, long long units, int n_nodes, uint32_t k0, uint32_t k1,
                  int T, int32_t *flag, int32_t *delta, cudaStream_t st, int part) {
  if (units <= 0) return SG_OK;
  static std::mutex mu;
  static int n_sm = 0;
  std::lock_guard<std::mutex> lock(mu);
  if (!n_sm) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        n_sm <= 0) {
      cudaGetLastError();
      n_sm = 0;
      return SG_ERR_CUDA;
    }
  }
  int *err = nullptr;
  int rc = gemm_err_buf(&err);
  if (rc) return rc;
  const long long tiles = (units + 127) / 128;
  if (tiles > (1ll << 30)) return SG_ERR_ARG;
  const int grid = (int)std::min<long long>(tiles, n_sm);
  EmuChainArgs a{};
  a.u = u;
  a.v = v;
  a.flag = flag;
  a.delta = delta;
  a.ep = ep;
  a.units = units;
  a.n_nodes = n_nodes;
  a.k0 = k0;
  a.k1 = k1;
  a.T = T;
  a.n_tiles = (int)tiles;
  a.err = err;
  if (part == 0) {
    // layer 1: features -> E4M3 activations (act0), range flags
    a.W = img + kEmuImgOff[0];
    a.bias = cw.b[0];
    a.inv_out = 1.0f / cw.act_scale[0];
    a.out = act0;
    launch_emu_layer<0>(a, grid, st);
    return cudaPeekAtLastError() == cudaSuccess ? SG_OK : SG_ERR_CUDA;
  }
  // layers 2 and 3: act0 -> act1 -> act0
  for (int l = 1; l <= 2; ++l) {
    a.A = l == 1 ? act0 : act1;
    a.out = l == 1 ? act1 : act0;
    a.W = img + kEmuImgOff[l];
    a.bias = cw.b[l];
    a.wscale = cw.wscale[l - 1];
    a.a_scale = cw.act_scale[l - 1];
    a.inv_out = 1.0f / cw.act_scale[l];
    launch_emu_layer<1>(a, grid, st);
  }
  // layer 4 and sampling: act0 -> delta
  a.A = act0;
  a.out = nullptr;
  a.W = img + kEmuImgOff[3];
  a.bias = hvec;
  a.wscale = hvec + kEmuHeadCols;
  a.a_scale = cw.act_scale[2];
  launch_emu_layer<2>(a, grid, st);
  return cudaPeekAtLastError() == cudaSuccess ? SG_OK : SG_ERR_CUDA;
}

}  // namespace sg

static unsigned grid_n(long long n, int block) {
  return (unsigned)std::max<long long>(1, std::min<long long>(16384, (n + block - 1) / block));
}

static int finish(cudaStream_t st) {
  if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    cudaGetLastError();
    return SG_ERR_CUDA;
  }
  return SG_OK;
}

extern "C" int sg_mlp_ce_loss(const float *logits, int32_t ldl, const int32_t *targets,
                              int32_t B, void *dlogits, int32_t ldd, double *loss_sum,
                              void *stream) {
  if (B < 0 || ldl < 387 || ldd < 387 || !logits || !targets || !dlogits || !loss_sum)
    return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (B) k_ce_loss<<<grid_n((long long)B * 32, 256), 256, 0, st>>>(
      logits, ldl, targets, B, (__nv_bfloat16 *)dlogits, ldd, ldd, loss_sum);
  return finish(st);
}

extern "C" int sg_gelu_backward(const float *dpost, const float *pre, int64_t n, void *dpre,
                                void *stream) {
  if (n < 0 || (n && (!dpost || !pre || !dpre))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (n) k_gelu_bwd<<<grid_n(n, 256), 256, 0, st>>>(dpost, pre, n, (__nv_bfloat16 *)dpre);
  return finish(st);
}

extern "C" int sg_transpose_bf16(const void *src, int32_t rows, int32_t cols, void *dst,
                                 void *stream) {
  if (rows < 0 || cols < 0 || (rows && cols && (!src || !dst))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (rows && cols)
    k_transpose<<<dim3((cols + 31) / 32, (rows + 31) / 32), dim3(32, 8), 0, st>>>(
        (const __nv_bfloat16 *)src, rows, cols, (__nv_bfloat16 *)dst);
  return finish(st);
}

extern "C" int sg_colsum_bf16(const void *src, int32_t rows, int32_t cols, float *out,
                              void *stream) {
  if (rows < 0 || cols < 0 || (cols && (!src || !out))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (cols) k_colsum<<<(cols + 127) / 128, 128, 0, st>>>((const __nv_bfloat16 *)src, rows, cols, out);
  return finish(st);
}

namespace {

// Up to four transposes in one launch (blockIdx.z picks one), 64 x 64 tiles.
struct TransposeJobs {
  const __nv_bfloat16 *src[4];
  __nv_bfloat16 *dst[4];
  int rows[4], cols[4];
  bool tiled[4];  // dst in the tiled layout (cols x rows), else row-major
};
__global__ void __launch_bounds__(256) k_transpose_jobs(const TransposeJobs t) {
  __shared__ __nv_bfloat16 tile[64][66];
  const int z = blockIdx.z, rows = t.rows[z], cols = t.cols[z];
  const int r0 = blockIdx.x * 64, c0 = blockIdx.y * 64;
  if (r0 >= rows || c0 >= cols) return;
  // every dimension here is a multiple of 8: pairs along both, 4 bytes each
  const int tx = (threadIdx.x & 31) * 2, ty = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 64; i += 8) {
    const int r = i + ty;
    if (r0 + r < rows && c0 + tx < cols) {
      const __nv_bfloat162 v = *reinterpret_cast<const __nv_bfloat162 *>(
          t.src[z] + (long long)(r0 + r) * cols + c0 + tx);
      tile[r][tx] = v.x;
      tile[r][tx + 1] = v.y;
    }
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 64; i += 8) {
    const int c = i + ty;
    if (c0 + c < cols && r0 + tx < rows) {
      __nv_bfloat16 *d = t.tiled[z]
                             ? t.dst[z] + tiled_off(c0 + c, r0 + tx, cols) / 2
                             : t.dst[z] + (long long)(c0 + c) * rows + r0 + tx;
      *reinterpret_cast<__nv_bfloat162 *>(d) = __halves2bfloat162(tile[tx][c], tile[tx + 1][c]);
    }
  }
}

// Sums of the rows of up to four tiled matrices (n columns, padded with
// zeros), one block per row: the bias gradients from the deltas.
struct RowsumJobs {
  const __nv_bfloat16 *src[4];
  float *dst[4];
  int rows[4];
};
__global__ void __launch_bounds__(256) k_rowsum_jobs(const RowsumJobs t, int n) {
  __shared__ float s_sum[8];
  int r = blockIdx.x, z = 0;
  while (z < 3 && r >= t.rows[z]) r -= t.rows[z++];
  const unsigned char *x = reinterpret_cast<const unsigned char *>(t.src[z]);
  float sum = 0.0f;
  for (int k = threadIdx.x * 8; k < n; k += 256 * 8) {
    const uint4 v = *reinterpret_cast<const uint4 *>(x + tiled_off(r, k, t.rows[z]));
    const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&v);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 f = __bfloat1622float2(h[j]);
      sum += f.x;
      sum += f.y;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    float v = 0.0f;
    for (int i = 0; i < 8; ++i) v += s_sum[i];
    t.dst[z][r] = v;
  }
}

constexpr int kLayerOut[4] = {kEmuHidden, kEmuHidden, kEmuHidden, kEmuOut};
constexpr int kLayerIn[4] = {kEmuIn, kEmuHidden, kEmuHidden, kEmuHidden};

// Scratch of one gradient pass over B rows, every part 256-byte aligned.
struct GradScratch {
  float *logits, *pre[3];
  __nv_bfloat16 *act[3], *in_t[4], *delta[4], *delta_t[4], *w_t[4];
  size_t bytes;
  GradScratch(unsigned char *base, size_t B) {
    const size_t Bp = (B + 63) / 64 * 64;  // the tiled operands' padded K
    size_t off = 0;
    auto place = [&](size_t n) {
      unsigned char *p = base + off;
      off += (n + 255) & ~(size_t)255;
      return p;
    };
    logits = (float *)place(B * kEmuOut * 4);
    for (int l = 0; l < 3; ++l) {
      pre[l] = (float *)place(B * kEmuHidden * 4);
      act[l] = (__nv_bfloat16 *)place(B * kEmuHidden * 2);
    }
    for (int l = 0; l < 4; ++l) {
      in_t[l] = (__nv_bfloat16 *)place(Bp * kLayerIn[l] * 2);
      delta[l] = (__nv_bfloat16 *)place(B * kLayerOut[l] * 2);
      delta_t[l] = (__nv_bfloat16 *)place(Bp * kLayerOut[l] * 2);
      w_t[l] = (__nv_bfloat16 *)place((size_t)kLayerOut[l] * kLayerIn[l] * 2);
    }
    bytes = off;
  }
};

}  // namespace

extern "C" int sg_mlp_forward(const void *feat, int32_t B, const void *const *W,
                              const float *const *b, void *const *act, float *const *pre,
                              float *logits, void *stream) {
  if (B < 0 || !W || !b || !act || (B > 0 && (!feat || !logits))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const void *x = feat;
  for (int l = 0; l < 4; ++l) {
    GemmArgs g{};
    g.A = (const __nv_bfloat16 *)x;
    g.Bt = (const __nv_bfloat16 *)W[l];
    g.lda = g.ldb = g.K = kLayerIn[l];
    g.M = B;
    g.N = g.ldc32 = g.ldc16 = kLayerOut[l];
    g.bias = b[l];
    g.act = l < 3 ? 1 : 0;
    g.C32 = l == 3 ? logits : pre ? pre[l] : nullptr;
    g.C16 = l < 3 ? (__nv_bfloat16 *)act[l] : nullptr;
    const int rc = sg::gemm_bf16(g, st);
    if (rc) return rc;
    if (l < 3) x = act[l];
  }
  return sg::gemm_check(st);
}

extern "C" int sg_mlp_forward_fp8(const void *feat, int32_t B, const void *W0,
                                  const void *const *W8, const float *const *wscale,
                                  const float *act_scale, const float *const *b, void *buf_a,
                                  void *buf_b, float *logits, void *stream) {
  if (B < 0 || !W0 || !W8 || !wscale || !act_scale || !b ||
      (B > 0 && (!feat || !buf_a || !buf_b || !logits)))
    return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  uint8_t *bufs[2] = {(uint8_t *)buf_a, (uint8_t *)buf_b};
  for (int l = 0; l < 4; ++l) {
    GemmArgs g{};
    g.lda = g.ldb = g.K = kLayerIn[l];
    g.M = B;
    g.N = g.ldc32 = g.ldc8 = kLayerOut[l];
    g.bias = b[l];
    if (l == 0) {
      g.A = (const __nv_bfloat16 *)feat;
      g.Bt = (const __nv_bfloat16 *)W0;
    } else {
      g.f8 = 1;
      g.A8 = bufs[(l - 1) & 1];
      g.B8 = (const uint8_t *)W8[l - 1];
      g.a_scale = act_scale[l - 1];
      g.b_scale = wscale[l - 1];
    }
    if (l < 3) {
      g.act = 1;
      g.C8 = bufs[l & 1];
      g.c8_inv_scale = 1.0f / act_scale[l];
    } else {
      g.C32 = logits;
    }
    const int rc = sg::gemm_bf16(g, st);
    if (rc) return rc;
  }
  return sg::gemm_check(st);
}

extern "C" int sg_mlp_gradients_scratch(int32_t B, int64_t *bytes) {
  if (B < 0 || !bytes) return SG_ERR_ARG;
  *bytes = (int64_t)GradScratch(nullptr, (size_t)B).bytes;
  return SG_OK;
}

extern "C" int sg_mlp_gradients(const void *feat, const int32_t *targets, int32_t B,
                                const void *const *W, const float *const *b, float *const *dW,
                                float *const *db, double *loss_sum, void *scratch,
                                int64_t scratch_bytes, void *stream) {
  // the weight gradients contract over the batch: whole 16-byte chunks of it
  if (B < 8 || B % 8 != 0 || !feat || !targets || !W || !b || !dW || !db || !loss_sum ||
      !scratch || ((uintptr_t)scratch & 255) != 0 ||
      scratch_bytes < (int64_t)GradScratch(nullptr, (size_t)B).bytes)
    return SG_ERR_ARG;
  // feat and W are read in 16-byte pieces
  uintptr_t low = (uintptr_t)feat;
  for (int l = 0; l < 4; ++l) {
    if (!W[l] || !b[l] || !dW[l] || !db[l]) return SG_ERR_ARG;
    low |= (uintptr_t)W[l];
  }
  if (low & 15) return SG_ERR_ARG;
  GroupArgs q{};
  int rc = gemm_err_buf(&q.err);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const GradScratch s((unsigned char *)scratch, (size_t)B);
  cudaMemsetAsync(loss_sum, 0, sizeof(double), st);
  if (B % 64) {
    // the last step's rows past the batch contribute zeros
    const size_t step = (size_t)(B / 64) * 64;
    for (int l = 0; l < 4; ++l) {
      cudaMemsetAsync(s.in_t[l] + step * kLayerIn[l], 0, (size_t)128 * kLayerIn[l], st);
      cudaMemsetAsync(s.delta_t[l] + step * kLayerOut[l], 0, (size_t)128 * kLayerOut[l], st);
    }
  }
  // transposes of the features and of the weights that the backward pass reads
  TransposeJobs t{};
  t.src[0] = (const __nv_bfloat16 *)feat;
  t.dst[0] = s.in_t[0];
  t.rows[0] = B;
  t.cols[0] = kEmuIn;
  t.tiled[0] = true;
  for (int l = 1; l < 4; ++l) {
    t.src[l] = (const __nv_bfloat16 *)W[l];
    t.dst[l] = s.w_t[l];
    t.rows[l] = kLayerOut[l];
    t.cols[l] = kLayerIn[l];
  }
  k_transpose_jobs<<<dim3((unsigned)((std::max(B, kEmuOut) + 63) / 64), 4, 4), 256, 0, st>>>(t);
  auto gemm = [&](const __nv_bfloat16 *A, const __nv_bfloat16 *Bt, int M, int N, int K,
                  GemmArgs g) {
    g.A = A;
    g.lda = K;
    g.Bt = Bt;
    g.ldb = K;
    g.M = M;
    g.N = N;
    g.K = K;
    g.ldc32 = g.ldc16 = N;
    if (!rc) rc = sg::gemm_bf16(g, st);
  };
  // forward: pre-activations, activations and their transposes
  const __nv_bfloat16 *x = (const __nv_bfloat16 *)feat;
  for (int l = 0; l < 4; ++l) {
    GemmArgs g{};
    g.bias = b[l];
    if (l < 3) {
      g.act = 1;
      g.C32 = s.pre[l];
      g.C16 = s.act[l];
      g.C16T = s.in_t[l + 1];
    } else {
      g.C32 = s.logits;
    }
    gemm(x, (const __nv_bfloat16 *)W[l], B, kLayerOut[l], kLayerIn[l], g);
    if (l < 3) x = s.act[l];
  }
  k_ce_loss<<<(B + 7) / 8, 256, 0, st>>>(s.logits, kEmuOut, targets, B, s.delta[3], kEmuOut,
                                         kEmuOut, loss_sum);
  TransposeJobs d{};
  d.src[0] = s.delta[3];
  d.dst[0] = s.delta_t[3];
  d.rows[0] = B;
  d.cols[0] = kEmuOut;
  d.tiled[0] = true;
  k_transpose_jobs<<<dim3((B + 63) / 64, (kEmuOut + 63) / 64, 1), 256, 0, st>>>(d);
  for (int l = 3; l > 0; --l) {
    GemmArgs h{};
    h.C16 = s.delta[l - 1];
    h.C16T = s.delta_t[l - 1];
    h.bwd_pre = s.pre[l - 1];
    gemm(s.delta[l], s.w_t[l], B, kLayerIn[l], kLayerOut[l], h);
  }
  q.n = 4;
  q.K = B;
  for (int l = 0; l < 4; ++l) {
    q.A[l] = (const unsigned char *)s.delta_t[l];
    q.B[l] = (const unsigned char *)s.in_t[l];
    q.C[l] = dW[l];
    q.M[l] = kLayerOut[l];
    q.N[l] = kLayerIn[l];
  }
  if (!rc) launch_gemm_group(q, st);
  RowsumJobs r{};
  int rows = 0;
  for (int l = 0; l < 4; ++l) {
    r.src[l] = s.delta_t[l];
    r.dst[l] = db[l];
    r.rows[l] = kLayerOut[l];
    rows += kLayerOut[l];
  }
  k_rowsum_jobs<<<rows, 256, 0, st>>>(r, B);
  if (rc) {
    cudaStreamSynchronize(st);
    cudaGetLastError();
    return rc;
  }
  return sg::gemm_check(st);
}

extern "C" int sg_quant_fp8_rows(const float *W, int32_t rows, int32_t cols, void *W8,
                                 float *scale, void *stream) {
  if (rows < 0 || cols < 0 || (rows && (!W || !W8 || !scale))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (rows) k_quant_rows_fp8<<<rows, 256, 0, st>>>(W, rows, cols, (uint8_t *)W8, scale);
  return finish(st);
}

extern "C" int sg_quant_fp8_bf16(const void *x, int64_t n, float inv_scale, void *out8,
                                 void *stream) {
  if (n < 0 || (n && (!x || !out8))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (n) {
    const unsigned g = (unsigned)std::min<long long>(4096, (n + 255) / 256);
    k_quant_bf16_fp8<<<g, 256, 0, st>>>((const __nv_bfloat16 *)x, n, inv_scale, (uint8_t *)out8);
  }
  return finish(st);
}

extern "C" int sg_absmax_bf16(const void *x, int64_t n, float *out, void *stream) {
  if (n < 0 || !out || (n && !x)) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  cudaMemsetAsync(out, 0, sizeof(float), st);
  if (n) {
    const unsigned g = (unsigned)std::min<long long>(4096, (n + 255) / 256);
    k_absmax_bf16<<<g, 256, 0, st>>>((const __nv_bfloat16 *)x, n, out);
  }
  return finish(st);
}

extern "C" int sg_adam_step(float *params, const float *grads, float *m, float *v, int64_t n,
                            float lr, float beta1, float beta2, float eps, int32_t step,
                            void *params_bf16, void *stream) {
  if (n < 0 || step < 1 || (n && (!params || !grads || !m || !v))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
  if (n)
    k_adam<<<grid_n(n, 256), 256, 0, st>>>(params, grads, m, v, n, lr, beta1, beta2, eps, c1, c2,
                                           (__nv_bfloat16 *)params_bf16);
  return finish(st);
}

extern "C" int sg_emu_features(const int32_t *u, const double *v, int64_t units,
                               const double *gdata, int32_t max_herd, double phi_lo,
                               double phi_hi, double min_rate, void *feat, int32_t *flag,
                               void *stream) {
  if (units < 0 || !gdata || (units && (!u || !v || !feat || !flag))) return SG_ERR_ARG;
  EmuParams ep{};
  for (int i = 0; i < 11; ++i) ep.gdata[i] = gdata[i];
  ep.max_herd = max_herd;
  ep.phi_lo = phi_lo;
  ep.phi_hi = phi_hi;
  ep.min_rate = min_rate;
  cudaStream_t st = (cudaStream_t)stream;
  if (units)
    k_emu_features<<<grid_n(units, 256), 256, 0, st>>>(u, v, units, ep, (__nv_bfloat16 *)feat,
                                                       flag);
  return finish(st);
}

extern "C" int sg_emu_targets(const int32_t *u_before, const int32_t *u_after, int64_t units,
                              int32_t *targets, void *stream) {
  if (units < 0 || (units && (!u_before || !u_after || !targets))) return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (units) k_emu_targets<<<grid_n(units, 256), 256, 0, st>>>(u_before, u_after, units, targets);
  return finish(st);
}

extern "C" int sg_emu_sample(const float *logits, int32_t ldl, const int32_t *u,
                             const int32_t *flag, int64_t units, int32_t n_nodes, uint64_t seed,
                             int32_t day, int32_t *delta, void *stream) {
  if (units < 0 || n_nodes < 1 || ldl < 387 || (units && (!logits || !u || !flag || !delta)))
    return SG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (units)
    k_emu_sample<<<grid_n(units * 32, 256), 256, 0, st>>>(
        logits, ldl, u, flag, units, n_nodes, (uint32_t)seed, (uint32_t)(seed >> 32), day, delta);
  return finish(st);
}
