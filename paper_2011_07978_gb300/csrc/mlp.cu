// The learned cost predictor / surrogate network: a multilayer perceptron
// n_in -> 256 -> 256 -> 256 -> n_out with SiLU, trained and run on the GPU by
// the kernels below. Every contraction runs on the fifth-generation tensor
// cores (tcgen05.mma, kind::f16) in BF16 with the FP32 accumulator in tensor
// memory: inference as one whole-network kernel per 128-row tile, training
// layer by layer (FP32 master weights and activations are rounded to BF16
// when a tile is staged in shared memory), the loss, its gradient and SiLU' in
// the epilogues, the bias sums beside the staging of the weight gradients, all
// in FP32. Adam is an FP32 element kernel.
//
// Inputs of the network for one cell: x = [T/1000, ln p, Y_1..Y_nsp, ln dt];
// outputs: [ln(attempted steps), dT, dY_1..dY_nsp]. Both are normalised by
// stored means and standard deviations.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/dlbchem.h"
#include "dlb_common.cuh"
#include "dlb_ctx.h"

namespace dlb {

// SiLU z sigma(z) through sigma(z) = (1 + tanh(z/2)) / 2, with the hardware
// tanh on a pair of half-precision values (tanh.approx.f16x2: one
// special-function operation for two activations instead of an exponential
// and a reciprocal for each; the fused forward's epilogue is bound by that
// unit). z/2 rounded to FP16 and the approximate tanh put an error of order
// 1e-3 into sigma, below the BF16 rounding the activations get next; |z/2|
// beyond the FP16 range gives tanh = +-1, the limits of sigma. Training uses
// the same sigma, so the layer-by-layer and fused passes agree.
__device__ __forceinline__ float2 tanh2_half(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  uint32_t y;
  asm("tanh.approx.f16x2 %0, %1;" : "=r"(y) : "r"(*reinterpret_cast<const uint32_t*>(&h)));
  return __half22float2(*reinterpret_cast<const __half2*>(&y));
}
__device__ __forceinline__ float2 silu2_f(float z0, float z1) {
  const float h0 = 0.5f * z0, h1 = 0.5f * z1;
  const float2 t = tanh2_half(h0, h1);
  return make_float2(fmaf(h0, t.x, h0), fmaf(h1, t.y, h1));
}
__device__ __forceinline__ float silu_f(float z) { return silu2_f(z, 0.0f).x; }
// d/dz z sigma(z) = sigma (1 + z (1 - sigma)), with the same sigma
__device__ __forceinline__ float dsilu_f(float z) {
  const float s = fmaf(0.5f, tanh2_half(0.5f * z, 0.0f).x, 0.5f);
  return s * fmaf(z, 1.0f - s, 1.0f);
}

// C[M x N] = A[M x K] B[K x N] with an epilogue, on the fifth-generation tensor
// cores: BF16 operands (FP32 rounded while staged) in shared memory in the
// canonical K-major layout without swizzle (8 x 8 core matrices of 128 B, the
// K-groups of a row group contiguous), FP32 accumulator in tensor memory. One
// CTA computes a tile: eight warps stage k-tiles of 64 into a ring of four
// buffers, one thread of a ninth issues the MMAs of a k-tile (K = 16 each) as
// its buffer fills and commits them to the buffer's release, and the eight
// warps read the accumulator from tensor memory for the epilogue. Waits are on
// mbarriers and bounded; one that gives up stops the others, sets *status,
// writes NaN and still frees the tensor memory. (With a CTA barrier per k-tile
// the staging warps waited for each other and for the issue: 2,070 cycles a
// k-tile of the weight gradients.)
constexpr int kTM = 128, kTN = 64, kTK = 64;
constexpr int kGemmThreads = 256;    // staging and epilogue; a warp of its own issues the MMAs
constexpr int kGemmStages = 4;       // operand buffers
constexpr int kWaitLimit = 1 << 24;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

// shared-memory matrix descriptor: start, leading-dimension byte offset (between
// core matrices along K), stride byte offset (between 8-row groups), version 1
// (the sm_100 family), no swizzle
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((addr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}

// Staging goes through registers, 16 bytes per load and store, with the loads of
// the next two k-tiles in flight while the tensor cores work on this one.
// An operand's values of consecutive k are adjacent (KC: p[row ld + k]): a thread
// takes chunks of one row and eight k; or those of consecutive rows are
// (p[k ld + row]): a thread takes four rows and eight k, eight loads for four
// chunks (with one row per thread the loads and their addresses were 500
// instructions per thread and tile, and the weight gradients of 4,096 rows took
// 112 us instead of 62). Row groups lie kRowGroup bytes apart, 16 more than
// their eight core matrices, so that a warp's stores of every fourth row hit
// all banks.
constexpr int kRowGroup = (kTK / 8) * 128 + 16;
__host__ __device__ constexpr int tile_bytes(int nt) { return kGemmStages * ((kTM + nt) / 8) * kRowGroup; }   // dynamic shared memory
template <bool KC, int ROWS>
struct TileSource {
  static constexpr int kItems = KC ? ROWS * 8 : ROWS * 2;                       // chunks, or groups of four rows
  static constexpr int kPer = (kItems + kGemmThreads - 1) / kGemmThreads;       // per thread
  static constexpr int kRegs = kPer * (KC ? 8 : 32);
  const float* p;
  int ld, rows, kend;   // rows and k beyond these are zero
  bool vec;             // 16-byte loads
  __device__ TileSource(const float* p_, int ld_, int rows_, int kend_)
      : p(p_), ld(ld_), rows(rows_), kend(kend_), vec((ld_ & 3) == 0 && (reinterpret_cast<uintptr_t>(p_) & 15) == 0) {}
  // item e of a tile: its (first) row and first k
  static __device__ __forceinline__ void place(int e, int& row, int& k) {
    if (KC) { row = (e & 7) + ((e >> 6) << 3); k = ((e >> 3) & 7) * 8; }
    else { row = (e % (ROWS / 4)) * 4; k = (e / (ROWS / 4)) * 8; }
  }
  // the tile at (r0, k0) into v[kRegs]
  __device__ __forceinline__ void fetch(int r0, int k0, float* v) const {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = threadIdx.x + kGemmThreads * i;
      if (kItems % kGemmThreads != 0 && e >= kItems) break;
      int row, k;
      place(e, row, k);
      row += r0;
      k += k0;
      if (KC) {
        float* x = v + 8 * i;
        const float* q = p + int64_t(row) * ld + k;
        if (vec && row < rows && k + 8 <= kend) {
          *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(q);
          *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(q + 4);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) x[j] = row < rows && k + j < kend ? q[j] : 0.0f;
        }
      } else {
        float* x = v + 32 * i;   // four rows of eight k
        const float* q = p + int64_t(k) * ld + row;
        if (vec && row + 4 <= rows && k + 8 <= kend) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 f = *reinterpret_cast<const float4*>(q);
            x[j] = f.x; x[8 + j] = f.y; x[16 + j] = f.z; x[24 + j] = f.w;
            q += ld;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
#pragma unroll
            for (int r = 0; r < 4; ++r) x[8 * r + j] = row + r < rows && k + j < kend ? q[r] : 0.0f;
            q += ld;
          }
        }
      }
    }
  }
  // v as BF16 into the operand tile; with sums, sums[r] += the r-th row's FP32 values
  __device__ __forceinline__ static void store(unsigned char* base, const float* v, float* sums);
};

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);   // a in the low half (lower k)
  return *reinterpret_cast<const uint32_t*>(&h);
}

template <bool KC, int ROWS>
__device__ __forceinline__ void TileSource<KC, ROWS>::store(unsigned char* base, const float* v, float* sums) {
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int e = threadIdx.x + kGemmThreads * i;
    if (kItems % kGemmThreads != 0 && e >= kItems) break;
    int row, k;
    place(e, row, k);
#pragma unroll
    for (int r = 0; r < (KC ? 1 : 4); ++r) {
      const float* x = v + (KC ? 8 * i : 32 * i + 8 * r);
      *reinterpret_cast<uint4*>(base + ((row + r) >> 3) * kRowGroup + (k >> 3) * 128 + ((row + r) & 7) * 16) =
          make_uint4(pack_bf16x2(x[0], x[1]), pack_bf16x2(x[2], x[3]), pack_bf16x2(x[4], x[5]), pack_bf16x2(x[6], x[7]));
      if (sums) sums[r] += ((x[0] + x[1]) + (x[2] + x[3])) + ((x[4] + x[5]) + (x[6] + x[7]));
    }
  }
}

// The 128 x NT tile at (m0, n0): epi(gm, gn, v, nv) takes nv <= 16 consecutive
// columns of one row. With BSUM, bsum[n] (NT floats of shared memory) receives
// the sums over k of B's FP32 values.
template <int NT, bool BSUM, bool AKC, bool BKC, class Epi>
__device__ __forceinline__ void gemm_tile(const TileSource<AKC, kTM>& A, const TileSource<BKC, NT>& B, int m0, int n0,
                                          float* bsum, int* __restrict__ status, Epi&& epi) {
  using SA = TileSource<AKC, kTM>;
  using SB = TileSource<BKC, NT>;
  constexpr int kBuf = tile_bytes(NT) / kGemmStages;
  static_assert(!BSUM || (!BKC && SB::kPer == 1), "one group of four rows per thread");
  extern __shared__ __align__(1024) unsigned char sop[];   // the ring of operand buffers, tile_bytes(NT)
  __shared__ __align__(8) unsigned long long full[kGemmStages], empty[kGemmStages], done;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int b = 0; b < kGemmStages; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[b])), "r"(kGemmThreads / 32) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[b])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&done)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(uint32_t(NT)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int K = A.kend, ntiles = (K + kTK - 1) / kTK;
  float ra[2][SA::kRegs], rb[2][SB::kRegs];
  auto fetch = [&](int set, int k0) {
    A.fetch(m0, k0, ra[set]);
    B.fetch(n0, k0, rb[set]);
  };
  const bool stager = warp < kGemmThreads / 32;
  if (stager) {
    fetch(0, 0);
    if (ntiles > 1) fetch(1, kTK);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  auto wait = [&](unsigned long long* bar, int use) {   // the use-th phase (bounded)
    uint32_t ok = 0;
    for (int it = 0; it < kWaitLimit && !ok; ++it)
      asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                   : "=r"(ok) : "r"(smem_u32(bar)), "r"(uint32_t(use) & 1u) : "memory");
    return ok != 0;
  };
  bool ok = true;
  float sums[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (stager) {
    for (int t0 = 0; t0 < ntiles && ok; t0 += 2) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int t = t0 + b, st = t % kGemmStages;
        if (t < ntiles && ok) {
          unsigned char* sA = sop + st * kBuf;
          if (t >= kGemmStages) ok = wait(&empty[st], t / kGemmStages - 1);
          SA::store(sA, ra[b], nullptr);
          SB::store(sA + kTM / 8 * kRowGroup, rb[b], BSUM ? sums : nullptr);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy stores -> tensor cores
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&full[st])) : "memory");
          if (t + 2 < ntiles) fetch(b, (t + 2) * kTK);
        }
      }
    }
  } else if (lane == 0) {
    // kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, N and M
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(NT >> 3) << 17) | (uint32_t(kTM >> 4) << 24);
    for (int t = 0; t < ntiles; ++t) {
      const int st = t % kGemmStages;
      if (!wait(&full[st], t / kGemmStages)) { ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sA = smem_u32(sop + st * kBuf), sB = sA + kTM / 8 * kRowGroup;
#pragma unroll
      for (int kk = 0; kk < kTK / 16; ++kk) {
        const uint64_t ad = umma_desc(sA + kk * 256, 128, kRowGroup);
        const uint64_t bd = umma_desc(sB + kk * 256, 128, kRowGroup);
        const uint32_t acc = (t > 0 || kk > 0) ? 1u : 0u;
        asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                     "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem),
                     "l"(ad), "l"(bd), "r"(idesc), "r"(acc) : "memory");
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                       smem_u32(&empty[st]))
                   : "memory");
    }
    // covers every MMA issued, also after a wait that gave up
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&done))
                 : "memory");
  }
  __syncwarp();   // the issuer's other lanes wait here, not in a poll beside it
  ok = wait(&done, 0) && ok;
  ok = __syncthreads_and(ok);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (!ok && tid == 0 && status) atomicExch(status, 1);
  if (BSUM) {   // thread t < NT / 4 * 8 has rows 4 (t % (NT / 4)) .. + 3 of k-group t / (NT / 4)
    float* part = reinterpret_cast<float*>(sop);   // the operand tiles are done with
    if (tid < SB::kItems) *reinterpret_cast<float4*>(part + 4 * tid) = make_float4(sums[0], sums[1], sums[2], sums[3]);
    __syncthreads();
    if (tid < NT) {
      float sum = 0.0f;
      for (int g = 0; g < kTK / 8; ++g) sum += part[g * NT + tid];
      bsum[tid] = sum;
    }
    __syncthreads();
  }
  // epilogue: warps w and w + 4 hold rows 32 (w % 4) .. + 31 of the tile, half of the columns each, 16 per load
  const int gm = m0 + 32 * (warp & 3) + lane;
  for (int c0 = (NT / 2) * (warp >> 2), c1 = stager ? c0 + NT / 2 : 0; c0 < c1; c0 += 16) {
    uint32_t r[16];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(tmem + (uint32_t(32 * (warp & 3)) << 16) + uint32_t(c0)));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int nv = min(16, B.rows - (n0 + c0));
    if (gm < A.rows && nv > 0) {
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = ok ? __uint_as_float(r[j]) : __int_as_float(0x7fc00000);
      epi(gm, n0 + c0, v, nv);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(uint32_t(NT)) : "memory");
}

// nv <= 16 consecutive values, 16 bytes at a time where the row allows it
__device__ __forceinline__ void store_row(float* dst, const float* v, int nv) {
  if (nv == 16 && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
    for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(dst + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (j < nv) dst[j] = v[j];
  }
}

// One layer forward: C = act(in W + bias), the pre-activations to Z if given.
// With a target (the output layer of a training step) C instead receives the
// gradient of the MSE, 2 (out - y) scale, and *loss the sum of scale (out - y)^2.
__global__ void __launch_bounds__(kGemmThreads + 32) layer_forward_kernel(int M, int N, int K, const float* __restrict__ in,
                                                            const float* __restrict__ W, float* __restrict__ C,
                                                            const float* __restrict__ bias, float* __restrict__ Z,
                                                            int act, const float* __restrict__ target, float scale,
                                                            float* __restrict__ loss, int* __restrict__ status) {
  float s = 0.0f;
  gemm_tile<kTN, false>(TileSource<true, kTM>(in, K, M, K), TileSource<false, kTN>(W, N, N, K), int(blockIdx.y) * kTM,
                        int(blockIdx.x) * kTN, nullptr, status, [&](int gm, int gn, float* v, int nv) {
              const int64_t at = int64_t(gm) * N + gn;
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] += j < nv ? bias[gn + j] : 0.0f;
              if (Z) store_row(Z + at, v, nv);
              if (act) {
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] = silu_f(v[j]);
              }
              if (target) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  const float d = j < nv ? v[j] - target[at + j] : 0.0f;
                  s += d * d;
                  v[j] = 2.0f * d * scale;
                }
              }
              store_row(C + at, v, nv);
            });
  if (target && loss) {
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(loss, s * scale);
  }
}

// One layer backward: Z <- (dZ_next W^T) silu'(Z), in place (M rows, N = the
// layer's width, K = the next layer's).
__global__ void __launch_bounds__(kGemmThreads + 32) layer_backward_kernel(int M, int N, int K, const float* __restrict__ dZn,
                                                             const float* __restrict__ W, float* __restrict__ Z,
                                                             int* __restrict__ status) {
  gemm_tile<kTN, false>(TileSource<true, kTM>(dZn, K, M, K), TileSource<true, kTN>(W, K, N, K), int(blockIdx.y) * kTM,
                        int(blockIdx.x) * kTN, nullptr, status, [&](int gm, int gn, float* v, int nv) {
              float* z = Z + int64_t(gm) * N + gn;
#pragma unroll
              for (int j = 0; j < 16; ++j) v[j] *= j < nv ? dsilu_f(z[j]) : 0.0f;
              store_row(z, v, nv);
            });
}

// Weight and bias gradients of every layer in one launch: block x is a tile of
// one layer's dW = in^T dZ (M = fan-in, N = fan-out, K = batch). The contraction
// is long and the output small (42 tiles of 128 x 32 for the 13-256-256-256-12
// network), so a tile's k-tiles in sequence are what it takes; splitting the
// batch over CTAs would be faster but sum in another order (8.6e-5 relative
// from the sequential FP32 accumulation at 4,096 rows).
struct GradLayer {
  const float *in, *dz;
  int fi, fo, tile0;   // first tile; tiles run over n, then m
  int64_t off;         // of the layer's parameters [W b]
};
constexpr int kGradTN = 32;
struct GradArgs {
  int nl, B;
  float* grad;
  GradLayer layer[8];
};
__global__ void __launch_bounds__(kGemmThreads + 32) weight_grad_kernel(const GradArgs a, int* __restrict__ status) {
  __shared__ float bsum[kGradTN];
  int l = 0;
  while (l + 1 < a.nl && int(blockIdx.x) >= a.layer[l + 1].tile0) ++l;
  const GradLayer& g = a.layer[l];
  const int nt = (g.fo + kGradTN - 1) / kGradTN, t = int(blockIdx.x) - g.tile0;
  const int m0 = t / nt * kTM, n0 = t % nt * kGradTN;
  float* out = a.grad + g.off;
  gemm_tile<kGradTN, true>(TileSource<false, kTM>(g.in, g.fi, g.fi, a.B), TileSource<false, kGradTN>(g.dz, g.fo, g.fo, a.B), m0, n0,
                           bsum, status,
                           [&](int gm, int gn, float* v, int nv) { store_row(out + int64_t(gm) * g.fo + gn, v, nv); });
  if (m0 == 0 && int(threadIdx.x) < kGradTN && n0 + int(threadIdx.x) < g.fo)
    out[int64_t(g.fi) * g.fo + n0 + threadIdx.x] = bsum[threadIdx.x];
}

// ---------------------------------------------------------------------------
// Whole-network forward pass for inference: one persistent CTA per SM, three
// roles in warps of their own. The weights, packed once into BF16 k-tiles of
// 64 (four MMAs of K = 16 each) in exactly the shared-memory layout the MMA
// reads, stream through a two-deep ring of 32 KB buffers filled by bulk
// copies (cp.async.bulk, the TMA engine, completing on mbarriers) from a
// producer warp; an output layer of at most 16 KB is copied once and stays. An MMA warp issues tcgen05.mma (kind::f16, BF16 operands,
// FP32 accumulator in tensor memory) and commits each k-tile to free its
// buffer. Eight epilogue warps (two per tensor-memory lane quarter, 32 rows
// each, alternate 16-column chunks) read the accumulator, add the bias, apply
// SiLU and write the activations back to shared memory as BF16: the next
// layer's A operand. Activations never leave shared memory; only the network
// input and output cross HBM. The CTA keeps two 128-row tiles in flight, each
// with its own activation tile and accumulator, and alternates them layer by
// layer, so the epilogue of one tile runs while the tensor cores work on the
// other. Arithmetic per element is that of the layered path above: BF16
// operands, FP32 accumulation over k-tiles of 64, FP32 bias and SiLU,
// activations rounded to BF16 as the next layer's operand. Supported shapes:
// hidden widths multiples of 64 up to 256, n_in and n_out up to 256, at most
// kFusedMaxLayers layers.
// ---------------------------------------------------------------------------
constexpr int kFusedMaxLayers = 8;
constexpr int kFusedMaxN = 256;
constexpr int kFK = 64;                                       // k-tile of the weight stream
constexpr int kFusedStages = 2;                               // weight ring depth
constexpr int kFusedSmemH = kTM * kFusedMaxN * 2;             // 64 KB per activation tile
constexpr int kFusedSmemW = kFusedMaxN * kFK * 2;             // 32 KB per weight buffer
constexpr int kFusedBias = kFusedMaxLayers * kFusedMaxN * 4;  // every layer's bias
// the output layer's packed weights stay in shared memory when they fit here
// (a narrow output: they then skip the ring and its per-k-tile round trips)
constexpr int kFusedResident = 16 * 1024;
constexpr int kFusedSmem = 2 * kFusedSmemH + kFusedStages * kFusedSmemW + kFusedBias + kFusedResident + 1024;
constexpr int kFusedEpiWarps = 8;                             // two per tensor-memory lane quarter
constexpr int kFusedThreads = 32 * (kFusedEpiWarps + 2);      // + producer warp + MMA warp

struct FusedNet {
  int nl;                                       // layers
  int fi[kFusedMaxLayers], fo[kFusedMaxLayers];
  int kp[kFusedMaxLayers], np[kFusedMaxLayers];  // fan-in padded to kFK, fan-out padded to 16
  int64_t woff[kFusedMaxLayers];                // byte offset of the layer's packed weights
  const float* bias[kFusedMaxLayers];
  const unsigned char* wpk;
  uint32_t res_bytes;                           // output layer resident in shared memory (0: streamed)
};

// byte offset of (row, k) in a tile of rows x kext BF16 values (kext a multiple of 8)
__device__ __forceinline__ int core_off(int row, int k, int kext) {
  return ((row >> 3) * (kext >> 3) + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2;
}

// Layer weights W [fi][fo] (FP32, row-major) as BF16 k-tiles for the fused
// pass: k-tile t holds rows n < np and k in [kFK t, kFK t + kFK) of W^T in
// core matrices (the B operand, K-major), zero outside W.
__global__ void pack_weights_kernel(int fi, int fo, int kp, int np, const float* __restrict__ W,
                                    unsigned char* __restrict__ dst) {
  const int64_t total = int64_t(kp) * np;
  for (int64_t e = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; e < total; e += int64_t(gridDim.x) * blockDim.x) {
    const int n = int(e % np), k = int(e / np);
    const float v = (n < fo && k < fi) ? W[int64_t(k) * fo + n] : 0.0f;
    const int kt = k / kFK;
    *reinterpret_cast<__nv_bfloat16*>(dst + int64_t(kt) * np * kFK * 2 + core_off(n, k - kt * kFK, kFK)) =
        __float2bfloat16_rn(v);
  }
}

// bounded mbarrier wait on the phase of the given parity; true once it completed
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  for (int it = 0; it < kWaitLimit && !done; ++it)
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// Work order of one CTA: its row tiles in pairs; within a pair, unit
// (tile, layer) in the order (t0, 0), (t1, 0), (t0, 1), (t1, 1), ...; tile j of
// the pair uses slot j (activation tile and accumulator). All three roles walk
// this order.
struct FusedOrder {
  int64_t ntiles, first, stride, mine;   // row tiles, this CTA's first, grid stride, count
  int nl;
  // unit u -> (local tile index, layer); units per pair = nl * tiles in the pair
  __device__ void unit(int64_t u, int64_t& lt, int& l) const {
    const int64_t per_pair = 2 * int64_t(nl);
    const int64_t pair = u / per_pair;
    int64_t r = u - pair * per_pair;
    const int64_t in_pair = mine - 2 * pair >= 2 ? 2 : 1;
    l = int(r / in_pair);
    lt = 2 * pair + (r - int64_t(l) * in_pair);
  }
  __device__ int64_t units() const { return mine * nl; }
};

__global__ void __launch_bounds__(kFusedThreads, 1) mlp_fused_forward_kernel(int64_t B, const float* __restrict__ X,
                                                                             float* __restrict__ out,
                                                                             const FusedNet net,
                                                                             int* __restrict__ status) {
  extern __shared__ unsigned char fused_smem_raw[];
  unsigned char* sH0 =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(fused_smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sW = sH0 + 2 * kFusedSmemH;                               // kFusedStages buffers
  float* sbias = reinterpret_cast<float*>(sW + kFusedStages * kFusedSmemW);  // [layer][kFusedMaxN]
  unsigned char* sR = reinterpret_cast<unsigned char*>(sbias) + kFusedBias;    // resident output layer
  __shared__ __align__(8) unsigned long long full[kFusedStages], empty[kFusedStages], acc_full[2], h_ready[2], res_bar, drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  FusedOrder ord;
  ord.ntiles = (B + kTM - 1) / kTM;
  ord.first = blockIdx.x;
  ord.stride = gridDim.x;
  ord.mine = ord.first < ord.ntiles ? (ord.ntiles - 1 - ord.first) / ord.stride + 1 : 0;
  ord.nl = net.nl;
  const int64_t nunits = ord.units();
  if (tid == 0) {
    for (int b = 0; b < kFusedStages; ++b) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[b])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[b])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&res_bar)) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&drain_bar)) : "memory");
    for (int j = 0; j < 2; ++j) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&acc_full[j])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&h_ready[j])), "r"(kFusedEpiWarps)
                   : "memory");
    }
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int l = 0; l < net.nl; ++l)
    for (int n = tid; n < net.np[l]; n += kFusedThreads) sbias[l * kFusedMaxN + n] = n < net.fo[l] ? net.bias[l][n] : 0.0f;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(uint32_t(2 * kFusedMaxN)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  // a wait that gives up stops every role: the others skip their later waits
  auto wait = [&](unsigned long long* bar, uint32_t parity) {
    if (abort_flag) return false;
    if (mbar_wait(smem_u32(bar), parity)) return true;
    abort_flag = 1;
    return false;
  };
  if (warp == kFusedEpiWarps) {
    // producer: weight k-tile g of the stream into buffer g % kFusedStages
    if (lane == 0) {
      int64_t g = 0;
      for (int64_t u = 0; u < nunits && !abort_flag; ++u) {
        int64_t lt;
        int l;
        ord.unit(u, lt, l);
        if (l + 1 == net.nl && net.res_bytes) continue;   // resident: not streamed
        const uint32_t bytes = uint32_t(net.np[l]) * kFK * 2;
        for (int kt = 0; kt < net.kp[l] / kFK; ++kt, ++g) {
          const int st = int(g % kFusedStages);
          if (g >= kFusedStages && !wait(&empty[st], uint32_t(g / kFusedStages - 1) & 1u)) break;
          const uint32_t bar = smem_u32(&full[st]);
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
          asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                           smem_u32(sW + st * kFusedSmemW)),
                       "l"(net.wpk + net.woff[l] + size_t(kt) * bytes), "r"(bytes), "r"(bar)
                       : "memory");
        }
      }
      // on a give-up, let the copies in flight land before the CTA leaves
      if (abort_flag && g > 0) mbar_wait(smem_u32(&full[(g - 1) % kFusedStages]), uint32_t((g - 1) / kFusedStages) & 1u);
    }
  } else if (warp == kFusedEpiWarps + 1) {
    // MMA issuer
    if (lane == 0) {
      int64_t g = 0, done_units[2] = {0, 0};
      bool res_ready = false;
      if (net.res_bytes && nunits > 0) {   // the output layer's weights, once
        const uint32_t bar = smem_u32(&res_bar);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(net.res_bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(sR)),
                     "l"(net.wpk + net.woff[net.nl - 1]), "r"(net.res_bytes), "r"(bar)
                     : "memory");
      }
      for (int64_t u = 0; u < nunits && !abort_flag; ++u) {
        int64_t lt;
        int l;
        ord.unit(u, lt, l);
        const int slot = int(lt & 1);
        const int kp = net.kp[l], np = net.np[l];
        // the slot's activations are written and its accumulator drained
        if (!wait(&h_ready[slot], uint32_t(done_units[slot]) & 1u)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t idesc =
            (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(np >> 3) << 17) | (uint32_t(kTM >> 4) << 24);
        const uint32_t hbase = smem_u32(sH0 + slot * kFusedSmemH);
        const uint32_t dtm = tmem + uint32_t(slot * kFusedMaxN);
        bool ok = true;
        if (l + 1 == net.nl && net.res_bytes) {
          // resident output layer: no ring, one commit for the whole unit
          if (!res_ready) {
            if (!wait(&res_bar, 0u)) break;
            res_ready = true;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          for (int kt = 0; kt < kp / kFK; ++kt) {
#pragma unroll
            for (int kk = 0; kk < kFK / 16; ++kk) {
              const uint64_t ad = umma_desc(hbase + uint32_t(kt * (kFK / 8) + kk * 2) * 128u, 128, uint32_t(kp) * 16u);
              const uint64_t bd = umma_desc(smem_u32(sR) + uint32_t(kt) * uint32_t(np) * (kFK * 2) + uint32_t(kk) * 256u,
                                            128, (kFK / 8) * 128);
              const uint32_t acc = (kt > 0 || kk > 0) ? 1u : 0u;
              asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                           "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtm),
                           "l"(ad), "l"(bd), "r"(idesc), "r"(acc) : "memory");
            }
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(&acc_full[slot]))
                       : "memory");
          ++done_units[slot];
          continue;
        }
        for (int kt = 0; kt < kp / kFK; ++kt, ++g) {
          const int st = int(g % kFusedStages);
          if (!wait(&full[st], uint32_t(g / kFusedStages) & 1u)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int kk = 0; kk < kFK / 16; ++kk) {
            const uint64_t ad = umma_desc(hbase + uint32_t(kt * (kFK / 8) + kk * 2) * 128u, 128, uint32_t(kp) * 16u);
            const uint64_t bd = umma_desc(smem_u32(sW + st * kFusedSmemW) + uint32_t(kk) * 256u, 128, (kFK / 8) * 128);
            const uint32_t acc = (kt > 0 || kk > 0) ? 1u : 0u;
            asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                         "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtm),
                         "l"(ad), "l"(bd), "r"(idesc), "r"(acc) : "memory");
          }
          // the buffer is free once these MMAs complete
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_u32(&empty[st]))
                       : "memory");
        }
        if (!ok) break;
        // the unit's accumulator is complete when its MMAs are
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&acc_full[slot]))
                     : "memory");
        ++done_units[slot];
      }
      // on a give-up, let the copy and the MMAs in flight finish before tensor
      // memory is freed: one more commit covers every MMA issued so far
      if (abort_flag) {
        if (net.res_bytes && nunits > 0 && !res_ready) mbar_wait(smem_u32(&res_bar), 0u);
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(&drain_bar))
                     : "memory");
        mbar_wait(smem_u32(&drain_bar), 0u);
      }
    }
  } else {
    // epilogue warps: warp w reads tensor-memory lane quarter w % 4 (rows
    // 32 (w % 4) + lane of each tile) and the 16-column chunks of parity w / 4
    const int quarter = warp & 3, half = warp >> 2;
    const int row = 32 * quarter + lane;
    auto stage_input = [&](int64_t lt) {
      const int slot = int(lt & 1);
      unsigned char* sH = sH0 + slot * kFusedSmemH;
      const int64_t r0 = (ord.first + lt * ord.stride) * kTM;
      const int kp = net.kp[0], fi = net.fi[0];
      const float* x = X + (r0 + row) * fi;
      const bool in = r0 + row < B;
      for (int k0 = 8 * half; k0 < kp; k0 += 16) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (in && k0 + j < fi) ? x[k0 + j] : 0.0f;
        *reinterpret_cast<uint4*>(sH + core_off(row, k0, kp)) = make_uint4(
            pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&h_ready[slot])) : "memory");
    };
    if (ord.mine > 0) stage_input(0);
    if (ord.mine > 1) stage_input(1);
    int64_t seen[2] = {0, 0};
    for (int64_t u = 0; u < nunits; ++u) {
      int64_t lt;
      int l;
      ord.unit(u, lt, l);
      const int slot = int(lt & 1);
      // warp-uniform, since the tensor-memory loads below are warp-collective
      const bool ok = __all_sync(0xffffffffu, wait(&acc_full[slot], uint32_t(seen[slot]) & 1u));
      ++seen[slot];
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int np = net.np[l], fo = net.fo[l];
      const bool last = l + 1 == net.nl;
      const float* bias = sbias + l * kFusedMaxN;
      const int64_t gr = (ord.first + lt * ord.stride) * kTM + row;
      unsigned char* sH = sH0 + slot * kFusedSmemH;
      const int kpn = last ? 0 : net.kp[l + 1];
      if (ok) {
        // this warp's 16-column chunks c0 = 16 half + 32 i; four tensor-memory
        // loads in flight per wait
        const int nch = (np - 16 * half + 31) / 32;
        for (int i0 = 0; i0 < nch; i0 += 4) {
          uint32_t r[4][16];
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (i0 + q < nch)
              tmem_ld16(tmem + (uint32_t(32 * quarter) << 16) + uint32_t(slot * kFusedMaxN + 16 * half + 32 * (i0 + q)),
                        r[q]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (i0 + q >= nch) break;
            const int c0 = 16 * half + 32 * (i0 + q);
            float b[16];
#pragma unroll
            for (int j = 0; j < 16; j += 4)
              *reinterpret_cast<float4*>(b + j) = *reinterpret_cast<const float4*>(bias + c0 + j);
            if (last) {
              if (gr < B) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (c0 + j < fo) out[gr * fo + c0 + j] = __uint_as_float(r[q][j]) + b[j];
              }
            } else {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t w[4];
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                  const int n = c0 + 8 * h + j;
                  const float2 a = silu2_f(__uint_as_float(r[q][8 * h + j]) + b[8 * h + j],
                                           __uint_as_float(r[q][8 * h + j + 1]) + b[8 * h + j + 1]);
                  w[j / 2] = pack_bf16x2(n < fo ? a.x : 0.0f, n + 1 < fo ? a.y : 0.0f);
                }
                *reinterpret_cast<uint4*>(sH + core_off(row, c0 + 8 * h, kpn)) = make_uint4(w[0], w[1], w[2], w[3]);
              }
            }
          }
        }
      } else if (last && gr < B) {
        for (int n = half; n < fo; n += 2) out[gr * fo + n] = __int_as_float(0x7fc00000);
      }
      if (!last) {
        for (int k0 = np + 8 * half; k0 < kpn; k0 += 16)
          *reinterpret_cast<uint4*>(sH + core_off(row, k0, kpn)) = make_uint4(0, 0, 0, 0);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&h_ready[slot])) : "memory");
      } else if (lt + 2 < ord.mine) {
        // this slot's next tile (its accumulator has been read)
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        stage_input(lt + 2);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && abort_flag && status) atomicExch(status, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(uint32_t(2 * kFusedMaxN)) : "memory");
}

// Adam (Kingma & Ba 2015, Algorithm 1), bias-corrected, FP32.
__global__ void adam_kernel(int64_t n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// Normalised network input of cell i from the species-major FP64 state.
__global__ void features_kernel(int64_t n, int nsp, const double* __restrict__ T, const double* __restrict__ p,
                                const double* __restrict__ Y, double dt, const float* __restrict__ mu,
                                const float* __restrict__ isd, float* __restrict__ X) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int nin = nsp + 3;
  float* x = X + i * nin;
  x[0] = (float(T[i] * 1e-3) - mu[0]) * isd[0];
  x[1] = (float(log(p[i])) - mu[1]) * isd[1];
  for (int k = 0; k < nsp; ++k) x[2 + k] = (float(Y[int64_t(k) * n + i]) - mu[2 + k]) * isd[2 + k];
  x[nin - 1] = (float(log(dt)) - mu[nin - 1]) * isd[nin - 1];
}

// Physical predictions from the normalised network output: ln steps, dT,
// dY (species-major, FP64).
__global__ void predictions_kernel(int64_t n, int nsp, const float* __restrict__ out, const float* __restrict__ mu,
                                   const float* __restrict__ sd, float* __restrict__ lnsteps,
                                   double* __restrict__ dT, double* __restrict__ dY) {
  const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (i >= n) return;
  const int nout = nsp + 2;
  const float* o = out + i * nout;
  lnsteps[i] = o[0] * sd[0] + mu[0];
  dT[i] = double(o[1] * sd[1] + mu[1]);
  for (int k = 0; k < nsp; ++k) dY[int64_t(k) * n + i] = double(o[2 + k] * sd[2 + k] + mu[2 + k]);
}

}  // namespace dlb

struct dlbchem_mlp {
  int n_in = 0, n_hidden = 256, n_out = 0, n_layers = 3;
  int64_t nparams = 0;
  float* d_params = nullptr;   // [W1 b1 W2 b2 W3 b3 W4 b4], W row-major [fan_in, fan_out]
  float* d_m = nullptr;
  float* d_v = nullptr;
  float* d_grad = nullptr;
  float* d_norm = nullptr;     // mu_x, isd_x, mu_y, sd_y
  int* d_status = nullptr;     // set to 1 by a GEMM whose tensor-core wait gave up
  int adam_t = 0;
  // fused forward (inference): BF16 weights packed as the fused kernel's
  // k-tiles, repacked after every parameter change
  bool fused_ok = false;       // the shape is one the fused kernel takes
  bool fused_on = true;        // dlbchem_mlp_set_fused
  bool packed_dirty = true;
  unsigned char* d_wpk = nullptr;
  dlb::FusedNet fnet{};
  int num_sms = 0;
  // activations for the largest batch seen
  int64_t cap = 0;
  float* d_act = nullptr;
  std::string err;
};

namespace {

int mfail(dlbchem_mlp* m, int code, const std::string& msg) {
  if (m) m->err = msg;
  return code;
}

struct LayerOff {
  int64_t w, b;
  int fi, fo;
};

std::vector<LayerOff> layers_of(const dlbchem_mlp* m) {
  std::vector<int> dims = {m->n_in};
  for (int i = 0; i < m->n_layers; ++i) dims.push_back(m->n_hidden);
  dims.push_back(m->n_out);
  std::vector<LayerOff> L;
  int64_t o = 0;
  for (size_t i = 0; i + 1 < dims.size(); ++i) {
    LayerOff l;
    l.fi = dims[i];
    l.fo = dims[i + 1];
    l.w = o;
    o += int64_t(l.fi) * l.fo;
    l.b = o;
    o += l.fo;
    L.push_back(l);
  }
  return L;
}

dim3 tiles_of(int64_t rows, int cols) {
  return dim3((cols + dlb::kTN - 1) / dlb::kTN, unsigned((rows + dlb::kTM - 1) / dlb::kTM));
}

// activation workspace: per hidden layer Z and H [cap x n_hidden], output
// (or its gradient) [cap x n_out].
int ensure_act(dlbchem_mlp* m, int64_t batch) {
  if (batch <= m->cap) return DLBCHEM_OK;
  if (m->d_act) cudaFree(m->d_act);
  m->d_act = nullptr;
  m->cap = 0;
  const int64_t per = 2 * int64_t(m->n_layers) * m->n_hidden + m->n_out;
  if (cudaMalloc(&m->d_act, size_t(batch) * per * 4) != cudaSuccess) {
    m->d_act = nullptr;
    return mfail(m, DLBCHEM_OOM, "network activation allocation failed");
  }
  m->cap = batch;
  return DLBCHEM_OK;
}

// Fused-forward tables of the network (weights still to pack); false if the
// shape is not one the fused kernel takes.
bool plan_fused(dlbchem_mlp* m) {
  const auto L = layers_of(m);
  if (int(L.size()) > dlb::kFusedMaxLayers) return false;
  if (m->n_hidden % 64 != 0 || m->n_hidden > dlb::kFusedMaxN || m->n_in > dlb::kFusedMaxN ||
      m->n_out > dlb::kFusedMaxN)
    return false;
  dlb::FusedNet& f = m->fnet;
  f.nl = int(L.size());
  int64_t off = 0;
  for (int l = 0; l < f.nl; ++l) {
    f.fi[l] = L[l].fi;
    f.fo[l] = L[l].fo;
    f.kp[l] = (L[l].fi + dlb::kFK - 1) / dlb::kFK * dlb::kFK;
    f.np[l] = (L[l].fo + 15) / 16 * 16;
    f.woff[l] = off;
    off += int64_t(f.kp[l]) * f.np[l] * 2;
  }
  if (cudaMalloc(&m->d_wpk, size_t(off)) != cudaSuccess) {
    m->d_wpk = nullptr;
    return false;
  }
  f.wpk = m->d_wpk;
  for (int l = 0; l < f.nl; ++l) f.bias[l] = m->d_params + L[l].b;
  const int64_t last_bytes = int64_t(f.kp[f.nl - 1]) * f.np[f.nl - 1] * 2;
  f.res_bytes = last_bytes <= dlb::kFusedResident ? uint32_t(last_bytes) : 0u;
  return cudaFuncSetAttribute(dlb::mlp_fused_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              dlb::kFusedSmem) == cudaSuccess;
}

cudaError_t forward_fused(dlbchem_mlp* m, int64_t B, const float* X, float* out, cudaStream_t s) {
  const auto L = layers_of(m);
  cudaError_t e = cudaSuccess;
  if (m->packed_dirty) {
    for (int l = 0; l < m->fnet.nl && e == cudaSuccess; ++l) {
      const int64_t tot = int64_t(m->fnet.kp[l]) * m->fnet.np[l];
      dlb::pack_weights_kernel<<<unsigned(std::min<int64_t>((tot + 255) / 256, 1024)), 256, 0, s>>>(
          L[l].fi, L[l].fo, m->fnet.kp[l], m->fnet.np[l], m->d_params + L[l].w, m->d_wpk + m->fnet.woff[l]);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    m->packed_dirty = false;
  }
  // persistent: one CTA per SM (its two accumulators fill tensor memory)
  const int64_t tiles = (B + dlb::kTM - 1) / dlb::kTM;
  const int64_t grid = std::min<int64_t>(tiles, int64_t(m->num_sms));
  dlb::mlp_fused_forward_kernel<<<unsigned(grid), dlb::kFusedThreads, dlb::kFusedSmem, s>>>(B, X, out, m->fnet,
                                                                                           m->d_status);
  return cudaGetLastError();
}

// Forward; with keep the pre-activations are stored for the backward pass (and
// with a target out receives the gradient of the MSE, *loss its value).
// Without keep (inference) the fused whole-network kernel runs where the
// shape allows it.
cudaError_t forward(dlbchem_mlp* m, int64_t B, const float* X, float* out, bool keep, cudaStream_t s,
                    const float* target = nullptr, float scale = 0.0f, float* loss = nullptr) {
  if (!keep && m->fused_ok && m->fused_on) return forward_fused(m, B, X, out, s);
  const auto L = layers_of(m);
  const int64_t H = m->n_hidden;
  float* Zs = m->d_act;                                  // n_layers x [B x H]
  float* Hs = Zs + int64_t(m->n_layers) * B * H;         // n_layers x [B x H]
  const float* in = X;
  cudaError_t e = cudaSuccess;
  for (int li = 0; li < int(L.size()) && e == cudaSuccess; ++li) {
    const bool last = li + 1 == int(L.size());
    float* dst = last ? out : Hs + int64_t(li) * B * H;
    float* z = (!last && keep) ? Zs + int64_t(li) * B * H : nullptr;
    dlb::layer_forward_kernel<<<tiles_of(B, L[li].fo), dlb::kGemmThreads + 32, dlb::tile_bytes(dlb::kTN), s>>>(int(B), L[li].fo, L[li].fi, in, m->d_params + L[li].w,
                                                                   dst, m->d_params + L[li].b, z, last ? 0 : 1,
                                                                   last ? target : nullptr, scale, loss, m->d_status);
    e = cudaGetLastError();
    in = dst;
  }
  return e;
}

}  // namespace

extern "C" {

int dlbchem_mlp_create(int n_in, int n_hidden, int n_out, dlbchem_mlp** out) {
  if (!out || n_in < 1 || n_hidden < 1 || n_out < 1) return DLBCHEM_BAD_ARG;
  *out = nullptr;
  auto* m = new dlbchem_mlp;
  m->n_in = n_in; m->n_hidden = n_hidden; m->n_out = n_out;
  const auto L = layers_of(m);
  m->nparams = L.back().b + L.back().fo;
  const size_t bytes = size_t(m->nparams) * 4;
  if (cudaMalloc(&m->d_params, bytes) != cudaSuccess || cudaMalloc(&m->d_m, bytes) != cudaSuccess ||
      cudaMalloc(&m->d_v, bytes) != cudaSuccess || cudaMalloc(&m->d_grad, bytes) != cudaSuccess ||
      cudaMalloc(&m->d_norm, size_t(2 * (n_in + n_out)) * 4) != cudaSuccess ||
      cudaMalloc(&m->d_status, sizeof(int)) != cudaSuccess) {
    dlbchem_mlp_destroy(m);
    return DLBCHEM_OOM;
  }
  cudaMemset(m->d_params, 0, bytes);
  cudaMemset(m->d_status, 0, sizeof(int));
  cudaMemset(m->d_m, 0, bytes);
  cudaMemset(m->d_v, 0, bytes);
  std::vector<float> norm(2 * (n_in + n_out), 0.0f);
  for (int i = 0; i < n_in; ++i) norm[n_in + i] = 1.0f;
  for (int i = 0; i < n_out; ++i) norm[2 * n_in + n_out + i] = 1.0f;
  cudaMemcpy(m->d_norm, norm.data(), norm.size() * 4, cudaMemcpyHostToDevice);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    m->num_sms = 1;
  // operand buffers beyond the default 48 KB (a failure shows at the launch)
  (void)cudaFuncSetAttribute(dlb::layer_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dlb::tile_bytes(dlb::kTN));
  (void)cudaFuncSetAttribute(dlb::weight_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dlb::tile_bytes(dlb::kGradTN));
  (void)cudaFuncSetAttribute(dlb::layer_backward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dlb::tile_bytes(dlb::kTN));
  m->fused_ok = plan_fused(m);
  *out = m;
  return DLBCHEM_OK;
}

int64_t dlbchem_mlp_nparams(const dlbchem_mlp* m) { return m ? m->nparams : -1; }

int dlbchem_mlp_set_params(dlbchem_mlp* m, const float* params, void* stream) {
  if (!m || !params) return DLBCHEM_BAD_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  m->packed_dirty = true;
  cudaError_t e = cudaMemcpyAsync(m->d_params, params, size_t(m->nparams) * 4, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->d_m, 0, size_t(m->nparams) * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->d_v, 0, size_t(m->nparams) * 4, s);
  m->adam_t = 0;
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

int dlbchem_mlp_get_params(dlbchem_mlp* m, float* params, void* stream) {
  if (!m || !params) return DLBCHEM_BAD_ARG;
  const cudaError_t e = cudaMemcpyAsync(params, m->d_params, size_t(m->nparams) * 4, cudaMemcpyDeviceToDevice,
                                        static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

int dlbchem_mlp_set_norm(dlbchem_mlp* m, const float* mu_x, const float* sd_x, const float* mu_y, const float* sd_y) {
  if (!m || !mu_x || !sd_x || !mu_y || !sd_y) return DLBCHEM_BAD_ARG;
  std::vector<float> norm;
  for (int i = 0; i < m->n_in; ++i) norm.push_back(mu_x[i]);
  for (int i = 0; i < m->n_in; ++i) {
    if (!(sd_x[i] > 0)) return mfail(m, DLBCHEM_BAD_ARG, "input scales must be positive");
    norm.push_back(1.0f / sd_x[i]);
  }
  for (int i = 0; i < m->n_out; ++i) norm.push_back(mu_y[i]);
  for (int i = 0; i < m->n_out; ++i) norm.push_back(sd_y[i]);
  const cudaError_t e = cudaMemcpy(m->d_norm, norm.data(), norm.size() * 4, cudaMemcpyHostToDevice);
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

int dlbchem_mlp_forward(dlbchem_mlp* m, int64_t batch, const float* X, float* out, void* stream) {
  if (!m || batch < 0 || (batch > 0 && (!X || !out))) return DLBCHEM_BAD_ARG;
  if (batch == 0) return DLBCHEM_OK;
  int rc = ensure_act(m, batch);
  if (rc != DLBCHEM_OK) return rc;
  const cudaError_t e = forward(m, batch, X, out, false, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

// Loss and gradient of the MSE on one batch (X [B x n_in], Y [B x n_out],
// normalised). grad: device [nparams] or NULL (internal buffer); loss:
// device float or NULL.
int dlbchem_mlp_grad(dlbchem_mlp* m, int64_t B, const float* X, const float* Y, float* grad, float* loss, void* stream) {
  if (!m || B < 1 || !X || !Y) return DLBCHEM_BAD_ARG;
  int rc = ensure_act(m, B);
  if (rc != DLBCHEM_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* g = grad ? grad : m->d_grad;
  const auto L = layers_of(m);
  const int64_t H = m->n_hidden;
  float* Zs = m->d_act;                                  // pre-activations, then their gradients
  float* Hs = Zs + int64_t(m->n_layers) * B * H;
  float* dout = Hs + int64_t(m->n_layers) * B * H;
  cudaError_t e = loss ? cudaMemsetAsync(loss, 0, 4, s) : cudaSuccess;
  if (e == cudaSuccess) e = forward(m, B, X, dout, true, s, Y, 1.0f / float(B * m->n_out), loss);
  dlb::GradArgs a;
  a.nl = int(L.size()); a.B = int(B); a.grad = g;
  int tiles = 0;
  for (int li = 0; li < a.nl; ++li) {
    const int n = (L[li].fo + dlb::kGradTN - 1) / dlb::kGradTN * ((L[li].fi + dlb::kTM - 1) / dlb::kTM);
    a.layer[li] = {li == 0 ? X : Hs + int64_t(li - 1) * B * H, li + 1 == a.nl ? dout : Zs + int64_t(li) * B * H,
                   L[li].fi, L[li].fo, tiles, L[li].w};
    tiles += n;
  }
  for (int li = a.nl - 1; li > 0 && e == cudaSuccess; --li) {
    dlb::layer_backward_kernel<<<tiles_of(B, L[li].fi), dlb::kGemmThreads + 32, dlb::tile_bytes(dlb::kTN), s>>>(int(B), L[li].fi, L[li].fo, a.layer[li].dz,
                                                                     m->d_params + L[li].w,
                                                                     Zs + int64_t(li - 1) * B * H, m->d_status);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    dlb::weight_grad_kernel<<<unsigned(tiles), dlb::kGemmThreads + 32, dlb::tile_bytes(dlb::kGradTN), s>>>(a, m->d_status);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

int dlbchem_mlp_adam(dlbchem_mlp* m, const float* grad, float lr, void* stream) {
  if (!m || !(lr > 0)) return DLBCHEM_BAD_ARG;
  m->adam_t += 1;
  m->packed_dirty = true;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - std::pow(b1, float(m->adam_t)), c2 = 1.0f - std::pow(b2, float(m->adam_t));
  dlb::adam_kernel<<<unsigned(std::min<int64_t>((m->nparams + 255) / 256, 2048)), 256, 0,
                     static_cast<cudaStream_t>(stream)>>>(m->nparams, m->d_params, grad ? grad : m->d_grad, m->d_m,
                                                          m->d_v, lr, b1, b2, 1e-8f, c1, c2);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? DLBCHEM_OK : mfail(m, DLBCHEM_CUDA, cudaGetErrorString(e));
}

int dlbchem_mlp_train_step(dlbchem_mlp* m, int64_t B, const float* X, const float* Y, float lr, float* loss,
                           void* stream) {
  int rc = dlbchem_mlp_grad(m, B, X, Y, nullptr, loss, stream);
  return rc == DLBCHEM_OK ? dlbchem_mlp_adam(m, nullptr, lr, stream) : rc;
}

int dlbchem_mlp_set_fused(dlbchem_mlp* m, int enable) {
  if (!m || (enable != 0 && enable != 1)) return DLBCHEM_BAD_ARG;
  m->fused_on = enable != 0;
  return DLBCHEM_OK;
}

int dlbchem_mlp_fused(const dlbchem_mlp* m) { return m ? int(m->fused_ok && m->fused_on) : -1; }

const char* dlbchem_mlp_last_error(const dlbchem_mlp* m) { return m ? m->err.c_str() : ""; }

void dlbchem_mlp_destroy(dlbchem_mlp* m) {
  if (!m) return;
  cudaDeviceSynchronize();
  for (float* p : {m->d_params, m->d_m, m->d_v, m->d_grad, m->d_norm, m->d_act})
    if (p) cudaFree(p);
  if (m->d_status) cudaFree(m->d_status);
  if (m->d_wpk) cudaFree(m->d_wpk);
  delete m;
}

}  // extern "C"

namespace dlb {

// Network predictions for n cells of one context's field (used by
// dlbchem_integrate when the predictor or the surrogate is on): features ->
// forward -> physical ln steps, dT, dY. X, out, lnsteps, dT, dY are caller
// workspace.
cudaError_t mlp_predict(dlbchem_mlp* m, int64_t n, int nsp, const double* T, const double* p, const double* Y,
                        double dt, float* X, float* out, float* lnsteps, double* dT, double* dY, cudaStream_t s) {
  if (ensure_act(m, std::min<int64_t>(n, 65536)) != DLBCHEM_OK) return cudaErrorMemoryAllocation;
  const float* mu_x = m->d_norm;
  const float* isd_x = mu_x + m->n_in;
  const float* mu_y = isd_x + m->n_in;
  const float* sd_y = mu_y + m->n_out;
  features_kernel<<<unsigned((n + 255) / 256), 256, 0, s>>>(n, nsp, T, p, Y, dt, mu_x, isd_x, X);
  cudaError_t e = cudaGetLastError();
  for (int64_t b0 = 0; b0 < n && e == cudaSuccess; b0 += 65536) {
    const int64_t b = std::min<int64_t>(65536, n - b0);
    e = forward(m, b, X + b0 * m->n_in, out + b0 * m->n_out, false, s);
  }
  if (e == cudaSuccess) {
    predictions_kernel<<<unsigned((n + 255) / 256), 256, 0, s>>>(n, nsp, out, mu_y, sd_y, lnsteps, dT, dY);
    e = cudaGetLastError();
  }
  return e;
}

int mlp_shape(const dlbchem_mlp* m, int* n_in, int* n_out) {
  *n_in = m->n_in;
  *n_out = m->n_out;
  return 0;
}

}  // namespace dlb
