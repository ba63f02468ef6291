// Learned surrogate of the UQ map (stochastic process inputs -> the
// microstructure outputs of Section 2.6, Eq. 22-23), replacing the plain
// solve inside Monte Carlo sampling (Section 2.7 uses a polynomial-chaos
// surrogate for the same role).
//
// A multilayer perceptron with GELU hidden layers and a linear output,
// BF16 weights and activations, FP32 accumulation in tensor memory on the
// tcgen05 tensor cores, FP32 master weights and Adam moments.  Every
// dimension is padded to a multiple of 16 with zeros that stay zero.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"

namespace fvs {

#define GS(i, n) for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

enum { EPI_GELU = 0, EPI_LINEAR = 1, EPI_DGRAD = 2 };

struct Epi {
  const float* bias;   // [N]           (GELU, LINEAR)
  float* z;            // [M x ldo] f32  pre-activations to keep (GELU, LINEAR) or read (DGRAD)
  bf16* hout;          // [M x ldo] bf16 activations (GELU) / previous delta (DGRAD)
  float* fout;         // [M x ldo] f32  output (LINEAR)
  int ldo;
};

// ---------------------------------------------------------------------------
// C[M x N] = sum_k A(m, k) B(n, k) with A(m, k) = A[m*am + k*ak], B(n, k) =
// B[n*bn + k*bk] (BF16), N <= 128, K a multiple of 16, on the
// 5th-generation tensor cores (tcgen05) with a fused epilogue: one CTA of
// four warps per 128 rows of C, all N (<= 128) columns in one tile, K in
// chunks of 64.  Each chunk of A (128 x 64) and B (N x 64) is staged in
// shared memory in the canonical K-major layout without swizzle (core
// matrices of 8 rows x 16 bytes; 128 bytes between core matrices along K,
// 1024 bytes between groups of 8 rows), one thread issues the chunk's
// 128 x N x 16 BF16 MMAs into an FP32 accumulator in tensor memory and
// commits them to an mbarrier, and after the last chunk every warp reads
// its 32 accumulator lanes with tcgen05.ld for the fused epilogue.  Waits are
// bounded: a wait that runs out sets *err and the CTA still frees its
// tensor memory.
// ---------------------------------------------------------------------------
constexpr int TC_KC = 64;
constexpr int TC_COLS = 128;   // tensor-memory columns of a CTA (N <= 128)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ int tc_off(int r, int k) { return (r >> 3) * 1024 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2; }
// shared-memory matrix descriptor: start address, leading and stride byte
// offsets (16-byte units), descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46);
}
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t phase) {
  uint32_t done = 0;
  for (int it = 0; it < (1 << 22) && !done; ++it)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(phase));
  return done != 0;
}

// fused epilogue of one 128-row tile: warp group `warp` (0-3) reads its 32
// accumulator lanes (rows m0 + 32 warp + lane) from tensor memory, 16
// columns at a time from c_begin in steps of c_step (two warps of the same
// group split the columns by starting 16 apart with a step of 32)
template <int EPI>
__device__ __forceinline__ void tc_epilogue(uint32_t taddr, int warp, int lane, int m0, int M, int N, const Epi& e,
                                            int c_begin = 0, int c_step = 16) {
  const int m = m0 + warp * 32 + lane;
  for (int c0 = c_begin; c0 < N; c0 += c_step) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0));
    asm volatile("tcgen05.wait::ld.sync.aligned;");
    if (m >= M) continue;
    const int64_t o0 = (int64_t)m * e.ldo + c0;
    if ((e.ldo & 7) == 0) {
      // a lane's 16 columns as 16-byte vectors (row offsets are multiples of 8 elements)
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
      if (EPI == EPI_GELU || EPI == EPI_LINEAR) {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] += e.bias[c0 + j];
      }
      if (EPI == EPI_DGRAD) {
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
          const float4 z = *reinterpret_cast<const float4*>(e.z + o0 + j);
          v[j] *= gelu_grad(z.x); v[j + 1] *= gelu_grad(z.y); v[j + 2] *= gelu_grad(z.z); v[j + 3] *= gelu_grad(z.w);
        }
      }
      float* f32out = EPI == EPI_GELU ? e.z : e.fout;
      if ((EPI == EPI_LINEAR || EPI == EPI_GELU) && f32out) {
#pragma unroll
        for (int j = 0; j < 16; j += 4)
          *reinterpret_cast<float4*>(f32out + o0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
      if (EPI == EPI_GELU || EPI == EPI_DGRAD) {
        uint32_t h[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float a = EPI == EPI_GELU ? gelu(v[2 * j]) : v[2 * j];
          const float b = EPI == EPI_GELU ? gelu(v[2 * j + 1]) : v[2 * j + 1];
          const __nv_bfloat162 hb = __floats2bfloat162_rn(a, b);
          h[j] = *reinterpret_cast<const uint32_t*>(&hb);
        }
        uint4* dst = reinterpret_cast<uint4*>(e.hout + o0);
        dst[0] = make_uint4(h[0], h[1], h[2], h[3]);
        dst[1] = make_uint4(h[4], h[5], h[6], h[7]);
      }
      continue;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int n = c0 + j;
      const int64_t o = o0 + j;
      float v = __uint_as_float(r[j]);
      if (EPI == EPI_GELU) {
        v += e.bias[n];
        if (e.z) e.z[o] = v;
        e.hout[o] = __float2bfloat16(gelu(v));
      } else if (EPI == EPI_LINEAR) {
        v += e.bias[n];
        e.fout[o] = v;
      } else {
        e.hout[o] = __float2bfloat16(v * gelu_grad(e.z[o]));
      }
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(128, 1) k_mlp_gemm_tc(int M, int N, int K, const bf16* __restrict__ A, int am, int ak,
                                                        const bf16* __restrict__ B, int bn, int bk, Epi e, int* err) {
  __shared__ __align__(1024) unsigned char sa[128 * TC_KC * 2];
  __shared__ __align__(1024) unsigned char sb[TC_COLS * TC_KC * 2];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t taddr_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * 128;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_s)),
                 "r"(TC_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)));
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = taddr_s;
  // kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both
  // K-major, N >> 3, M >> 4
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  const bf16 zero = __float2bfloat16(0.f);
  uint32_t phase = 0;
  bool ok = true;
  for (int k0 = 0; k0 < K && ok; k0 += TC_KC) {
    const int kc = min(TC_KC, K - k0);
    // stage A(m, k) and B(n, k).  Rows contiguous in k go as 16-byte core
    // matrix rows (eight consecutive threads take the eight rows of one core
    // matrix: one 128-byte shared-memory wavefront, no bank conflicts);
    // otherwise element by element with the index that is contiguous in
    // memory running fastest.
    const int nch = kc >> 3;
    if (ak == 1 && (am & 7) == 0) {
      for (int t = tid; t < 128 * nch; t += 128) {
        const int q = t >> 3, ch = q % nch, r = (q / nch) * 8 + (t & 7);
        const int m = m0 + r;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (m < M) v = *reinterpret_cast<const uint4*>(A + (int64_t)m * am + k0 + ch * 8);
        *reinterpret_cast<uint4*>(sa + tc_off(r, ch * 8)) = v;
      }
    } else {
      for (int t = tid; t < 128 * kc; t += 128) {
        const int r = ak == 1 ? t / kc : t % 128, k = ak == 1 ? t % kc : t / 128;
        const int m = m0 + r;
        *(bf16*)(sa + tc_off(r, k)) = m < M ? A[(int64_t)m * am + (int64_t)(k0 + k) * ak] : zero;
      }
    }
    if (bk == 1 && (bn & 7) == 0) {
      for (int t = tid; t < N * nch; t += 128) {
        const int q = t >> 3, ch = q % nch, r = (q / nch) * 8 + (t & 7);
        *reinterpret_cast<uint4*>(sb + tc_off(r, ch * 8)) =
            *reinterpret_cast<const uint4*>(B + (int64_t)r * bn + k0 + ch * 8);
      }
    } else {
      for (int t = tid; t < N * kc; t += 128) {
        const int r = bk == 1 ? t / kc : t % N, k = bk == 1 ? t % kc : t / N;
        *(bf16*)(sb + tc_off(r, k)) = B[(int64_t)r * bn + (int64_t)(k0 + k) * bk];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      for (int kk = 0; kk < kc / 16; ++kk) {
        const uint64_t ad = tc_desc(smem_u32(sa) + kk * 256), bd = tc_desc(smem_u32(sb) + kk * 256);
        const uint32_t accum = (k0 > 0 || kk > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(taddr),
            "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(&mbar)));
    }
    if (!tc_wait(smem_u32(&mbar), phase)) {
      ok = false;
      if (lane == 0) atomicOr(err, 1);
      tc_wait(smem_u32(&mbar), phase);   // give the MMAs in flight a second bounded chance
    }
    phase ^= 1;
    asm volatile("tcgen05.fence::after_thread_sync;");
    __syncthreads();
  }
  if (ok) tc_epilogue<EPI>(taddr, warp, lane, m0, M, N, e);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TC_COLS));
}

// ---------------------------------------------------------------------------
// Forward GEMM (activations A [M x K] row-major times weights B [N x K],
// K <= 128, N <= 128) as a persistent kernel: each CTA stages the weights
// once, allocates its tensor-memory accumulator once, and walks the 128-row
// tiles t = blockIdx.x, blockIdx.x + gridDim.x, ... with eight warps (two per
// accumulator lane group in the epilogue)  The A tile of the next
// tile is copied into the other of two shared-memory buffers (cp.async,
// 16-byte core-matrix rows, zero fill past M) while the current tile's MMAs
// and epilogue run.  Layouts, descriptors and the epilogue are those of
// k_mlp_gemm_tc; every wait on the MMAs is bounded and the decision to stop
// is taken by the whole CTA (__syncthreads_or), which then drains its copies
// and frees its tensor memory.
// ---------------------------------------------------------------------------
constexpr int TC_CHUNK_BYTES = 128 * TC_KC * 2;   // one K chunk of 128 rows
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
// rows of A's tile m0 into buffer sa (K in chunks of TC_KC, 16-byte pieces)
__device__ __forceinline__ void tc_stage_a_async(unsigned char* sa, const bf16* A, int M, int K, int m0, int tid,
                                                 int nthr) {
  const int nchunk = (K + TC_KC - 1) / TC_KC;
  for (int c = 0; c < nchunk; ++c) {
    const int k0 = c * TC_KC, kc = min(TC_KC, K - k0), nch = kc >> 3;
    unsigned char* base = sa + c * TC_CHUNK_BYTES;
    for (int t = tid; t < 128 * nch; t += nthr) {
      const int q = t >> 3, ch = q % nch, r = (q / nch) * 8 + (t & 7);
      const int m = m0 + r;
      const bf16* src = m < M ? A + (int64_t)m * K + k0 + ch * 8 : A;
      cp_async16(smem_u32(base + tc_off(r, ch * 8)), src, m < M ? 16 : 0);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int EPI>
__global__ void __launch_bounds__(256, 1) k_mlp_fwd_tc(int M, int N, int K, const bf16* __restrict__ A,
                                                       const bf16* __restrict__ B, Epi e, int* err) {
  extern __shared__ __align__(1024) unsigned char tc_dyn[];
  const int nchunk = (K + TC_KC - 1) / TC_KC;
  unsigned char* sb = tc_dyn;                               // nchunk chunks
  unsigned char* sa0 = tc_dyn + nchunk * TC_CHUNK_BYTES;    // 2 x nchunk chunks
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t taddr_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int ntiles = (M + 127) / 128;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_s)),
                 "r"(TC_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)));
  // the weights, once
  for (int c = 0; c < nchunk; ++c) {
    const int k0 = c * TC_KC, kc = min(TC_KC, K - k0), nch = kc >> 3;
    for (int t = tid; t < N * nch; t += blockDim.x) {
      const int q = t >> 3, ch = q % nch, r = (q / nch) * 8 + (t & 7);
      *reinterpret_cast<uint4*>(sb + c * TC_CHUNK_BYTES + tc_off(r, ch * 8)) =
          *reinterpret_cast<const uint4*>(B + (int64_t)r * K + k0 + ch * 8);
    }
  }
  if (blockIdx.x < ntiles) tc_stage_a_async(sa0, A, M, K, blockIdx.x * 128, tid, blockDim.x);
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = taddr_s;
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
  uint32_t phase = 0;
  int buf = 0;
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int next = tile + gridDim.x;
    if (next < ntiles) {
      tc_stage_a_async(sa0 + (buf ^ 1) * nchunk * TC_CHUNK_BYTES, A, M, K, next * 128, tid, blockDim.x);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      const unsigned char* sa = sa0 + buf * nchunk * TC_CHUNK_BYTES;
      for (int c = 0; c < nchunk; ++c) {
        const int kc = min(TC_KC, K - c * TC_KC);
        for (int kk = 0; kk < kc / 16; ++kk) {
          const uint64_t ad = tc_desc(smem_u32(sa + c * TC_CHUNK_BYTES) + kk * 256);
          const uint64_t bd = tc_desc(smem_u32(sb + c * TC_CHUNK_BYTES) + kk * 256);
          const uint32_t accum = (c > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(taddr),
              "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
        }
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(&mbar)));
    }
    const bool late = __syncthreads_or(!tc_wait(smem_u32(&mbar), phase) ? 1 : 0);
    if (late) {
      if (tid == 0) atomicOr(err, 1);
      tc_wait(smem_u32(&mbar), phase);   // the MMAs in flight get a second bounded chance
      break;
    }
    phase ^= 1;
    asm volatile("tcgen05.fence::after_thread_sync;");
    // eight warps: warp w reads accumulator lanes 32 (w % 4) .. +31, the
    // 16-column blocks starting at 16 (w / 4), every other one
    tc_epilogue<EPI>(taddr, warp & 3, lane, tile * 128, M, N, e, 16 * (warp >> 2), 32);
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();   // accumulator read before the next tile's MMAs; buffer free for reuse
    asm volatile("tcgen05.fence::after_thread_sync;");
    buf ^= 1;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TC_COLS));
}

// ---------------------------------------------------------------------------
// The whole network in one kernel.  With the layers as separate launches a
// million samples move 256 B of activations a row and layer to memory and
// back and the input and output conversions are passes of their own; a
// training epoch of a few hundred rows is launch after launch of a handful
// of CTAs.  Here every layer's weights stay in shared memory (104 KB for 3 ->
// 128 x 4 -> 4), a 128-row tile goes through all layers in place, and only
// inputs and outputs (and, in training, what the weight gradients need) touch
// memory.  What is left is bound by the FP32 pipe: about 64 issue slots a
// GELU (erff), 512 GELUs a sample.
//
// Operands lie in the canonical layouts without swizzle: core matrices of
// 8 rows x 16 bytes, those along the row's direction 128 bytes apart, groups
// of eight rows 16 K bytes apart (fu_off).  A weight matrix W [N x K] staged
// that way is the K-major B operand of the forward product (leading offset
// 128, stride offset 16 K) and, the same bytes, the MN-major B operand of the
// product delta W of the back-propagation (leading offset 16 K along the
// reduction over n, stride offset 128 along k).
// ---------------------------------------------------------------------------
constexpr int FU_MAXL = 17;       // layers of the largest network (16 hidden + output)
constexpr int FU_ACT = 128 * 128 * 2;   // one activation tile
struct FusedNet {
  int L, nin, nout;
  int kd[FU_MAXL + 1];   // padded widths
  int woff[FU_MAXL];     // weights of layer l: elements into the BF16 copy
  int boff[FU_MAXL];     // biases: elements into the FP32 parameters
  int soff[FU_MAXL];     // weights in shared memory: bytes
  int wbytes;
};
__device__ __forceinline__ int fu_off(int r, int k, int K) {
  return (r >> 3) * (K * 16) + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
__device__ __forceinline__ uint64_t fu_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         ((uint64_t)1 << 46);
}
__device__ __forceinline__ void fu_mma(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(ad), "l"(bd), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void fu_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar));
}
// FP32 accumulator, BF16 operands, 128 x N tile; tr_a / tr_b: that operand is MN-major
__device__ __forceinline__ uint32_t fu_idesc(int N, uint32_t tr_a, uint32_t tr_b) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (tr_a << 15) | (tr_b << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void fu_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}
__device__ __forceinline__ void fu_pack16(const float* v, uint4& lo, uint4& hi) {
  uint32_t h[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const __nv_bfloat162 hb = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    h[j] = *reinterpret_cast<const uint32_t*>(&hb);
  }
  lo = make_uint4(h[0], h[1], h[2], h[3]);
  hi = make_uint4(h[4], h[5], h[6], h[7]);
}
__device__ __forceinline__ void fu_bias16(const float* bias, float* v) {
#pragma unroll
  for (int j = 0; j < 16; j += 4) {
    const float4 b = *reinterpret_cast<const float4*>(bias + j);
    v[j] += b.x; v[j + 1] += b.y; v[j + 2] += b.z; v[j + 3] += b.w;
  }
}
// every layer's weights into shared memory (cp.async, one group)
__device__ __forceinline__ void fu_stage_weights(unsigned char* sw, const FusedNet& net, const bf16* wb) {
  for (int l = 0; l < net.L; ++l) {
    const int K = net.kd[l], N = net.kd[l + 1], nch = K >> 3;
    for (int t = threadIdx.x; t < N * nch; t += blockDim.x) {
      const int q = t >> 3, ch = q % nch, r = (q / nch) * 8 + (t & 7);
      cp_async16(smem_u32(sw + net.soff[l] + fu_off(r, ch * 8, K)), wb + net.woff[l] + r * K + ch * 8, 16);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// normalised BF16 inputs of eight columns of one row (zero past the inputs)
__device__ __forceinline__ uint4 fu_input8(const double* X, int64_t m, int64_t n, int nin, int c0, const float* mu,
                                           const float* sd) {
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = c0 + j;
    v[j] = (m < n && c < nin) ? (float)((X[m * nin + c] - (double)mu[c]) / (double)sd[c]) : 0.f;
  }
  uint32_t h[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 hb = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    h[j] = *reinterpret_cast<const uint32_t*>(&hb);
  }
  return make_uint4(h[0], h[1], h[2], h[3]);
}

// Prediction: one CTA per SM, up to three groups of eight warps, each group
// with its own tile, activation buffer and accumulator, so that one group's
// MMAs and waits pass under another's epilogue.  A wait that runs out sets
// *err; the group then leaves its loop, waits once more (bounded) for the
// MMAs in flight, and the CTA frees its tensor memory.
// A million samples of 3 -> 128 x 4 -> 4: 1363 us as eight launches, 756 us
// as one; 1000 samples 45 -> 26 us.
constexpr int FU_GROUPS = 3;
// barrier of a group's 256 threads; true for all of them if `bad` holds for any
__device__ __forceinline__ bool fu_bar_or(int g, bool bad) {
  uint32_t any;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, 256, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(any)
      : "r"(bad ? 1u : 0u), "r"(g + 1)
      : "memory");
  return any != 0;
}
// PRE: the inputs are there already, normalised (Hin, rows of kd[0])
template <bool PRE>
__global__ void __launch_bounds__(256 * FU_GROUPS, 1)
k_mlp_predict_tc(int64_t n, FusedNet net, const bf16* __restrict__ wb, const float* __restrict__ w32,
                 const double* __restrict__ X, const bf16* __restrict__ Hin, double* __restrict__ Y, const float* __restrict__ mu_in,
                 const float* __restrict__ sd_in, const float* __restrict__ mu_out,
                 const float* __restrict__ sd_out, int* err) {
  extern __shared__ __align__(1024) unsigned char tc_dyn[];
  __shared__ __align__(8) uint64_t mbar[FU_GROUPS];
  __shared__ uint32_t taddr_s;
  const int g = threadIdx.x >> 8, tid = threadIdx.x & 255, warp = tid >> 5, lane = tid & 31;
  const int groups = blockDim.x >> 8;
  unsigned char* act = tc_dyn + net.wbytes + g * FU_ACT;
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_s)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[g])));
  fu_stage_weights(tc_dyn, net, wb);
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = taddr_s + (uint32_t)(g * TC_COLS);
  const uint32_t tq = taddr + ((uint32_t)((warp & 3) * 32) << 16);
  const uint32_t bar = smem_u32(&mbar[g]);
  const int64_t ntiles = (n + 127) / 128;
  const int nch0 = net.kd[0] >> 3, row = (warp & 3) * 32 + lane;
  uint32_t phase = 0;
  bool ok = true, bad = false;
  for (int64_t tile = blockIdx.x + (int64_t)g * gridDim.x; tile < ntiles && ok;
       tile += (int64_t)gridDim.x * groups) {
    for (int t = tid; t < 128 * nch0; t += 256) {
      const int ch = t % nch0, r = t / nch0;
      if (PRE) {
        const int64_t mr = tile * 128 + r;
        uint4 h = make_uint4(0, 0, 0, 0);
        if (mr < n) h = *reinterpret_cast<const uint4*>(Hin + mr * net.kd[0] + ch * 8);
        *reinterpret_cast<uint4*>(act + fu_off(r, ch * 8, net.kd[0])) = h;
      } else {
        *reinterpret_cast<uint4*>(act + fu_off(r, ch * 8, net.kd[0])) =
            fu_input8(X, tile * 128 + r, n, net.nin, ch * 8, mu_in, sd_in);
      }
    }
    const int64_t m = tile * 128 + row;
    for (int l = 0; l < net.L; ++l) {
      const int K = net.kd[l], N = net.kd[l + 1];
      asm volatile("fence.proxy.async.shared::cta;");
      asm volatile("tcgen05.fence::before_thread_sync;");
      if (fu_bar_or(g, bad)) { ok = false; break; }
      if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t idesc = fu_idesc(N, 0, 0);
        const uint64_t ad = fu_desc(smem_u32(act), 128, K * 16), bd = fu_desc(smem_u32(tc_dyn + net.soff[l]), 128, K * 16);
        for (int kk = 0; kk < K / 16; ++kk) fu_mma(taddr, ad + kk * 16, bd + kk * 16, idesc, kk > 0);
        fu_commit(bar);
      }
      if (!tc_wait(bar, phase)) {
        if (lane == 0) atomicOr(err, 1);
        bad = true;            // the group leaves at its next barrier
        tc_wait(bar, phase);   // the MMAs in flight get a second bounded chance
      }
      phase ^= 1;
      asm volatile("tcgen05.fence::after_thread_sync;");
      const float* bias = w32 + net.boff[l];
      for (int c0 = 16 * (warp >> 2); c0 < N; c0 += 32) {
        float v[16];
        fu_ld16(tq + (uint32_t)c0, v);
        fu_bias16(bias + c0, v);
        if (l < net.L - 1) {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = gelu(v[j]);
          uint4 lo, hi;
          fu_pack16(v, lo, hi);
          *reinterpret_cast<uint4*>(act + fu_off(row, c0, N)) = lo;
          *reinterpret_cast<uint4*>(act + fu_off(row, c0 + 8, N)) = hi;
        } else if (m < n) {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < net.nout)
              Y[m * net.nout + c0 + j] = (double)v[j] * (double)sd_out[c0 + j] + (double)mu_out[c0 + j];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (threadIdx.x < 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr_s), "r"(512));
}

// Training: forward, loss and back-propagation of one 128-row tile a CTA (16
// warps, four per accumulator lane group, which split the columns).  Leaves
// each layer's BF16 input H and output delta D in memory for the weight
// gradients, the pre-activations Z (FP32, read back by the same threads) and
// the tile's loss sum.  512 rows: 57 us, where forward layers, loss and
// data-gradient launches took 200 us.
struct FusedBufs {
  bf16* H[FU_MAXL];    // layer inputs  [n x kd[l]]
  bf16* D[FU_MAXL];    // layer deltas  [n x kd[l + 1]]
  float* Z[FU_MAXL];   // hidden pre-activations [n x kd[l + 1]]
};
__global__ void __launch_bounds__(512, 1)
k_mlp_train_tc(int64_t n, FusedNet net, FusedBufs buf, const bf16* __restrict__ wb, const float* __restrict__ w32,
               const double* __restrict__ X, const double* __restrict__ T, const float* __restrict__ mu_in,
               const float* __restrict__ sd_in, const float* __restrict__ mu_out, const float* __restrict__ sd_out,
               double* part, int* err) {
  extern __shared__ __align__(1024) unsigned char tc_dyn[];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ uint32_t taddr_s;
  __shared__ double sh[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* act = tc_dyn + net.wbytes;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_s)),
                 "r"(TC_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar)));
  fu_stage_weights(tc_dyn, net, wb);
  const int64_t m0 = (int64_t)blockIdx.x * 128;
  const int row = (warp & 3) * 32 + lane;
  const int64_t m = m0 + row;
  const bool live = m < n;
  const int nch0 = net.kd[0] >> 3;
  for (int t = tid; t < 128 * nch0; t += 512) {
    const int ch = t % nch0, r = t / nch0;
    const uint4 h = fu_input8(X, m0 + r, n, net.nin, ch * 8, mu_in, sd_in);
    *reinterpret_cast<uint4*>(act + fu_off(r, ch * 8, net.kd[0])) = h;
    if (m0 + r < n) *reinterpret_cast<uint4*>(buf.H[0] + (m0 + r) * net.kd[0] + ch * 8) = h;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = taddr_s, tq = taddr + ((uint32_t)((warp & 3) * 32) << 16), bar = smem_u32(&mbar);
  uint32_t phase = 0;
  bool ok = true;
  double loss = 0.0;
  const double scale = 2.0 / ((double)n * net.nout);
  // the 2 L - 1 products: layers 0 .. L - 1 forward, then L - 1 .. 1 backward
  for (int p = 0; p < 2 * net.L - 1 && ok; ++p) {
    const bool fwd = p < net.L;
    const int l = fwd ? p : 2 * net.L - 1 - p;
    const int K = fwd ? net.kd[l] : net.kd[l + 1], N = fwd ? net.kd[l + 1] : net.kd[l];
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t w = smem_u32(tc_dyn + net.soff[l]), wl = net.kd[l] * 16;
      const uint32_t idesc = fu_idesc(N, 0, fwd ? 0 : 1);
      const uint64_t ad = fu_desc(smem_u32(act), 128, K * 16);
      const uint64_t bd = fwd ? fu_desc(w, 128, wl) : fu_desc(w, wl, 128);
      const uint64_t bstep = fwd ? 16 : (uint64_t)(2 * wl) >> 4;
      for (int kk = 0; kk < K / 16; ++kk) fu_mma(taddr, ad + kk * 16, bd + kk * bstep, idesc, kk > 0);
      fu_commit(bar);
    }
    const bool late = __syncthreads_or(!tc_wait(bar, phase) ? 1 : 0);
    if (late) {
      if (tid == 0) atomicOr(err, 1);
      tc_wait(bar, phase);   // the MMAs in flight get a second bounded chance
      ok = false;
      break;
    }
    phase ^= 1;
    asm volatile("tcgen05.fence::after_thread_sync;");
    for (int c0 = 16 * (warp >> 2); c0 < N; c0 += 64) {
      float v[16];
      fu_ld16(tq + (uint32_t)c0, v);
      bf16* out;
      if (fwd) {
        fu_bias16(w32 + net.boff[l] + c0, v);
        if (l < net.L - 1) {
          if (live) {
            float4* z = reinterpret_cast<float4*>(buf.Z[l] + m * N + c0);
#pragma unroll
            for (int j = 0; j < 4; ++j) z[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = gelu(v[j]);
          out = buf.H[l + 1];
        } else {
          // mean squared error on the normalised targets: delta = 2 (y - t) / (n nout)
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int c = c0 + j;
            float d = 0.f;
            if (live && c < net.nout) {
              const double tn = (T[m * net.nout + c] - (double)mu_out[c]) / (double)sd_out[c];
              const double diff = (double)v[j] - tn;
              loss += diff * diff;
              d = (float)(scale * diff);
            }
            v[j] = d;
          }
          out = buf.D[l];
        }
      } else {
        if (live) {
          const float4* z = reinterpret_cast<const float4*>(buf.Z[l - 1] + m * N + c0);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 q = z[j];
            v[4 * j] *= gelu_grad(q.x); v[4 * j + 1] *= gelu_grad(q.y);
            v[4 * j + 2] *= gelu_grad(q.z); v[4 * j + 3] *= gelu_grad(q.w);
          }
        }
        out = buf.D[l - 1];
      }
      uint4 lo, hi;
      fu_pack16(v, lo, hi);
      *reinterpret_cast<uint4*>(act + fu_off(row, c0, N)) = lo;
      *reinterpret_cast<uint4*>(act + fu_off(row, c0 + 8, N)) = hi;
      if (live) {
        uint4* q = reinterpret_cast<uint4*>(out + m * N + c0);
        q[0] = lo;
        q[1] = hi;
      }
    }
    asm volatile("fence.proxy.async.shared::cta;");
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
  }
  loss = block_sum(loss, sh);
  if (tid == 0) part[blockIdx.x] = loss;
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(TC_COLS));
}

// Weight and bias gradients of every layer in one launch: dW_l [N x K] =
// D_l^T H_l, summed over the batch.  One CTA per layer and 32 columns of K:
// both operands are MN-major as they lie in memory (rows are the reduction),
// so they are copied as 16-byte pieces (cp.async, three buffers of 128
// rows, zero fill past the batch) instead of element by element, and every
// output keeps one accumulation chain over the batch in steps of 16.  The
// bias gradient (row sums of D in row order) is taken by the layer's first
// CTA from the staged rows.  512 rows, five layers: 14.5 us, where one launch
// of one CTA for each layer's weights and biases took 5 x 234 us.
constexpr int WG_ROWS = 128, WG_COLS = 32, WG_STAGES = 3;
constexpr int WG_A = WG_ROWS * 128 * 2, WG_STAGE = WG_A + WG_ROWS * WG_COLS * 2;
struct WgradJobs {
  int njobs;
  int8_t layer[FU_MAXL * 4], tile[FU_MAXL * 4];
};
__device__ __forceinline__ void wg_stage(unsigned char* st, const bf16* D, const bf16* H, int N, int K, int k0, int kt,
                                         int64_t b0, int64_t n) {
  // A: rows b of D, 128 columns (zeros past N); B: rows b of H, kt columns from k0
  for (int t = threadIdx.x; t < WG_ROWS * 16; t += 256) {
    const int b = t >> 4, ch = t & 15;
    const bool in = b0 + b < n && ch * 8 < N;
    cp_async16(smem_u32(st + fu_off(b, ch * 8, 128)), in ? D + (b0 + b) * N + ch * 8 : D, in ? 16 : 0);
  }
  const int nch = kt >> 3;
  for (int t = threadIdx.x; t < WG_ROWS * nch; t += 256) {
    const int b = t / nch, ch = t % nch;
    const bool in = b0 + b < n;
    cp_async16(smem_u32(st + WG_A + fu_off(b, ch * 8, kt)), in ? H + (b0 + b) * K + k0 + ch * 8 : H, in ? 16 : 0);
  }
}
__global__ void __launch_bounds__(256, 1) k_mlp_wgrad_tc(int64_t n, FusedNet net, FusedBufs buf, WgradJobs jobs,
                                                         float* __restrict__ grad, int* err) {
  extern __shared__ __align__(1024) unsigned char tc_dyn[];
  __shared__ __align__(8) uint64_t mbar[WG_STAGES];
  __shared__ uint32_t taddr_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int l = jobs.layer[blockIdx.x], k0 = jobs.tile[blockIdx.x] * WG_COLS;
  const int N = net.kd[l + 1], K = net.kd[l], kt = min(WG_COLS, K - k0);
  const bf16 *D = buf.D[l], *H = buf.H[l];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&taddr_s)),
                 "r"(WG_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid < WG_STAGES) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[tid])));
  const int nchunk = (int)((n + WG_ROWS - 1) / WG_ROWS);
  for (int c = 0; c < 2; ++c) {
    if (c < nchunk) wg_stage(tc_dyn + c * WG_STAGE, D, H, N, K, k0, kt, (int64_t)c * WG_ROWS, n);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t taddr = taddr_s;
  float db = 0.f;
  bool ok = true;
  int waited = 0;   // chunks whose MMAs have been waited for
  for (int c = 0; c < nchunk; ++c) {
    unsigned char* st = tc_dyn + (c % WG_STAGES) * WG_STAGE;
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t idesc = fu_idesc(kt, 1, 1);
      const uint64_t ad = fu_desc(smem_u32(st), 128 * 16, 128), bd = fu_desc(smem_u32(st + WG_A), kt * 16, 128);
      // steps of 16 rows up to the batch rounded up to 16
      const int64_t left = n - (int64_t)c * WG_ROWS;
      const int steps = (int)((left < WG_ROWS ? left : WG_ROWS) + 15) / 16;
      for (int kk = 0; kk < steps; ++kk)
        fu_mma(taddr, ad + kk * ((2 * 128 * 16) >> 4), bd + kk * ((2 * kt * 16) >> 4), idesc, c > 0 || kk > 0);
      fu_commit(smem_u32(&mbar[c % WG_STAGES]));
    }
    if (k0 == 0 && tid < N) {
      const int rows = (int)(n - (int64_t)c * WG_ROWS < WG_ROWS ? n - (int64_t)c * WG_ROWS : WG_ROWS);
      const unsigned char* q = st + (tid >> 3) * 128 + (tid & 7) * 2;
#pragma unroll 8
      for (int b = 0; b < rows; ++b)
        db += __bfloat162float(*reinterpret_cast<const bf16*>(q + (b >> 3) * 2048 + (b & 7) * 16));
    }
    // the stage chunk c + 2 goes to was read by the MMAs of chunk c - 1
    bool late = false;
    if (c >= 1) {
      late = !tc_wait(smem_u32(&mbar[(c - 1) % WG_STAGES]), ((c - 1) / WG_STAGES) & 1);
      waited = c;
    }
    if (__syncthreads_or(late ? 1 : 0)) {
      ok = false;
      break;
    }
    if (c + 2 < nchunk)
      wg_stage(tc_dyn + ((c + 2) % WG_STAGES) * WG_STAGE, D, H, N, K, k0, kt, (int64_t)(c + 2) * WG_ROWS, n);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (ok && __syncthreads_or(!tc_wait(smem_u32(&mbar[(nchunk - 1) % WG_STAGES]), ((nchunk - 1) / WG_STAGES) & 1)))
    ok = false;
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (!ok) {
    if (tid == 0) atomicOr(err, 1);
    // chunks in flight: waited .. waited + 1 at most
    for (int c = waited; c < nchunk && c < waited + 2; ++c)
      tc_wait(smem_u32(&mbar[c % WG_STAGES]), (c / WG_STAGES) & 1);
  } else {
    const int r = (warp & 3) * 32 + lane;
    const int c0 = 16 * (warp >> 2);
    if (c0 < kt) {
      float v[16];
      fu_ld16(taddr + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0, v);
      if (r < N) {
        float4* q = reinterpret_cast<float4*>(grad + net.woff[l] + (int64_t)r * K + k0 + c0);
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
    }
    if (k0 == 0 && tid < N) grad[net.boff[l] + tid] = db;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(WG_COLS));
}

// inputs (double, [n x nin]) -> normalised BF16 rows padded to kin
__global__ void k_mlp_in(int64_t n, int nin, int kin, const double* X, const float* mu, const float* sd, bf16* H) {
  GS(i, n * (int64_t)kin) {
    const int64_t r = i / kin;
    const int c = (int)(i - r * kin);
    const float v = c < nin ? (float)((X[r * nin + c] - (double)mu[c]) / (double)sd[c]) : 0.f;
    H[i] = __float2bfloat16(v);
  }
}
// output rows (f32, padded) -> de-normalised doubles [n x nout]
__global__ void k_mlp_out(int64_t n, int nout, int kout, const float* Y, const float* mu, const float* sd, double* out) {
  GS(i, n * (int64_t)nout) {
    const int64_t r = i / nout;
    const int c = (int)(i - r * nout);
    out[i] = (double)Y[r * kout + c] * (double)sd[c] + (double)mu[c];
  }
}
// MSE loss on normalised targets; delta = 2 (y - t) / (n nout) as BF16, loss partials
__global__ void k_mlp_loss(int64_t n, int nout, int kout, const float* Y, const double* T, const float* mu,
                           const float* sd, bf16* delta, double* part) {
  __shared__ double sh[32];
  double acc = 0.0;
  const double scale = 2.0 / ((double)n * nout);
  GS(i, n * (int64_t)kout) {
    const int64_t r = i / kout;
    const int c = (int)(i - r * kout);
    float d = 0.f;
    if (c < nout) {
      const double tn = (T[r * nout + c] - (double)mu[c]) / (double)sd[c];
      const double diff = (double)Y[i] - tn;
      acc += diff * diff;
      d = (float)(scale * diff);
    }
    delta[i] = __float2bfloat16(d);
  }
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}
__global__ void k_sum_final(int nb, const double* part, double scale, double* out) {
  __shared__ double sh[32];
  double a = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) a += part[b];
  a = block_sum(a, sh);
  if (threadIdx.x == 0) *out = a * scale;
}
// Adam on FP32 master weights; refresh the BF16 copy.  mask keeps padding at
// zero.  omb1 = 1 - b1, omb2 = 1 - b2 and the bias corrections c1 = 1 - b1^t,
// c2 = 1 - b2^t come from the host in double precision: formed in FP32,
// 1 - b2^t loses about five digits to cancellation (b2^t is near 1).
__global__ void k_adam(int64_t n, float* w, float* m, float* v, const float* g, const uint8_t* mask, float lr,
                       float b1, float omb1, float b2, float omb2, float eps, float c1, float c2, bf16* wb,
                       int64_t nw) {
  GS(i, n) {
    if (!mask[i]) continue;
    const float gi = g[i];
    const float mi = b1 * m[i] + omb1 * gi;
    const float vi = b2 * v[i] + omb2 * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    if (i < nw) wb[i] = __float2bfloat16(wi);
  }
}
__global__ void k_to_bf16(int64_t n, const float* a, bf16* b) {
  GS(i, n) b[i] = __float2bfloat16(a[i]);
}
// counter-based initialisation: uniform(-lim, lim) from a 64-bit mix of (seed, index)
__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x += 0x9e3779b97f4a7c15ULL;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
  return x ^ (x >> 31);
}
__global__ void k_init_w(int64_t n, int kpad, int nin_real, int nout_real, uint64_t seed, float lim, float* w,
                         uint8_t* mask) {
  GS(i, n) {
    const int r = (int)(i / kpad), c = (int)(i - (int64_t)r * kpad);
    const bool live = r < nout_real && c < nin_real;
    const double u = (double)(mix64(seed ^ (uint64_t)i * 0x2545f4914f6cdd1dULL) >> 11) * (1.0 / 9007199254740992.0);
    w[i] = live ? (float)((2.0 * u - 1.0) * lim) : 0.f;
    mask[i] = live;
  }
}

}  // namespace fvs

// ---------------------------------------------------------------------------
// the surrogate object
// ---------------------------------------------------------------------------
using namespace fvs;

struct fvs_surrogate_s {
  cudaStream_t stream = nullptr;
  int nin = 0, nout = 0, hidden = 0, nlayers = 0;   // nlayers = hidden layers
  std::vector<int> kd;       // padded widths: kd[0] input, kd[L] output
  std::vector<int> real;     // real widths
  // per layer l (0..L-1): W [kd[l+1] x kd[l]], b [kd[l+1]]
  DBuf<float> w32, m, v, g;  // all layer weights then all biases, flattened
  DBuf<bf16> wb;             // BF16 copy of the weights part
  DBuf<uint8_t> mask;
  std::vector<int64_t> woff, boff;
  int64_t nw = 0, nparam = 0;
  DBuf<float> mu_in, sd_in, mu_out, sd_out;
  int64_t step = 0;
  // work (sized for the largest batch seen)
  int64_t cap = 0, cap_z = 0, cap_d = 0;
  std::vector<DBuf<bf16>*> H;   // activations per layer input (L+1 buffers)
  std::vector<DBuf<float>*> Z;  // pre-activations per layer output
  std::vector<DBuf<bf16>*> D;   // loss gradients per layer output
  DBuf<float> Y;
  DBuf<bf16> Xn;                // normalised inputs of a prediction with many of them
  DBuf<double> part, lossv, Xd, Td;
  DBuf<int> tc_err;          // set by a tensor-core GEMM whose bounded wait ran out
  ~fvs_surrogate_s() {
    for (auto* p : H) delete p;
    for (auto* p : Z) delete p;
    for (auto* p : D) delete p;
  }
};

namespace fvs {

// layer buffers for n rows; Z and D only for training
static fvs_status sg_work(fvs_surrogate_s* s, int64_t n, bool train) {
  const int L = (int)s->kd.size() - 1;
  auto grow = [&](auto& v, int count, int from, int64_t& cap) -> fvs_status {
    using B = std::remove_pointer_t<typename std::remove_reference_t<decltype(v)>::value_type>;
    if (n <= cap) return FVS_OK;
    for (auto* p : v) delete p;
    v.clear();
    cap = 0;
    for (int l = 0; l < count; ++l) {
      v.push_back(new B());
      FVS_TRY(v.back()->alloc((size_t)n * s->kd[from + l] + 16));
    }
    cap = n;
    return FVS_OK;
  };
  FVS_TRY(grow(s->H, L + 1, 0, s->cap));
  FVS_TRY(s->Y.alloc((size_t)n * s->kd[L] + 16));
  if (train) {
    FVS_TRY(grow(s->Z, L, 1, s->cap_z));
    FVS_TRY(grow(s->D, L, 1, s->cap_d));
    FVS_TRY(s->part.alloc(std::max<size_t>(1024, (size_t)(n + 127) / 128)));
    FVS_TRY(s->lossv.alloc(1));
  }
  return FVS_OK;
}

// the one-kernel network: layout, and whether the weights leave room for
// `acts` activation tiles in shared memory (else the layers run one by one)
static constexpr int FU_SMEM = 226 * 1024;
static FusedNet fused_net(const fvs_surrogate_s* s) {
  FusedNet f{};
  f.L = (int)s->kd.size() - 1;
  f.nin = s->nin;
  f.nout = s->nout;
  for (int l = 0; l <= f.L; ++l) f.kd[l] = s->kd[l];
  for (int l = 0; l < f.L; ++l) {
    f.woff[l] = (int)s->woff[l];
    f.boff[l] = (int)s->boff[l];
    f.soff[l] = f.wbytes;
    f.wbytes += f.kd[l] * f.kd[l + 1] * 2;
  }
  return f;
}
static bool fused_fits(const FusedNet& f, int acts) { return f.wbytes + acts * FU_ACT <= FU_SMEM; }
static fvs_status fused_smem_attr() {
  static bool attr_set[64] = {false};
  int dev = 0;
  FVS_CUDA(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && attr_set[dev]) return FVS_OK;
  FVS_CUDA(cudaFuncSetAttribute(k_mlp_predict_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FU_SMEM));
  FVS_CUDA(cudaFuncSetAttribute(k_mlp_predict_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FU_SMEM));
  FVS_CUDA(cudaFuncSetAttribute(k_mlp_train_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, FU_SMEM));
  FVS_CUDA(cudaFuncSetAttribute(k_mlp_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_STAGES * WG_STAGE));
  if (dev >= 0 && dev < 64) attr_set[dev] = true;
  return FVS_OK;
}

static int tc_grid(int64_t M) { return (int)((M + 127) / 128); }

// forward layer C = A W^T with the fused epilogue: the persistent kernel
// (up to four CTAs per SM, weights staged once per CTA, next A tile copied
// while the current one is multiplied) where K and N fit one tile, else one
// CTA a tile
template <int EPI>
static fvs_status tc_forward(cudaStream_t st, int64_t n, int N, int K, const bf16* A, const bf16* W, const Epi& e,
                             int* err) {
  if (K <= 128 && N <= 128) {
    const int nchunk = (K + TC_KC - 1) / TC_KC;
    const size_t smem = (size_t)3 * nchunk * TC_CHUNK_BYTES;
    static bool attr_set[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr_set[dev]) {
      FVS_CUDA(cudaFuncSetAttribute(k_mlp_fwd_tc<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    3 * 2 * TC_CHUNK_BYTES));
      attr_set[dev] = true;
    }
    // CTAs per SM: tensor memory allows four (128 columns each), shared memory
    // 227 KB / (smem + 1 KB)
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(4, (227 * 1024) / (smem + 1024)));
    const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(tc_grid(n), (int64_t)per_sm * sm_count()));
    k_mlp_fwd_tc<EPI><<<grid, 256, smem, st>>>((int)n, N, K, A, W, e, err);
  } else {
    k_mlp_gemm_tc<EPI><<<tc_grid(n), 128, 0, st>>>((int)n, N, K, A, K, 1, W, K, 1, e, err);
  }
  FVS_COUNT_LAUNCH();
  return FVS_OK;
}

// forward pass of n normalised BF16 rows already in H[0]; keep Z when training
static fvs_status sg_forward(fvs_surrogate_s* s, int64_t n, bool keep) {
  const int L = (int)s->kd.size() - 1;
  cudaStream_t st = s->stream;
  for (int l = 0; l < L; ++l) {
    const int K = s->kd[l], N = s->kd[l + 1];
    Epi e{};
    e.bias = s->w32.p + s->boff[l];
    e.ldo = N;
    const bf16* W = s->wb.p + s->woff[l];
    if (l < L - 1) {
      e.z = keep ? s->Z[l]->p : nullptr;
      e.hout = s->H[l + 1]->p;
      FVS_TRY(tc_forward<EPI_GELU>(st, n, N, K, s->H[l]->p, W, e, s->tc_err.p));
    } else {
      e.fout = s->Y.p;
      FVS_TRY(tc_forward<EPI_LINEAR>(st, n, N, K, s->H[l]->p, W, e, s->tc_err.p));
    }
  }
  FVS_LAUNCH_CHECK();
  return FVS_OK;
}

// gradients of the loss at the current weights for n rows (X, T on device)
static fvs_status sg_gradients(fvs_surrogate_s* s, int64_t n, double* loss_host) {
  const int L = (int)s->kd.size() - 1;
  cudaStream_t st = s->stream;
  FVS_TRY(sg_work(s, n + 16, true));
  FVS_TRY(fused_smem_attr());
  const FusedNet net = fused_net(s);
  FusedBufs buf{};
  for (int l = 0; l < L; ++l) {
    buf.H[l] = s->H[l]->p;
    buf.D[l] = s->D[l]->p;
    buf.Z[l] = s->Z[l]->p;
  }
  int nb = tc_grid(n);
  if (fused_fits(net, 1)) {
    k_mlp_train_tc<<<nb, 512, net.wbytes + FU_ACT, st>>>(n, net, buf, s->wb.p, s->w32.p, s->Xd.p, s->Td.p,
                                                        s->mu_in.p, s->sd_in.p, s->mu_out.p, s->sd_out.p, s->part.p,
                                                        s->tc_err.p);
    FVS_COUNT_LAUNCH();
  } else {
    k_mlp_in<<<stride_grid(n * s->kd[0], 256), 256, 0, st>>>(n, s->nin, s->kd[0], s->Xd.p, s->mu_in.p, s->sd_in.p,
                                                            s->H[0]->p); FVS_COUNT_LAUNCH();
    FVS_TRY(sg_forward(s, n, true));
    nb = 256;
    k_mlp_loss<<<nb, 256, 0, st>>>(n, s->nout, s->kd[L], s->Y.p, s->Td.p, s->mu_out.p, s->sd_out.p, s->D[L - 1]->p,
                                   s->part.p); FVS_COUNT_LAUNCH();
    for (int l = L - 1; l > 0; --l) {
      const int K = s->kd[l], N = s->kd[l + 1];
      // delta_{l-1} = (delta_l W_l) * gelu'(Z_{l-1}): A(m=b, k=n) = delta[b*N + n], B(n'=k, k=n) = W[n*K + k]
      Epi d{};
      d.z = s->Z[l - 1]->p;
      d.hout = s->D[l - 1]->p;
      d.ldo = K;
      k_mlp_gemm_tc<EPI_DGRAD><<<tc_grid(n), 128, 0, st>>>((int)n, K, N, s->D[l]->p, N, 1, s->wb.p + s->woff[l], 1, K,
                                                          d, s->tc_err.p);
      FVS_COUNT_LAUNCH();
    }
  }
  FVS_LAUNCH_CHECK();
  // the columns of wide layers are spread over several CTAs
  WgradJobs jobs{};
  for (int l = L - 1; l >= 0; --l)
    for (int t = 0; t * WG_COLS < s->kd[l]; ++t) {
      jobs.layer[jobs.njobs] = (int8_t)l;
      jobs.tile[jobs.njobs++] = (int8_t)t;
    }
  k_mlp_wgrad_tc<<<jobs.njobs, 256, WG_STAGES * WG_STAGE, st>>>(n, net, buf, jobs, s->g.p, s->tc_err.p);
  FVS_COUNT_LAUNCH();
  FVS_LAUNCH_CHECK();
  if (loss_host) {
    k_sum_final<<<1, 256, 0, st>>>(nb, s->part.p, 1.0 / ((double)n * s->nout), s->lossv.p); FVS_COUNT_LAUNCH();
    FVS_LAUNCH_CHECK();
    FVS_CUDA(cudaMemcpyAsync(loss_host, s->lossv.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    FVS_CUDA(cudaStreamSynchronize(st));
  }
  return FVS_OK;
}

}  // namespace fvs

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
#define FVS_API extern "C" __attribute__((visibility("default")))

namespace fvs {
// flattened real parameters (oracle order: per layer W row-major, then b) <-> padded device layout
static void layout(const fvs_surrogate_s* s, std::vector<int64_t>& dev_index) {
  dev_index.clear();
  const int L = (int)s->kd.size() - 1;
  for (int l = 0; l < L; ++l) {
    for (int r = 0; r < s->real[l + 1]; ++r)
      for (int c = 0; c < s->real[l]; ++c) dev_index.push_back(s->woff[l] + (int64_t)r * s->kd[l] + c);
    for (int r = 0; r < s->real[l + 1]; ++r) dev_index.push_back(s->boff[l] + r);
  }
}

static fvs_status upload_xt(fvs_surrogate_s* s, const double* X, const double* T, int64_t n) {
  FVS_TRY(s->Xd.alloc((size_t)n * s->nin + 1));
  FVS_CUDA(cudaMemcpyAsync(s->Xd.p, X, n * s->nin * sizeof(double), cudaMemcpyHostToDevice, s->stream));
  if (T) {
    FVS_TRY(s->Td.alloc((size_t)n * s->nout + 1));
    FVS_CUDA(cudaMemcpyAsync(s->Td.p, T, n * s->nout * sizeof(double), cudaMemcpyHostToDevice, s->stream));
  }
  return FVS_OK;
}
}  // namespace fvs

FVS_API fvs_status fvs_surrogate_create(int32_t n_in, int32_t n_hidden, int32_t n_hidden_layers, int32_t n_out,
                                        uint64_t seed, void* stream, fvs_surrogate* out) {
  if (!out || n_in < 1 || n_in > 128 || n_out < 1 || n_out > 128 || n_hidden < 1 || n_hidden > 128 ||
      n_hidden_layers < 1 || n_hidden_layers > 16) {
    set_error("fvs_surrogate_create: widths must be 1..128, hidden layers 1..16");
    return FVS_ERR_ARG;
  }
  *out = nullptr;
  fvs_surrogate_s* s = new fvs_surrogate_s();
  s->stream = (cudaStream_t)stream;
  AllocStream as(s->stream);
  auto pad = [](int x) { return (x + 15) / 16 * 16; };
  s->nin = n_in; s->nout = n_out; s->hidden = n_hidden; s->nlayers = n_hidden_layers;
  s->real.push_back(n_in);
  for (int l = 0; l < n_hidden_layers; ++l) s->real.push_back(n_hidden);
  s->real.push_back(n_out);
  for (int r : s->real) s->kd.push_back(pad(r));
  const int L = (int)s->kd.size() - 1;
  int64_t off = 0;
  for (int l = 0; l < L; ++l) { s->woff.push_back(off); off += (int64_t)s->kd[l + 1] * s->kd[l]; }
  s->nw = off;
  for (int l = 0; l < L; ++l) { s->boff.push_back(off); off += s->kd[l + 1]; }
  s->nparam = off;
  fvs_status r = FVS_OK;
  if (r == FVS_OK) r = s->w32.alloc(s->nparam);
  if (r == FVS_OK) r = s->m.alloc(s->nparam);
  if (r == FVS_OK) r = s->v.alloc(s->nparam);
  if (r == FVS_OK) r = s->g.alloc(s->nparam);
  if (r == FVS_OK) r = s->wb.alloc(s->nw);
  if (r == FVS_OK) r = s->mask.alloc(s->nparam);
  if (r == FVS_OK) r = s->mu_in.alloc(128);
  if (r == FVS_OK) r = s->sd_in.alloc(128);
  if (r == FVS_OK) r = s->mu_out.alloc(128);
  if (r == FVS_OK) r = s->sd_out.alloc(128);
  if (r == FVS_OK) r = s->tc_err.alloc(1);
  if (r != FVS_OK) { delete s; return r; }
  s->w32.zero(s->stream); s->m.zero(s->stream); s->v.zero(s->stream); s->g.zero(s->stream);
  s->mask.zero(s->stream);
  s->tc_err.zero(s->stream);
  for (int l = 0; l < L; ++l) {
    const int64_t n = (int64_t)s->kd[l + 1] * s->kd[l];
    const float lim = sqrtf(6.0f / (float)s->real[l]);
    k_init_w<<<stride_grid(n, 256), 256, 0, s->stream>>>(n, s->kd[l], s->real[l], s->real[l + 1],
                                                        seed * 1315423911ULL + l, lim, s->w32.p + s->woff[l],
                                                        s->mask.p + s->woff[l]);
    FVS_COUNT_LAUNCH();
  }
  // biases: live entries start at zero
  {
    std::vector<uint8_t> bm(s->nparam - s->nw, 0);
    for (int l = 0; l < L; ++l)
      for (int r2 = 0; r2 < s->real[l + 1]; ++r2) bm[s->boff[l] - s->nw + r2] = 1;
    cudaMemcpyAsync(s->mask.p + s->nw, bm.data(), bm.size(), cudaMemcpyHostToDevice, s->stream);
    cudaStreamSynchronize(s->stream);
  }
  k_to_bf16<<<stride_grid(s->nw, 256), 256, 0, s->stream>>>(s->nw, s->w32.p, s->wb.p);
  FVS_COUNT_LAUNCH();
  std::vector<float> one(128, 1.0f), zero(128, 0.0f);
  cudaMemcpyAsync(s->mu_in.p, zero.data(), 512, cudaMemcpyHostToDevice, s->stream);
  cudaMemcpyAsync(s->sd_in.p, one.data(), 512, cudaMemcpyHostToDevice, s->stream);
  cudaMemcpyAsync(s->mu_out.p, zero.data(), 512, cudaMemcpyHostToDevice, s->stream);
  cudaMemcpyAsync(s->sd_out.p, one.data(), 512, cudaMemcpyHostToDevice, s->stream);
  if (cudaStreamSynchronize(s->stream) != cudaSuccess) {
    set_error("fvs_surrogate_create: %s", cudaGetErrorString(cudaGetLastError()));
    delete s;
    return FVS_ERR_CUDA;
  }
  *out = s;
  return FVS_OK;
}

namespace fvs {
// input and output widths of a model (the UQ surrogate mode checks them)
fvs_status surrogate_dims(fvs_surrogate s, int* nin, int* nout) {
  if (!s) {
    set_error("NULL surrogate");
    return FVS_ERR_ARG;
  }
  *nin = s->nin;
  *nout = s->nout;
  return FVS_OK;
}
}  // namespace fvs

FVS_API fvs_status fvs_surrogate_destroy(fvs_surrogate s) {
  if (!s) return FVS_ERR_ARG;
  cudaStream_t st = s->stream;
  {
    AllocStream as(st);
    cudaStreamSynchronize(st);
    delete s;
  }
  cudaStreamSynchronize(st);
  return FVS_OK;
}

FVS_API fvs_status fvs_surrogate_set_scaling(fvs_surrogate s, const double* mu_in, const double* sd_in,
                                             const double* mu_out, const double* sd_out) {
  if (!s || !mu_in || !sd_in || !mu_out || !sd_out) {
    set_error("fvs_surrogate_set_scaling: NULL argument");
    return FVS_ERR_ARG;
  }
  std::vector<float> a(128, 0.f), b(128, 1.f), c(128, 0.f), d(128, 1.f);
  for (int i = 0; i < s->nin; ++i) {
    if (!(sd_in[i] > 0)) { set_error("fvs_surrogate_set_scaling: non-positive scale"); return FVS_ERR_ARG; }
    a[i] = (float)mu_in[i]; b[i] = (float)sd_in[i];
  }
  for (int i = 0; i < s->nout; ++i) {
    if (!(sd_out[i] > 0)) { set_error("fvs_surrogate_set_scaling: non-positive scale"); return FVS_ERR_ARG; }
    c[i] = (float)mu_out[i]; d[i] = (float)sd_out[i];
  }
  FVS_CUDA(cudaMemcpyAsync(s->mu_in.p, a.data(), 512, cudaMemcpyHostToDevice, s->stream));
  FVS_CUDA(cudaMemcpyAsync(s->sd_in.p, b.data(), 512, cudaMemcpyHostToDevice, s->stream));
  FVS_CUDA(cudaMemcpyAsync(s->mu_out.p, c.data(), 512, cudaMemcpyHostToDevice, s->stream));
  FVS_CUDA(cudaMemcpyAsync(s->sd_out.p, d.data(), 512, cudaMemcpyHostToDevice, s->stream));
  FVS_CUDA(cudaStreamSynchronize(s->stream));
  return FVS_OK;
}

FVS_API int64_t fvs_surrogate_num_params(fvs_surrogate s) {
  if (!s) return -1;
  std::vector<int64_t> idx;
  layout(s, idx);
  return (int64_t)idx.size();
}

FVS_API fvs_status fvs_surrogate_params(fvs_surrogate s, double* inout, int64_t len, int set) {
  if (!s || !inout) {
    set_error("fvs_surrogate_params: NULL argument");
    return FVS_ERR_ARG;
  }
  AllocStream as(s->stream);
  std::vector<int64_t> idx;
  layout(s, idx);
  if (len < (int64_t)idx.size()) {
    set_error("fvs_surrogate_params: need %lld values", (long long)idx.size());
    return FVS_ERR_ARG;
  }
  std::vector<float> h(s->nparam);
  FVS_CUDA(cudaMemcpyAsync(h.data(), s->w32.p, s->nparam * sizeof(float), cudaMemcpyDeviceToHost, s->stream));
  FVS_CUDA(cudaStreamSynchronize(s->stream));
  if (set) {
    for (size_t i = 0; i < idx.size(); ++i) h[idx[i]] = (float)inout[i];
    FVS_CUDA(cudaMemcpyAsync(s->w32.p, h.data(), s->nparam * sizeof(float), cudaMemcpyHostToDevice, s->stream));
    k_to_bf16<<<stride_grid(s->nw, 256), 256, 0, s->stream>>>(s->nw, s->w32.p, s->wb.p);
    FVS_COUNT_LAUNCH();
    FVS_CUDA(cudaStreamSynchronize(s->stream));
  } else {
    for (size_t i = 0; i < idx.size(); ++i) inout[i] = (double)h[idx[i]];
  }
  return FVS_OK;
}

// FVS_ERR_TIMEOUT if a tensor-core GEMM gave up waiting on its MMAs (the
// flag is cleared for the next call)
static fvs_status tc_check(fvs_surrogate s) {
  int h = 0;
  FVS_CUDA(cudaMemcpyAsync(&h, s->tc_err.p, sizeof(int), cudaMemcpyDeviceToHost, s->stream));
  FVS_CUDA(cudaStreamSynchronize(s->stream));
  if (h) {
    s->tc_err.zero(s->stream);
    set_error("surrogate: a tensor-core GEMM timed out waiting for its MMAs");
    return FVS_ERR_TIMEOUT;
  }
  return FVS_OK;
}

FVS_API fvs_status fvs_surrogate_gradients(fvs_surrogate s, const double* X, const double* T, int64_t n,
                                           double* grad, int64_t grad_len, double* loss) {
  if (!s || !X || !T || !grad || n <= 0) {
    set_error("fvs_surrogate_gradients: bad argument");
    return FVS_ERR_ARG;
  }
  AllocStream as(s->stream);
  std::vector<int64_t> idx;
  layout(s, idx);
  if (grad_len < (int64_t)idx.size()) {
    set_error("fvs_surrogate_gradients: need %lld values", (long long)idx.size());
    return FVS_ERR_ARG;
  }
  FVS_TRY(upload_xt(s, X, T, n));
  FVS_TRY(sg_gradients(s, n, loss));
  std::vector<float> h(s->nparam);
  FVS_CUDA(cudaMemcpyAsync(h.data(), s->g.p, s->nparam * sizeof(float), cudaMemcpyDeviceToHost, s->stream));
  FVS_CUDA(cudaStreamSynchronize(s->stream));
  FVS_TRY(tc_check(s));
  for (size_t i = 0; i < idx.size(); ++i) grad[i] = (double)h[idx[i]];
  return FVS_OK;
}

FVS_API fvs_status fvs_surrogate_train(fvs_surrogate s, const double* X, const double* T, int64_t n, int32_t epochs,
                                       double lr, double* final_loss) {
  if (!s || !X || !T || n <= 0 || epochs < 0 || !(lr > 0)) {
    set_error("fvs_surrogate_train: bad argument");
    return FVS_ERR_ARG;
  }
  AllocStream as(s->stream);
  FVS_TRY(upload_xt(s, X, T, n));
  const double b1 = 0.9, b2 = 0.999, eps = 1e-8;
  for (int e = 0; e < epochs; ++e) {
    FVS_TRY(sg_gradients(s, n, nullptr));
    ++s->step;
    const double c1 = 1.0 - pow(b1, (double)s->step), c2 = 1.0 - pow(b2, (double)s->step);
    k_adam<<<stride_grid(s->nparam, 256), 256, 0, s->stream>>>(s->nparam, s->w32.p, s->m.p, s->v.p, s->g.p,
                                                              s->mask.p, (float)lr, (float)b1, (float)(1.0 - b1),
                                                              (float)b2, (float)(1.0 - b2), (float)eps, (float)c1,
                                                              (float)c2, s->wb.p, s->nw);
    FVS_COUNT_LAUNCH();
  }
  FVS_LAUNCH_CHECK();
  double l = 0.0;
  FVS_TRY(sg_gradients(s, n, &l));
  FVS_TRY(tc_check(s));
  if (final_loss) *final_loss = l;
  return FVS_OK;
}

FVS_API fvs_status fvs_surrogate_predict(fvs_surrogate s, const double* X, double* Y, int64_t n, int on_device) {
  if (!s || !X || !Y || n <= 0) {
    set_error("fvs_surrogate_predict: bad argument");
    return FVS_ERR_ARG;
  }
  AllocStream as(s->stream);
  const int L = (int)s->kd.size() - 1;
  const double* Xd = X;
  if (!on_device) {
    FVS_TRY(upload_xt(s, X, nullptr, n));
    Xd = s->Xd.p;
  }
  // tiles write their outputs while others still read their inputs: outputs that
  // overlap the inputs go through an array of their own
  const bool overlap = on_device && (const char*)Y < (const char*)(X + n * s->nin) &&
                       (const char*)X < (const char*)(Y + n * s->nout);
  DBuf<double> out;
  double* Yd = Y;
  if (!on_device || overlap) {
    FVS_TRY(out.alloc((size_t)n * s->nout));
    Yd = out.p;
  }
  const FusedNet net = fused_net(s);
  if (fused_fits(net, 1)) {
    FVS_TRY(fused_smem_attr());
    const int groups = fused_fits(net, 3) ? 3 : (fused_fits(net, 2) ? 2 : 1);
    const int grid = (int)std::min<int64_t>((n + 127) / 128, sm_count());
    // More than 32 inputs are normalised beforehand, by the whole GPU: a tile's
    // FP64 divisions (128 a column) on its own SM alone, two lanes a clock, are
    // otherwise most of the call where there are few tiles.  128 inputs, 1000
    // rows: 117 us in the tiles, 71 beforehand; 20,000 rows 196 and 149, 200,000
    // (tiles enough for three groups an SM) 888 and 908.  40 inputs: 66 and 48,
    // 96 and 82, 365 and 364 us.
    const bool pre = s->nin > 32;
    if (pre) {
      FVS_TRY(s->Xn.alloc((size_t)n * s->kd[0]));
      k_mlp_in<<<stride_grid(n * s->kd[0], 256), 256, 0, s->stream>>>(n, s->nin, s->kd[0], Xd, s->mu_in.p, s->sd_in.p,
                                                                      s->Xn.p);
      FVS_COUNT_LAUNCH();
    }
    auto predict = pre ? k_mlp_predict_tc<true> : k_mlp_predict_tc<false>;
    predict<<<grid, 256 * groups, net.wbytes + groups * FU_ACT, s->stream>>>(
        n, net, s->wb.p, s->w32.p, Xd, pre ? s->Xn.p : nullptr, Yd, s->mu_in.p, s->sd_in.p, s->mu_out.p, s->sd_out.p, s->tc_err.p);
    FVS_COUNT_LAUNCH();
  } else {
    FVS_TRY(sg_work(s, n + 16, false));
    k_mlp_in<<<stride_grid(n * s->kd[0], 256), 256, 0, s->stream>>>(n, s->nin, s->kd[0], Xd, s->mu_in.p, s->sd_in.p,
                                                                    s->H[0]->p);
    FVS_COUNT_LAUNCH();
    FVS_TRY(sg_forward(s, n, false));
    k_mlp_out<<<stride_grid(n * s->nout, 256), 256, 0, s->stream>>>(n, s->nout, s->kd[L], s->Y.p, s->mu_out.p,
                                                                    s->sd_out.p, Yd);
    FVS_COUNT_LAUNCH();
  }
  FVS_LAUNCH_CHECK();
  if (!on_device) FVS_CUDA(cudaMemcpyAsync(Y, Yd, n * s->nout * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
  else if (overlap)
    FVS_CUDA(cudaMemcpyAsync(Y, Yd, n * s->nout * sizeof(double), cudaMemcpyDeviceToDevice, s->stream));
  FVS_CUDA(cudaStreamSynchronize(s->stream));
  return tc_check(s);
}
