// Learned bandwidth proposal.  The paper points to fast bandwidth selection
// with the same FFT machinery (Sec. 1, Sec. 5); the network is not from the
// paper.  This file holds its GPU side:
//   - sample standardisation and features (moments, and a 32 x 32 block
//     downsampling of the binned grid of the standardised samples);
//   - a three-layer MLP (ReLU) with BF16 operands and FP32 accumulation,
//     trained with Adam on FP32 master weights.  Every matrix product runs on
//     the 5th-generation tensor cores: tcgen05.mma issued by one thread per
//     CTA, operands staged in shared memory by cp.async, accumulators in
//     tensor memory read back with tcgen05.ld for fused epilogues (bias,
//     ReLU, ReLU gradient, BF16 and transposed BF16 copies).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <random>
#include <vector>

#include "kde_internal.h"
#include "pdl.cuh"
#include "smem_limit.cuh"
#include "tc_wait.cuh"

namespace kde {
namespace {

using bf16 = __nv_bfloat16;

// ---------------------------------------------------------------------------
// Tensor-core GEMM: D[M x N] = A[M x K] B[N x K]^T, A and B K-major BF16,
// FP32 accumulation.  CTA tile 128 x BN, K in steps of 64 (four MMAs of
// K = 16).  Tiles sit in shared memory in the no-swizzle canonical layout:
// core matrices of 8 rows x 16 bytes, element (r, k) at byte
// (r/8) 1024 + (k/8) 128 + (r%8) 16 + (k%8) 2, i.e. 128 bytes between
// K-adjacent core matrices (leading byte offset) and 1024 bytes between
// 8-row groups (stride byte offset).  Sizes: M % 128 == 0, N % BN == 0,
// K % 64 == 0, row strides multiples of 8 elements, 16-byte aligned bases.
// ---------------------------------------------------------------------------
enum Epi { EPI_STORE = 0, EPI_BIAS_RELU = 1, EPI_BIAS = 2, EPI_RELU_GRAD = 3 };

struct GemmArgs {
  const bf16* A;
  int lda;
  const bf16* B;
  int ldb;
  int M, N, K;
  float* C;            // FP32 result after the epilogue (pre-activation for BIAS_RELU)
  int ldc;
  const float* bias;   // BIAS_RELU, BIAS: per column
  const float* Z;      // RELU_GRAD: D is multiplied by (Z > 0)
  int ldz;
  bf16* Cb;            // optional BF16 copy of the activation / gradient, row-major
  int ldcb;
  bf16* Ct;            // optional BF16 transposed copy: Ct[n ldct + m]
  int ldct;
  int* status;         // set to 1 if a wait for the tensor cores gave up
  int epi;
  bool vec;            // C, Z, Cb rows take 16-byte accesses
};
// Two independent products may share a launch (blockIdx.z).
struct GemmPair {
  GemmArgs g[2];
};


__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor: start >> 4 (bits 0-13), leading byte
// offset >> 4 (16-29), stride byte offset >> 4 (32-45), descriptor version
// 1 (bit 46), base offset 0, no swizzle.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(128u >> 4) << 16) |
         ((uint64_t)(1024u >> 4) << 32) | (1ull << 46);
}

// Stage the 64-wide K slice k0 of A's rows m0.. and B's rows n0.. into one
// shared-memory stage with 16-byte cp.async copies (one commit group).
template <int BN>
__device__ __forceinline__ void stage_tiles(const GemmArgs& g, uint8_t* sA, uint8_t* sB, int m0,
                                            int n0, int k0) {
  const int tid = threadIdx.x;
  for (int i = tid; i < 128 * 8; i += 128) {
    const int r = i >> 3, c = i & 7;
    const size_t src = __cvta_generic_to_global(g.A + (size_t)(m0 + r) * g.lda + k0 + 8 * c);
    const uint32_t dst = smem_u32(sA + (r >> 3) * 1024 + c * 128 + (r & 7) * 16);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  for (int i = tid; i < BN * 8; i += 128) {
    const int r = i >> 3, c = i & 7;
    const size_t src = __cvta_generic_to_global(g.B + (size_t)(n0 + r) * g.ldb + k0 + 8 * c);
    const uint32_t dst = smem_u32(sB + (r >> 3) * 1024 + c * 128 + (r & 7) * 16);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// kStages shared-memory stages: the copies of the next kStages - 1 K slices
// are in flight while the tensor cores work on one; a stage is refilled only
// after the MMAs that read it have completed (its mbarrier).  The network's
// products are a few CTAs each, so a slice's copy latency is their time: with
// two stages the 256 x 256 x 1088 product took 17 us, 1 us a slice (figures
// at mlp_backward).  The slices are accumulated in the same order whatever
// the stages.
template <int BN, int kStages>
__global__ void __launch_bounds__(128) kde_gemm_tc_kernel(GemmPair pair) {
  extern __shared__ __align__(1024) uint8_t smem[];
  constexpr int kStageBytes = 16384 + BN * 128;  // A 128 x 64 + B BN x 64, BF16
  __shared__ __align__(8) uint64_t mbar[kStages];
  __shared__ uint32_t tmem_slot;
  constexpr uint32_t kCols = BN < 32 ? 32 : BN;  // TMEM columns: a power of two >= 32
  const GemmArgs g = pair.g[blockIdx.z];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * 128, n0 = blockIdx.y * BN;
  pdl_trigger();
  if (m0 >= g.M || n0 >= g.N) return;   // the smaller product of a pair
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int b = 0; b < kStages; ++b)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mbar[b])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  // operands and Z come from the kernels before this one
  pdl_wait();
  // kind::f16 instruction descriptor: D FP32 (bits 4-5 = 1), A and B BF16
  // (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                         ((uint32_t)(128 >> 4) << 24);
  uint32_t phase = 0u, used = 0u;  // bit b: stage b's barrier phase / MMAs pending
  bool ok = true;
  const int nk = g.K / 64;
  auto stage = [&](int kt) {       // one commit group per slice, empty past the last
    if (kt < nk)
      stage_tiles<BN>(g, smem + (kt % kStages) * kStageBytes,
                      smem + (kt % kStages) * kStageBytes + 16384, m0, n0, kt * 64);
    else
      asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int kt = 0; kt < kStages - 1; ++kt) stage(kt);
  for (int kt = 0; kt < nk; ++kt) {
    const int st = kt % kStages;
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    // the tensor cores read shared memory through the async proxy
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t a0 = smem_u32(smem + st * kStageBytes), b0 = a0 + 16384u;
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint64_t da = umma_desc(a0 + 256u * s);
        const uint64_t db = umma_desc(b0 + 256u * s);
        const uint32_t acc = (kt > 0 || s > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(acc)
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_u32(&mbar[st]))
          : "memory");
    }
    used |= 1u << st;
    if (kt + kStages - 1 < nk) {
      // the stage to refill was read by the MMAs of slice kt - 1: wait for them
      const int nx = (kt + kStages - 1) % kStages;
      if ((used >> nx) & 1u) {
        const bool done = mbar_wait(smem_u32(&mbar[nx]), (phase >> nx) & 1u);
        if (!__syncthreads_and(done)) {
          ok = false;
          break;
        }
        phase ^= 1u << nx;
        used &= ~(1u << nx);
      }
    }
    stage(kt + kStages - 1);
  }
  // every MMA has been committed; the last commit tracks them all
  if (ok) {
    const int last = (nk - 1) % kStages;
    const bool done = mbar_wait(smem_u32(&mbar[last]), (phase >> last) & 1u);
    ok = __syncthreads_and(done);
  }
  if (!ok) {
    if (tid == 0) atomicExch(g.status, 1);
    // one more bounded chance for the MMAs in flight before TMEM is freed
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    for (int b = 0; b < kStages; ++b)
      if ((used >> b) & 1u) mbar_wait(smem_u32(&mbar[b]), (phase >> b) & 1u);
  }
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (ok) {
    const int row = m0 + warp * 32 + lane;
#pragma unroll 1
    for (int c0 = 0; c0 < BN; c0 += 16) {
      uint32_t v[16];
      const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "
          "[%16];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
            "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
            "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(taddr)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int n = n0 + c0;
      float x[16], z[16];
      float* crow = g.C + (size_t)row * g.ldc + n;
      if (g.epi == EPI_RELU_GRAD) {
        const float* zrow = g.Z + (size_t)row * g.ldz + n;
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
          const float4 q = g.vec ? *reinterpret_cast<const float4*>(zrow + j)
                                 : make_float4(zrow[j], zrow[j + 1], zrow[j + 2], zrow[j + 3]);
          z[j] = q.x, z[j + 1] = q.y, z[j + 2] = q.z, z[j + 3] = q.w;
        }
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        x[j] = __uint_as_float(v[j]);
        if (g.epi == EPI_BIAS_RELU || g.epi == EPI_BIAS) x[j] += g.bias[n + j];
        if (g.epi == EPI_RELU_GRAD) x[j] = z[j] > 0.f ? x[j] : 0.f;
      }
#pragma unroll
      for (int j = 0; j < 16; j += 4) {
        if (g.vec) {
          *reinterpret_cast<float4*>(crow + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) crow[j + i] = x[j + i];
        }
      }
      if (g.epi == EPI_BIAS_RELU || g.epi == EPI_RELU_GRAD) {
        __align__(16) bf16 b[16];
#pragma unroll
        for (int j = 0; j < 16; ++j)
          b[j] = __float2bfloat16_rn(g.epi == EPI_BIAS_RELU ? fmaxf(x[j], 0.f) : x[j]);
        if (g.Cb) {   // rows of the network's own buffers: always 16-byte aligned
          uint4* dst = reinterpret_cast<uint4*>(g.Cb + (size_t)row * g.ldcb + n);
          dst[0] = reinterpret_cast<const uint4*>(b)[0];
          dst[1] = reinterpret_cast<const uint4*>(b)[1];
        }
        if (g.Ct) {
#pragma unroll
          for (int j = 0; j < 16; ++j) g.Ct[(size_t)(n + j) * g.ldct + row] = b[j];
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols)
                 : "memory");
}

template <int BN, int kStages>
cudaError_t launch_gemm_st(const GemmPair& p, dim3 grid, cudaStream_t st) {
  // kStages stages of A (16 KB) and B (BN x 128 bytes); the narrow tiles ask
  // for as much as the wide ones, so that at most four CTAs share an SM and
  // their tensor memory (64 columns each) stays within its 512 columns.
  const int smem = kStages * (16384 + 64 * 128);
  cudaError_t e = allow_smem(kde_gemm_tc_kernel<BN, kStages>);
  if (e != cudaSuccess) return e;
  LaunchScope ls("kde_gemm_tc_kernel", st);
  e = launch_pdl(kde_gemm_tc_kernel<BN, kStages>, grid, dim3(128), (size_t)smem, st, p);
  return e == cudaSuccess ? cudaGetLastError() : e;
}

// Grids that leave SMs idle take eight stages (196 KB, one CTA an SM); larger
// ones two (four CTAs an SM, one's epilogue beside the others' slices: 4096^3
// 776 us, 792 with three stages, 889 with four).
template <int BN>
cudaError_t launch_gemm_bn(const GemmPair& p, int count, cudaStream_t st) {
  int M = 0, N = 0;
  for (int i = 0; i < count; ++i) {
    M = std::max(M, p.g[i].M);
    N = std::max(N, p.g[i].N);
  }
  const dim3 grid((unsigned)(M / 128), (unsigned)(N / BN), (unsigned)count);
  if ((int64_t)grid.x * grid.y * grid.z <= 128) return launch_gemm_st<BN, 8>(p, grid, st);
  return launch_gemm_st<BN, 2>(p, grid, st);
}

kde_status check_gemm(GemmArgs& g, int epi) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.M % 128 || g.N % 16 || g.K % 64 || g.lda % 8 ||
      g.ldb % 8 || ((uintptr_t)g.A & 15) || ((uintptr_t)g.B & 15) || !g.C || !g.status)
    return fail(KDE_ERR_INVALID_ARG,
                "tensor-core GEMM: need M % 128 == 0, N % 16 == 0, K % 64 == 0, row strides "
                "multiples of 8 elements and 16-byte aligned operands");
  g.epi = epi;
  g.vec = g.ldc % 4 == 0 && ((uintptr_t)g.C & 15) == 0 && (!g.Z || (g.ldz % 4 == 0 && ((uintptr_t)g.Z & 15) == 0));
  return KDE_OK;
}

kde_status launch_gemm(GemmArgs g, int epi, cudaStream_t st) {
  const kde_status s = check_gemm(g, epi);
  if (s != KDE_OK) return s;
  GemmPair p{};
  p.g[0] = g;
  const cudaError_t e = g.N % 64 == 0 ? launch_gemm_bn<64>(p, 1, st) : launch_gemm_bn<16>(p, 1, st);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_gemm_tc_kernel");
}

// Two products of N % 64 == 0 in one launch.
kde_status launch_gemm2(GemmArgs a, int epi_a, GemmArgs b, int epi_b, cudaStream_t st) {
  kde_status s = check_gemm(a, epi_a);
  if (s == KDE_OK) s = check_gemm(b, epi_b);
  if (s != KDE_OK) return s;
  GemmPair p{};
  p.g[0] = a;
  p.g[1] = b;
  const cudaError_t e = launch_gemm_bn<64>(p, 2, st);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_gemm_tc_kernel");
}

// ---------------------------------------------------------------------------
// Element-wise and reduction kernels of the MLP.
// ---------------------------------------------------------------------------
// X (B x in, FP32) -> Xb (Bp x in, BF16) and its transpose Xt (in x Bp);
// rows B .. Bp-1 are zero.  Tiles of 32 x 64 go through shared memory, so that
// both copies are written in rows.  One block a tile, (in / 64) (Bp / 32) along
// x: a batch may have more rows than the other grid dimensions take tiles.
__global__ void __launch_bounds__(256) kde_mlp_cast_kernel(const float* __restrict__ X, int B,
                                                           int Bp, int in, bf16* __restrict__ Xb,
                                                           bf16* __restrict__ Xt) {
  __shared__ bf16 tile[32][66];
  pdl_trigger();
  pdl_wait();   // X, and the last reader of Xb and Xt
  const int cols = in / 64, k0 = (int)(blockIdx.x % cols) * 64, b0 = (int)(blockIdx.x / cols) * 32,
            t = threadIdx.x;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int b = (t >> 6) + 4 * i, k = t & 63;
    const bf16 v = __float2bfloat16_rn(b0 + b < B ? X[(size_t)(b0 + b) * in + k0 + k] : 0.f);
    Xb[(size_t)(b0 + b) * in + k0 + k] = v;
    tile[b][k] = v;
  }
  if (!Xt) return;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = (t >> 5) + 8 * i, b = t & 31;
    Xt[(size_t)(k0 + k) * Bp + b0 + b] = tile[b][k];
  }
}

// Loss = (1/B) sum_{b < B, j < out} (Y - T)^2 and its gradient
// dY = (2/B)(Y - T): BF16 copies dYb (Bp x 64, zero beyond out) and
// dYt (outp x Bp), and db3 = sum_b dY (FP32, b in order).  One block, tiles
// of 256 rows: the gradient's values are formed side by side into shared
// memory, and only their additions are one after another (read one by one
// from global memory they took 44 us for 256 rows).
constexpr int kMaxOut = 16;
__global__ void __launch_bounds__(256) kde_mlp_loss_kernel(const float* __restrict__ Y, int ldy,
                                                           const float* __restrict__ T, int B,
                                                           int Bp, int out, int outp,
                                                           bf16* __restrict__ dYb,
                                                           bf16* __restrict__ dYt,
                                                           float* __restrict__ db3,
                                                           float* __restrict__ loss) {
  __shared__ double part[256];
  __shared__ float res[256][kMaxOut + 1], grd[256][kMaxOut + 1];   // Y - T, 2 (Y - T) / B
  pdl_trigger();
  pdl_wait();
  const int t = threadIdx.x;
  double acc = 0.0;
  float sum = 0.f;
  for (int b0 = 0; b0 < Bp; b0 += 256) {
    const int b = b0 + t;
    if (b < Bp) {
      __align__(16) bf16 row[kMaxOut];
#pragma unroll
      for (int j = 0; j < kMaxOut; ++j) {
        float r = 0.f, g = 0.f;
        if (b < B && j < out) {
          r = Y[(size_t)b * ldy + j] - T[(size_t)b * out + j];
          g = 2.f * r / (float)B;
        }
        res[t][j] = r;
        grd[t][j] = g;
        row[j] = __float2bfloat16_rn(g);
        if (j < outp) dYt[(size_t)j * Bp + b] = row[j];
      }
      uint4* dst = reinterpret_cast<uint4*>(dYb + (size_t)b * 64);
      dst[0] = reinterpret_cast<const uint4*>(row)[0];
      dst[1] = reinterpret_cast<const uint4*>(row)[1];
#pragma unroll
      for (int q = 2; q < 8; ++q) dst[q] = make_uint4(0, 0, 0, 0);
    }
    __syncthreads();
    const int nb = min(256, B - b0);
    // thread (t / 64, t mod 64): output t mod 64 of every fourth row
    if ((t & 63) < out)
      for (int i = t >> 6; i < nb; i += 4) {
        const float r = res[i][t & 63];
        acc += (double)r * r;
      }
    if (t < out) {
#pragma unroll 8
      for (int i = 0; i < nb; ++i) sum += grd[i][t];
    }
    __syncthreads();
  }
  part[t] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (t < s) part[t] += part[t + s];
    __syncthreads();
  }
  if (t == 0 && loss) *loss = (float)(part[0] / B);
  if (t < out) db3[t] = sum;
}

// The gradients that are not products, in one launch: db1 and db2 as the
// column sums of dZ1 and dZ2 (a thread a column, b in order, 32 loads in
// flight), and G_W3[j h] = dW3t[h j] for j < out.  Blocks of 32 threads: hid /
// 32 for each of db1 and db2, then out hid / 32.
__global__ void __launch_bounds__(32) kde_mlp_tail_kernel(const float* __restrict__ dZ1,
                                                          const float* __restrict__ dZ2, int hid,
                                                          int B, const float* __restrict__ dW3t,
                                                          int outp, int out,
                                                          float* __restrict__ db1,
                                                          float* __restrict__ db2,
                                                          float* __restrict__ gW3) {
  pdl_trigger();
  pdl_wait();
  const int nb = hid / 32, i = (blockIdx.x % nb) * 32 + threadIdx.x, part = blockIdx.x / nb;
  if (part < 2) {
    const float* dZ = (part ? dZ2 : dZ1) + i;
    float s = 0.f;
#pragma unroll 32
    for (int b = 0; b < B; ++b) s += dZ[(size_t)b * hid];
    (part ? db2 : db1)[i] = s;
  } else {
    gW3[(part - 2) * hid + i] = dW3t[(size_t)i * outp + part - 2];
  }
}

// Adam on the flat FP32 parameters.
__global__ void __launch_bounds__(256) kde_mlp_adam_kernel(float* __restrict__ P,
                                                           const float* __restrict__ G,
                                                           float* __restrict__ Mo,
                                                           float* __restrict__ Vo, int64_t n,
                                                           float lr, float b1, float b2, float eps,
                                                           float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float g = G[i];
    const float m = b1 * Mo[i] + (1.f - b1) * g;
    const float v = b2 * Vo[i] + (1.f - b2) * g * g;
    Mo[i] = m;
    Vo[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
  }
}

// BF16 working copies of the weights: W1b (hid x in), W2b (hid x hid),
// W2t (hid x hid, transposed), W3b (outp x hid, zero rows beyond out),
// W3t (hid x 64: W3t[h j] = W3[j h] for j < out, else 0), b3p (outp).
__global__ void __launch_bounds__(256) kde_mlp_refresh_kernel(
    const float* __restrict__ W1, const float* __restrict__ W2, const float* __restrict__ W3,
    const float* __restrict__ b3, int in, int hid, int out, int outp, bf16* __restrict__ W1b,
    bf16* __restrict__ W2b, bf16* __restrict__ W2t, bf16* __restrict__ W3b,
    bf16* __restrict__ W3t, float* __restrict__ b3p) {
  const int64_t n1 = (int64_t)hid * in, n2 = (int64_t)hid * hid, n3 = (int64_t)outp * hid,
                n4 = (int64_t)hid * 64;
  const int64_t total = n1 + n2 + n3 + n4 + outp;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i < n1) {
      W1b[i] = __float2bfloat16_rn(W1[i]);
    } else if (i < n1 + n2) {
      const int64_t t = i - n1;
      const int r = (int)(t / hid), c = (int)(t % hid);
      const bf16 v = __float2bfloat16_rn(W2[t]);
      W2b[t] = v;
      W2t[(int64_t)c * hid + r] = v;
    } else if (i < n1 + n2 + n3) {
      const int64_t t = i - n1 - n2;
      const int j = (int)(t / hid);
      W3b[t] = __float2bfloat16_rn(j < out ? W3[t] : 0.f);
    } else if (i < n1 + n2 + n3 + n4) {
      const int64_t t = i - n1 - n2 - n3;
      const int h = (int)(t / 64), j = (int)(t % 64);
      W3t[t] = __float2bfloat16_rn(j < out ? W3[(int64_t)j * hid + h] : 0.f);
    } else {
      const int j = (int)(i - n1 - n2 - n3 - n4);
      b3p[j] = j < out ? b3[j] : 0.f;
    }
  }
}

// Y[b j] (b < B, j < out) from the padded output.
__global__ void __launch_bounds__(256) kde_mlp_take_kernel(const float* __restrict__ Yp, int ldy,
                                                           int B, int out, float* __restrict__ Y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * out) return;
  Y[i] = Yp[(size_t)(i / out) * ldy + (i % out)];
}

// ---------------------------------------------------------------------------
// Standardisation and features (d = 2).  FP64 arithmetic runs at a small
// fraction of FP32's rate on this GPU, so the sums are FP32 trees (each
// thread about ten samples, then warp shuffles and one warp over the warp
// partials); only thread 0 forms the FP64 outputs.
// ---------------------------------------------------------------------------
__device__ float block_sum_f(float v, float* wbuf) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  if ((threadIdx.x & 31) == 0) wbuf[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    float w = threadIdx.x < (blockDim.x >> 5) ? wbuf[threadIdx.x] : 0.f;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) w += __shfl_down_sync(0xffffffffu, w, off);
    if (threadIdx.x == 0) wbuf[32] = w;
  }
  __syncthreads();
  const float r = wbuf[32];
  __syncthreads();
  return r;
}

// One block of 1024 threads.  moments = {mean0, mean1, sd0, sd1, corr,
// skew0, skew1, (kurt0 + kurt1)/2 - 3} (population moments); Z = (X - mean)
// / sd in FP32.
__device__ __forceinline__ void standardize2_body(const float* __restrict__ X, int64_t n,
                                                  float* __restrict__ Z, double* __restrict__ mom) {
  __shared__ float wbuf[33];
  const float inv_n = 1.0f / (float)n;
  float s0 = 0.f, s1 = 0.f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    s0 += X[2 * i];
    s1 += X[2 * i + 1];
  }
  const float m0 = block_sum_f(s0, wbuf) * inv_n, m1 = block_sum_f(s1, wbuf) * inv_n;
  float q00 = 0.f, q11 = 0.f, q01 = 0.f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const float a = X[2 * i] - m0, b = X[2 * i + 1] - m1;
    q00 = fmaf(a, a, q00);
    q11 = fmaf(b, b, q11);
    q01 = fmaf(a, b, q01);
  }
  const float v0 = block_sum_f(q00, wbuf) * inv_n, v1 = block_sum_f(q11, wbuf) * inv_n;
  const float c01 = block_sum_f(q01, wbuf) * inv_n;
  const float sd0 = sqrtf(v0), sd1 = sqrtf(v1);
  const float r0 = 1.0f / sd0, r1 = 1.0f / sd1;
  float t3a = 0.f, t3b = 0.f, t4a = 0.f, t4b = 0.f;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
    const float a = (X[2 * i] - m0) * r0, b = (X[2 * i + 1] - m1) * r1;
    Z[2 * i] = a;
    Z[2 * i + 1] = b;
    const float a2 = a * a, b2 = b * b;
    t3a = fmaf(a2, a, t3a);
    t3b = fmaf(b2, b, t3b);
    t4a = fmaf(a2, a2, t4a);
    t4b = fmaf(b2, b2, t4b);
  }
  const float sk0 = block_sum_f(t3a, wbuf) * inv_n, sk1 = block_sum_f(t3b, wbuf) * inv_n;
  const float k0 = block_sum_f(t4a, wbuf), k1 = block_sum_f(t4b, wbuf);
  if (threadIdx.x == 0) {
    mom[0] = m0;
    mom[1] = m1;
    mom[2] = sd0;
    mom[3] = sd1;
    mom[4] = (double)c01 / ((double)sd0 * sd1);
    mom[5] = sk0;
    mom[6] = sk1;
    mom[7] = 0.5 * ((double)k0 + k1) / (double)n - 3.0;
  }
}

__global__ void __launch_bounds__(1024) kde_standardize2_kernel(const float* __restrict__ X,
                                                                int64_t n, float* __restrict__ Z,
                                                                double* __restrict__ mom) {
  standardize2_body(X, n, Z, mom);
}

// One block per dataset of a batch: rows [off[b], off[b + 1]) of X and Z,
// moments at 8 b.
__global__ void __launch_bounds__(1024) kde_standardize2_sets_kernel(
    const float* __restrict__ X, const int64_t* __restrict__ off, float* __restrict__ Z,
    double* __restrict__ mom) {
  const int64_t a = off[blockIdx.x], b = off[blockIdx.x + 1];
  standardize2_body(X + 2 * a, b - a, Z + 2 * a, mom + 8 * (int64_t)blockIdx.x);
}

// 32 blocks of 256 threads, block `by` for the 32 block-features of one
// block row of the M x M grid (w = M/32 cells a side): thread (y0, bx) sums
// rows y0, y0 + 8, ... of block (by, bx); the rows are then added in shared
// memory.  feat[32 by + bx] = 8 sqrt(mass / n) with mass the block's counts
// times 2^-32; block 0 also writes feat[1024..] = corr, skew0, skew1, excess
// kurtosis, log10(n)/4, 1, then zeros.
__device__ __forceinline__ void features2_body(int by, const long long* __restrict__ counts,
                                               int M, int64_t n, const double* __restrict__ mom,
                                               float* __restrict__ feat) {
  __shared__ unsigned long long part[8][32];
  const int t = threadIdx.x, bx = t & 31, y0 = t >> 5, w = M / 32;
  unsigned long long s = 0;
  const bool vec = (w & 1) == 0 && ((uintptr_t)counts & 15) == 0;   // 16-byte loads
  for (int y = y0; y < w; y += 8) {
    const long long* row = counts + (size_t)(by * w + y) * M + bx * w;
    if (vec) {
#pragma unroll 4
      for (int x = 0; x < w / 2; ++x) {
        const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2*>(row) + x);
        s += v.x + v.y;
      }
    } else {
      for (int x = 0; x < w; ++x) s += (unsigned long long)row[x];
    }
  }
  part[y0][bx] = s;
  __syncthreads();
  if (t < 32) {
    unsigned long long tot = 0;
    for (int k = 0; k < 8; ++k) tot += part[k][t];
    // tot 2^-32 from its two 32-bit halves (no 64-bit integer conversion)
    const float mass =
        fmaf((float)(unsigned)(tot >> 32), 1.0f, (float)(unsigned)tot * 2.3283064365386963e-10f) /
        (float)n;
    feat[by * 32 + t] = 8.0f * sqrtf(mass);
  }
  if (by == 0 && t < 64) {
    float v = 0.f;
    if (t == 0) v = (float)mom[4];
    if (t == 1) v = (float)mom[5];
    if (t == 2) v = (float)mom[6];
    if (t == 3) v = (float)mom[7];
    if (t == 4) v = (float)(log10((double)n) / 4.0);
    if (t == 5) v = 1.f;
    feat[1024 + t] = v;
  }
}

__global__ void __launch_bounds__(256) kde_features2_kernel(const long long* __restrict__ counts,
                                                            int M, int64_t n,
                                                            const double* __restrict__ mom,
                                                            float* __restrict__ feat) {
  features2_body(blockIdx.x, counts, M, n, mom, feat);
}

// Grid (32, nsets): block row blockIdx.x of dataset blockIdx.y, whose
// counts start at y M^2, moments at 8 y and features at y KDE_FEAT_DIM.
__global__ void __launch_bounds__(256) kde_features2_sets_kernel(
    const long long* __restrict__ counts, int M, const int64_t* __restrict__ off,
    const double* __restrict__ mom, float* __restrict__ feat) {
  const int64_t y = blockIdx.y;
  features2_body(blockIdx.x, counts + y * M * M, M, off[y + 1] - off[y], mom + 8 * y,
                 feat + y * KDE_FEAT_DIM);
}

}  // namespace
}  // namespace kde

namespace kde {

kde_status standardize2_sets(const float* X, const int64_t* off_dev, int nsets, float* Z,
                             double* moments, cudaStream_t st) {
  LaunchScope ls("kde_standardize2_sets_kernel", st);
  kde_standardize2_sets_kernel<<<nsets, 1024, 0, st>>>(X, off_dev, Z, moments);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_standardize2_sets_kernel");
}

kde_status features2_sets(const int64_t* counts, int M, int nsets, const int64_t* off_dev,
                          const double* moments, float* feat, cudaStream_t st) {
  LaunchScope ls("kde_features2_sets_kernel", st);
  kde_features2_sets_kernel<<<dim3(32, (unsigned)nsets), 256, 0, st>>>(
      (const long long*)counts, M, off_dev, moments, feat);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_features2_sets_kernel");
}

}  // namespace kde

using namespace kde;

struct kde_mlp_s {
  int in, hid, out, outp, maxB;
  int64_t nparam, oW1, ob1, oW2, ob2, oW3, ob3;
  float *P, *G, *Mo, *Vo;
  bf16 *W1b, *W2b, *W2t, *W3b, *W3t;
  bf16 *Xb, *Xt, *A1b, *A1t, *A2b, *A2t, *dYb, *dYt, *dZ2b, *dZ2t, *dZ1t;
  float *Z1, *Z2, *Y, *dZ1, *dZ2, *dW3t, *b3p, *loss;
  int* status;
  int64_t step;
  std::vector<void*> allocs;
};

namespace {

template <typename T>
cudaError_t mlp_alloc(kde_mlp_s* m, T** p, size_t count) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, std::max<size_t>(16, count * sizeof(T)));
  if (e != cudaSuccess) return e;
  e = cudaMemset(q, 0, std::max<size_t>(16, count * sizeof(T)));
  m->allocs.push_back(q);
  *p = (T*)q;
  return e;
}

kde_status mlp_refresh(kde_mlp_s* m, cudaStream_t st) {
  LaunchScope ls("kde_mlp_refresh_kernel", st);
  kde_mlp_refresh_kernel<<<1024, 256, 0, st>>>(m->P + m->oW1, m->P + m->oW2, m->P + m->oW3,
                                                m->P + m->ob3, m->in, m->hid, m->out, m->outp,
                                                m->W1b, m->W2b, m->W2t, m->W3b, m->W3t, m->b3p);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_refresh_kernel");
}

GemmArgs gemm_args(const bf16* A, int lda, const bf16* B, int ldb, int M, int N, int K, float* C,
                   int ldc, int* status) {
  GemmArgs g{};
  g.A = A;
  g.lda = lda;
  g.B = B;
  g.ldb = ldb;
  g.M = M;
  g.N = N;
  g.K = K;
  g.C = C;
  g.ldc = ldc;
  g.status = status;
  return g;
}

// Forward pass on the first B rows of X (B <= maxB), padded to Bp rows.
kde_status mlp_forward(kde_mlp_s* m, const float* X, int B, int Bp, bool keep_t, cudaStream_t st) {
  {
    LaunchScope ls("kde_mlp_cast_kernel", st);
    const dim3 grid((unsigned)(m->in / 64) * (unsigned)(Bp / 32));
    const cudaError_t e = launch_pdl(kde_mlp_cast_kernel, grid, dim3(256), 0, st, X, B, Bp, m->in,
                                     m->Xb, keep_t ? m->Xt : (bf16*)nullptr);
    if (e != cudaSuccess) return cuda_fail(e, "kde_mlp_cast_kernel");
  }
  GemmArgs g1 = gemm_args(m->Xb, m->in, m->W1b, m->in, Bp, m->hid, m->in, m->Z1, m->hid, m->status);
  g1.bias = m->P + m->ob1;
  g1.Cb = m->A1b;
  g1.ldcb = m->hid;
  g1.Ct = keep_t ? m->A1t : nullptr;
  g1.ldct = Bp;
  kde_status s = launch_gemm(g1, EPI_BIAS_RELU, st);
  if (s != KDE_OK) return s;
  GemmArgs g2 = gemm_args(m->A1b, m->hid, m->W2b, m->hid, Bp, m->hid, m->hid, m->Z2, m->hid, m->status);
  g2.bias = m->P + m->ob2;
  g2.Cb = m->A2b;
  g2.ldcb = m->hid;
  g2.Ct = keep_t ? m->A2t : nullptr;
  g2.ldct = Bp;
  if ((s = launch_gemm(g2, EPI_BIAS_RELU, st)) != KDE_OK) return s;
  GemmArgs g3 = gemm_args(m->A2b, m->hid, m->W3b, m->hid, Bp, m->outp, m->hid, m->Y, m->outp, m->status);
  g3.bias = m->b3p;
  return launch_gemm(g3, EPI_BIAS, st);
}

// Loss and gradients into G (layout of m->P) for the first B rows.  Ten
// launches with the forward pass's four, each a programmatic dependent of the
// one before; 256 rows of 1088-256-256-3 took 243 us with 13 (products 17 us
// each with two stages, the loss 44, the column sums 10 each), now 87.
kde_status mlp_backward(kde_mlp_s* m, const float* T, int B, int Bp, float* G, float* loss_out,
                        cudaStream_t st) {
  cudaError_t e;
  {
    LaunchScope ls("kde_mlp_loss_kernel", st);
    e = launch_pdl(kde_mlp_loss_kernel, dim3(1), dim3(256), 0, st, m->Y, m->outp, T, B, Bp, m->out,
                   m->outp, m->dYb, m->dYt, G + m->ob3, loss_out ? loss_out : m->loss);
    if (e != cudaSuccess) return cuda_fail(e, "kde_mlp_loss_kernel");
  }
  // dZ2 = (dY W3) * (Z2 > 0)  (M = Bp, N = hid, K = 64)
  GemmArgs g5 = gemm_args(m->dYb, 64, m->W3t, 64, Bp, m->hid, 64, m->dZ2, m->hid, m->status);
  g5.Z = m->Z2;
  g5.ldz = m->hid;
  g5.Cb = m->dZ2b;
  g5.ldcb = m->hid;
  g5.Ct = m->dZ2t;
  g5.ldct = Bp;
  kde_status s = launch_gemm(g5, EPI_RELU_GRAD, st);
  if (s != KDE_OK) return s;
  // dZ1 = (dZ2 W2) * (Z1 > 0)  (M = Bp, N = hid, K = hid), and beside it
  // dW2 = dZ2^T A1  (M = hid, N = hid, K = Bp)
  GemmArgs g7 = gemm_args(m->dZ2b, m->hid, m->W2t, m->hid, Bp, m->hid, m->hid, m->dZ1, m->hid,
                          m->status);
  g7.Z = m->Z1;
  g7.ldz = m->hid;
  g7.Ct = m->dZ1t;
  g7.ldct = Bp;
  if ((s = launch_gemm2(g7, EPI_RELU_GRAD,
                        gemm_args(m->dZ2t, Bp, m->A1t, Bp, m->hid, m->hid, Bp, G + m->oW2, m->hid,
                                  m->status),
                        EPI_STORE, st)) != KDE_OK)
    return s;
  // dW3^T = A2^T dY  (M = hid, N = outp, K = Bp)
  if ((s = launch_gemm(gemm_args(m->A2t, Bp, m->dYt, Bp, m->hid, m->outp, Bp, m->dW3t, m->outp,
                                 m->status),
                       EPI_STORE, st)) != KDE_OK)
    return s;
  // dW1 = dZ1^T X  (M = hid, N = in, K = Bp)
  if ((s = launch_gemm(gemm_args(m->dZ1t, Bp, m->Xt, Bp, m->hid, m->in, Bp, G + m->oW1, m->in,
                                 m->status),
                       EPI_STORE, st)) != KDE_OK)
    return s;
  LaunchScope ls("kde_mlp_tail_kernel", st);
  e = launch_pdl(kde_mlp_tail_kernel, dim3((unsigned)(m->hid / 32 * (2 + m->out))), dim3(32), 0, st,
                 m->dZ1, m->dZ2, m->hid, B, m->dW3t, m->outp, m->out, G + m->ob1, G + m->ob2,
                 G + m->oW3);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_tail_kernel");
}

kde_status mlp_check_batch(const kde_mlp_s* m, int B, int* Bp) {
  if (!m || B <= 0 || B > m->maxB) return fail(KDE_ERR_INVALID_ARG, "batch size out of range");
  *Bp = (B + 127) / 128 * 128;
  return KDE_OK;
}

}  // namespace

extern "C" {

kde_status kde_gemm_bf16(int M, int N, int K, const void* A, int lda, const void* B, int ldb,
                         float* C, int ldc, int* status, kde_stream_t stream) {
  if (!A || !B || !C || !status) return fail(KDE_ERR_INVALID_ARG, "NULL pointer");
  return launch_gemm(gemm_args((const bf16*)A, lda, (const bf16*)B, ldb, M, N, K, C, ldc, status),
                     EPI_STORE, (cudaStream_t)stream);
}

kde_status kde_mlp_create(int in_dim, int hidden, int out_dim, int max_batch, uint64_t seed,
                          kde_mlp* out) {
  if (!out) return fail(KDE_ERR_INVALID_ARG, "NULL output");
  *out = nullptr;
  if (in_dim <= 0 || in_dim % 64 || hidden <= 0 || hidden % 128 || out_dim <= 0 || out_dim > 16 ||
      max_batch <= 0)
    return fail(KDE_ERR_INVALID_ARG,
                "MLP sizes: in_dim % 64 == 0, hidden % 128 == 0, 1 <= out_dim <= 16");
  kde_mlp_s* m = new kde_mlp_s();
  m->in = in_dim;
  m->hid = hidden;
  m->out = out_dim;
  m->outp = 16;
  m->maxB = max_batch;
  const int Bp = (max_batch + 127) / 128 * 128;
  m->oW1 = 0;
  m->ob1 = m->oW1 + (int64_t)hidden * in_dim;
  m->oW2 = m->ob1 + hidden;
  m->ob2 = m->oW2 + (int64_t)hidden * hidden;
  m->oW3 = m->ob2 + hidden;
  m->ob3 = m->oW3 + (int64_t)out_dim * hidden;
  m->nparam = m->ob3 + out_dim;
  cudaError_t e = cudaSuccess;
  auto A = [&](auto** p, size_t count) {
    if (e == cudaSuccess) e = mlp_alloc(m, p, count);
  };
  A(&m->P, m->nparam);
  A(&m->G, m->nparam);
  A(&m->Mo, m->nparam);
  A(&m->Vo, m->nparam);
  A(&m->W1b, (size_t)hidden * in_dim);
  A(&m->W2b, (size_t)hidden * hidden);
  A(&m->W2t, (size_t)hidden * hidden);
  A(&m->W3b, (size_t)m->outp * hidden);
  A(&m->W3t, (size_t)hidden * 64);
  A(&m->Xb, (size_t)Bp * in_dim);
  A(&m->Xt, (size_t)Bp * in_dim);
  A(&m->A1b, (size_t)Bp * hidden);
  A(&m->A1t, (size_t)Bp * hidden);
  A(&m->A2b, (size_t)Bp * hidden);
  A(&m->A2t, (size_t)Bp * hidden);
  A(&m->dYb, (size_t)Bp * 64);
  A(&m->dYt, (size_t)m->outp * Bp);
  A(&m->dZ2b, (size_t)Bp * hidden);
  A(&m->dZ2t, (size_t)Bp * hidden);
  A(&m->dZ1t, (size_t)Bp * hidden);
  A(&m->Z1, (size_t)Bp * hidden);
  A(&m->Z2, (size_t)Bp * hidden);
  A(&m->Y, (size_t)Bp * m->outp);
  A(&m->dZ1, (size_t)Bp * hidden);
  A(&m->dZ2, (size_t)Bp * hidden);
  A(&m->dW3t, (size_t)hidden * m->outp);
  A(&m->b3p, (size_t)m->outp);
  A(&m->loss, 4);
  A(&m->status, 4);
  if (e != cudaSuccess) {
    kde_mlp_destroy(m);
    return cuda_fail(e, "cudaMalloc(MLP)");
  }
  // He-normal weights, zero biases, from a seeded host generator.
  std::vector<float> h(m->nparam, 0.f);
  std::mt19937_64 rng(seed);
  auto fill = [&](int64_t off, int rows, int cols) {
    std::normal_distribution<double> nd(0.0, std::sqrt(2.0 / cols));
    for (int64_t i = 0; i < (int64_t)rows * cols; ++i) h[off + i] = (float)nd(rng);
  };
  fill(m->oW1, hidden, in_dim);
  fill(m->oW2, hidden, hidden);
  fill(m->oW3, out_dim, hidden);
  kde_status s = kde_mlp_set_params(m, h.data(), m->nparam);
  if (s != KDE_OK) {
    kde_mlp_destroy(m);
    return s;
  }
  *out = m;
  return KDE_OK;
}

kde_status kde_mlp_destroy(kde_mlp m) {
  if (!m) return KDE_OK;
  for (void* p : m->allocs) cudaFree(p);
  delete m;
  return KDE_OK;
}

kde_status kde_mlp_param_count(kde_mlp m, int64_t* count) {
  if (!m || !count) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  *count = m->nparam;
  return KDE_OK;
}

kde_status kde_mlp_get_params(kde_mlp m, float* host, int64_t count) {
  if (!m || !host || count != m->nparam) return fail(KDE_ERR_INVALID_ARG, "bad parameter buffer");
  cudaError_t e = cudaMemcpy(host, m->P, sizeof(float) * count, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaMemcpy(params)");
}

kde_status kde_mlp_set_params(kde_mlp m, const float* host, int64_t count) {
  if (!m || !host || count != m->nparam) return fail(KDE_ERR_INVALID_ARG, "bad parameter buffer");
  cudaError_t e = cudaMemcpy(m->P, host, sizeof(float) * count, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(params)");
  kde_status s = mlp_refresh(m, 0);
  if (s != KDE_OK) return s;
  e = cudaDeviceSynchronize();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_set_params");
}

kde_status kde_mlp_get_state(kde_mlp m, float* adam_m, float* adam_v, int64_t* step) {
  if (!m || !adam_m || !adam_v || !step) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  cudaError_t e = cudaMemcpy(adam_m, m->Mo, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(adam_v, m->Vo, sizeof(float) * m->nparam, cudaMemcpyDeviceToHost);
  *step = m->step;
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaMemcpy(optimizer state)");
}

kde_status kde_mlp_set_state(kde_mlp m, const float* adam_m, const float* adam_v, int64_t step) {
  if (!m || !adam_m || !adam_v || step < 0) return fail(KDE_ERR_INVALID_ARG, "bad optimizer state");
  cudaError_t e = cudaMemcpy(m->Mo, adam_m, sizeof(float) * m->nparam, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(m->Vo, adam_v, sizeof(float) * m->nparam, cudaMemcpyHostToDevice);
  m->step = step;
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaMemcpy(optimizer state)");
}

kde_status kde_mlp_forward(kde_mlp m, const float* X, int B, float* Y, kde_stream_t stream) {
  int Bp;
  kde_status s = mlp_check_batch(m, B, &Bp);
  if (s != KDE_OK) return s;
  if (!X || !Y) return fail(KDE_ERR_INVALID_ARG, "NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  if ((s = mlp_forward(m, X, B, Bp, false, st)) != KDE_OK) return s;
  LaunchScope ls("kde_mlp_take_kernel", st);
  kde_mlp_take_kernel<<<(B * m->out + 255) / 256, 256, 0, st>>>(m->Y, m->outp, B, m->out, Y);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_take_kernel");
}

kde_status kde_mlp_loss_grad(kde_mlp m, const float* X, const float* T, int B, float* loss,
                             float* grads, kde_stream_t stream) {
  int Bp;
  kde_status s = mlp_check_batch(m, B, &Bp);
  if (s != KDE_OK) return s;
  if (!X || !T) return fail(KDE_ERR_INVALID_ARG, "NULL pointer");
  cudaStream_t st = (cudaStream_t)stream;
  if ((s = mlp_forward(m, X, B, Bp, true, st)) != KDE_OK) return s;
  return mlp_backward(m, T, B, Bp, grads ? grads : m->G, loss, st);
}

kde_status kde_mlp_train_step(kde_mlp m, const float* X, const float* T, int B, float lr,
                              float* loss, kde_stream_t stream) {
  kde_status s = kde_mlp_loss_grad(m, X, T, B, loss, nullptr, stream);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  m->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - (float)std::pow((double)b1, (double)m->step);
  const float c2 = 1.f - (float)std::pow((double)b2, (double)m->step);
  {
    LaunchScope ls("kde_mlp_adam_kernel", st);
    kde_mlp_adam_kernel<<<512, 256, 0, st>>>(m->P, m->G, m->Mo, m->Vo, m->nparam, lr, b1, b2,
                                             1e-8f, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "kde_mlp_adam_kernel");
  }
  return mlp_refresh(m, st);
}

kde_status kde_mlp_status(kde_mlp m, int* flag) {
  if (!m || !flag) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(flag, m->status, sizeof(int), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_status");
}

kde_status kde_mlp_status_copy(kde_mlp m, int* dst, kde_stream_t stream) {
  if (!m || !dst) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  cudaError_t e = cudaMemcpyAsync(dst, m->status, sizeof(int), cudaMemcpyDefault,
                                  (cudaStream_t)stream);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_mlp_status_copy");
}

kde_status kde_standardize2(const float* X, int64_t n, float* Z, double* moments,
                            kde_stream_t stream) {
  if (!X || !Z || !moments || n < 2) return fail(KDE_ERR_INVALID_ARG, "bad standardisation input");
  cudaStream_t st = (cudaStream_t)stream;
  LaunchScope ls("kde_standardize2_kernel", st);
  kde_standardize2_kernel<<<1, 1024, 0, st>>>(X, n, Z, moments);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_standardize2_kernel");
}

kde_status kde_features2(const int64_t* counts, int M, int64_t n, const double* moments,
                         float* feat, kde_stream_t stream) {
  if (!counts || !moments || !feat || M < 32 || M % 32 || n < 1)
    return fail(KDE_ERR_INVALID_ARG, "features: M must be a multiple of 32");
  cudaStream_t st = (cudaStream_t)stream;
  LaunchScope ls("kde_features2_kernel", st);
  kde_features2_kernel<<<32, 256, 0, st>>>((const long long*)counts, M, n, moments, feat);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_features2_kernel");
}

}  // extern "C"
