// The convolution step (Eq. 10) in wrapped, zero-padded form:
//   kde_kernel_grid: k_l on |l_k| <= L_k at index l mod P_k (Eq. 6, Eq. 12
//                    without the shift), transformed to its real spectrum K;
//   kde_fft_eval:    C = F(c) of the zero-padded counts, S = C K,
//                    s = F^{-1}(S), cropped to [0, M_k) (Eq. 14 shifted).
// Passes (row-major, last axis contiguous, Q = P_last/2 + 1); every line is
// transformed by a group of tpl threads (line_fft), tpl chosen per launch:
//   rows_r2c  real rows -> half spectra; two real rows ride in one complex
//             FFT (x + i y) and are separated afterwards;
//   cols      FFT along a strided axis: a block stages W adjacent columns in
//             shared memory with coalesced loads, each thread group
//             transforms one, and the block stores them back coalesced.  Modes: forward,
//             forward-to-real (the kernel spectrum, written with the
//             transformed axis contiguous), forward * K * inverse with crop
//             (the leading axis), inverse with crop;
//   rows_c2r  half spectra -> real rows, cropped (two rows per complex FFT);
//   line1d    d = 1: forward, * K, inverse and crop.
// Only lines that hold data are transformed and only lines that survive the
// crop are inverse-transformed.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>
#include <type_traits>
#include <vector>

#include "fft_engine.cuh"
#include "fixed_pos.h"
#include "fx_pairs.h"
#include "kde_internal.h"
#include "kde_debug.cuh"
#include "kgen.cuh"
#include "pdl.cuh"
#include "smem_limit.cuh"

namespace kde {
namespace {


// Global loads issued back to back by one thread before their values are
// stored to shared memory (memory-level parallelism of the load phases).
// Loads of arrays that other blocks produce (counts, spectra) take the
// L2-only path (__ldcg): the persistent batch kernel reads, within one
// launch, data that other blocks wrote after a completion counter said so.
constexpr int kLoadBatch = 8;

// Twiddle table -> shared memory by asynchronous copies (cp.async): they
// hold no registers and are in flight together with a pass's own data
// loads; twiddles_wait() completes this thread's copies, and the block
// barrier after it publishes the table.  Every thread of the block calls
// both.  Tables start on 256-byte boundaries; one whose size is an odd
// multiple of 8 bytes ends with an 8-byte copy.
template <typename V>
__device__ __forceinline__ void twiddles_async(V* tw_s, const V* tw, int P) {
  const int bytes = P * (int)sizeof(V);
  const int n16 = bytes >> 4;
  const size_t src = __cvta_generic_to_global(tw);
  const unsigned dst = (unsigned)__cvta_generic_to_shared(tw_s);
  for (int i = threadIdx.x; i < n16; i += blockDim.x)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + 16u * i),
                 "l"(src + 16ull * i)
                 : "memory");
  if ((bytes & 15) && threadIdx.x == 0)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst + 16u * n16),
                 "l"(src + 16ull * n16)
                 : "memory");
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void twiddles_wait() {
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

template <typename T>
struct RowsParams {
  using V = typename Cplx<T>::type;
  int64_t nrows;      // real rows
  int Min;            // data length of a row (zero-padded to P)
  int64_t in_stride;  // elements between input rows
  int Q;
  V* out;             // complex half spectra, row stride Q
  T* out_real;        // real part only (d = 1 kernel spectrum)
  int tpl;           // threads per line
  LinePlan lp;
  const V* tw;
};

// Split Z = F(x + i y) into X = F(x), Y = F(y) for k in [0, Q) and store.
template <typename T>
__device__ __forceinline__ void store_r2c(const RowsParams<T>& p, const typename Cplx<T>::type* z,
                                          int64_t r0, const LineGroup& g) {
  using V = typename Cplx<T>::type;
  const int P = p.lp.N;
  for (int k = g.lt; k < p.Q; k += g.tpl) {
    V zk = z[k];
    V zm = z[k == 0 ? 0 : P - k];
    V X = mk<V>(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
    V Y = mk<V>(T(0.5) * (zk.y + zm.y), T(-0.5) * (zk.x - zm.x));
    if (!KDE_DCHECK(r0 < p.nrows, KDE_DBG_STOCKHAM)) continue;
    if (p.out_real) {
      p.out_real[r0 * p.Q + k] = X.x;
    } else {
      p.out[r0 * p.Q + k] = X;
      if (r0 + 1 < p.nrows) p.out[(r0 + 1) * p.Q + k] = Y;
    }
  }
}

// The line group of this thread (line li of the block).
__device__ __forceinline__ LineGroup line_group(int tpl, int& li) {
  li = threadIdx.x / tpl;
  return LineGroup{(int)threadIdx.x - li * tpl, tpl, 1 + li};
}

// Counts rows -> half spectra, one row pair per line group.  Counts are int64
// in units of 2^-32; the unit is folded into the kernel spectrum.
template <typename T>
__device__ __forceinline__ void rows_counts_body(const long long* __restrict__ counts,
                                                 const RowsParams<T>& p, int64_t vb) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = p.lp.N;
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  int li;
  const LineGroup g = line_group(p.tpl, li);
  V* a = tw_s + P + 2 * li * P;
  V* b = a + P;
  twiddles_async(tw_s, p.tw, P);
  const int64_t r0 = 2 * (vb * (blockDim.x / p.tpl) + li);
  const bool act = r0 < p.nrows;
  const long long* c0 = counts + r0 * p.in_stride;
  const long long* c1 = c0 + p.in_stride;
  const bool two = r0 + 1 < p.nrows;
  for (int x0 = g.lt; act && x0 < P; x0 += kLoadBatch * g.tpl) {
    long long u0[kLoadBatch], u1[kLoadBatch];
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int x = x0 + u * g.tpl;
      u0[u] = x < p.Min ? __ldcg(c0 + x) : 0;
      u1[u] = (x < p.Min && two) ? __ldcg(c1 + x) : 0;
    }
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int x = x0 + u * g.tpl;
      if (x < P) a[x] = mk<V>(count_value<T>(u0[u]), count_value<T>(u1[u]));
    }
  }
  twiddles_wait();
  __syncthreads();
  if (!act) return;
  V* z = line_fft<V, false>(a, b, p.lp, tw_s, g);
  store_r2c<T>(p, z, r0, g);
}

template <typename T>
__global__ void __launch_bounds__(256)
kde_rows_r2c_counts_kernel(const long long* __restrict__ counts, RowsParams<T> p) {
  rows_counts_body<T>(counts, p, blockIdx.x);
}

// Kernel-grid rows -> half spectra (or real spectrum for d = 1).  Row r
// enumerates the leading lags (l_0, ..., l_{d-2}) with |l_k| <= L_k; the last
// axis holds lag l at position l mod P.
template <typename T>
__device__ __forceinline__ void rows_kgen_body(const KGen<T>& gen, const RowsParams<T>& p,
                                               int64_t vb) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = p.lp.N;
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  int li;
  const LineGroup g = line_group(p.tpl, li);
  V* a = tw_s + P + 2 * li * P;
  V* b = a + P;
  twiddles_async(tw_s, p.tw, P);
  const int64_t r0 = 2 * (vb * (blockDim.x / p.tpl) + li);
  const bool act = r0 < p.nrows;
  const int Llast = gen.d == 1 ? gen.L[0] : (gen.d == 2 ? gen.L[1] : gen.L[2]);
  for (int x = g.lt; act && x < P; x += g.tpl) {
    T val[2] = {0, 0};
    const int ll = wrapped_lag(x, P, Llast);
    if (ll <= Llast) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t r = r0 + h;
        if (r >= p.nrows) break;
        // lags of this row and position, indexed statically (a runtime
        // index would put the array in local memory)
        int l[KDE_MAX_D] = {ll, 0, 0};
        if (gen.d == 2) {
          l[0] = (int)r - gen.L[0];
          l[1] = ll;
        } else if (gen.d == 3) {
          const int w1 = 2 * gen.L[1] + 1;
          l[0] = (int)(r / w1) - gen.L[0];
          l[1] = (int)(r % w1) - gen.L[1];
          l[2] = ll;
        }
        val[h] = kernel_value<T>(gen, l);
      }
    }
    a[x] = mk<V>(val[0], val[1]);
  }
  twiddles_wait();
  __syncthreads();
  if (!act) return;
  V* z = line_fft<V, false>(a, b, p.lp, tw_s, g);
  store_r2c<T>(p, z, r0, g);
}

template <typename T>
__global__ void __launch_bounds__(256)
kde_rows_r2c_kgen_kernel(KGen<T> gen, RowsParams<T> p) {
  rows_kgen_body<T>(gen, p, blockIdx.x);
}

template <typename T>
struct C2RParams {
  using V = typename Cplx<T>::type;
  const V* in;        // half spectra, row stride Q
  T* out;             // real rows, row stride Mout
  int64_t nrows;
  int Mout;
  int Q;
  int tpl;
  LinePlan lp;
  const V* tw;
};

// Half spectra -> real rows cropped to [0, Mout).  Z = X + i Y is rebuilt on
// the full length from Hermitian symmetry: Z_k = conj(X_{P-k}) + i conj(Y_{P-k})
// for k >= Q; then x + i y = F^{-1}(Z).
template <typename T>
__device__ __forceinline__ void rows_c2r_body(const C2RParams<T>& p, int64_t vb) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = p.lp.N;
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  int li;
  const LineGroup g = line_group(p.tpl, li);
  V* a = tw_s + P + 2 * li * P;
  V* b = a + P;
  twiddles_async(tw_s, p.tw, P);
  const int64_t r0 = 2 * (vb * (blockDim.x / p.tpl) + li);
  const bool act = r0 < p.nrows;
  const bool two = r0 + 1 < p.nrows;
  const V* x0 = p.in + r0 * p.Q;
  const V* x1 = x0 + p.Q;
  for (int k0 = g.lt; act && k0 < p.Q; k0 += kLoadBatch * g.tpl) {
    V X[kLoadBatch], Y[kLoadBatch];
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int k = k0 + u * g.tpl;
      X[u] = k < p.Q ? __ldcg(x0 + k) : mk<V>(0, 0);
      Y[u] = (k < p.Q && two) ? __ldcg(x1 + k) : mk<V>(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int k = k0 + u * g.tpl;
      if (k >= p.Q) continue;
      a[k] = mk<V>(X[u].x - Y[u].y, X[u].y + Y[u].x);
      if (k > 0 && P - k >= p.Q) a[P - k] = mk<V>(X[u].x + Y[u].y, Y[u].x - X[u].y);
    }
  }
  twiddles_wait();
  __syncthreads();
  if (!act) return;
  V* z = line_fft<V, true>(a, b, p.lp, tw_s, g);
  T* o0 = p.out + r0 * p.Mout;
  T* o1 = o0 + p.Mout;
  for (int m = g.lt; m < p.Mout; m += g.tpl) {
    V v = z[m];
    o0[m] = v.x;
    if (two) o1[m] = v.y;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) kde_rows_c2r_kernel(C2RParams<T> p) {
  rows_c2r_body<T>(p, blockIdx.x);
}

// d = 1: counts -> F -> * K (real, even: K_k = K_{P-k}) -> F^{-1} -> crop.
template <typename T>
__global__ void __launch_bounds__(256)
kde_line1d_kernel(const long long* __restrict__ counts, const T* __restrict__ K, T* out, int M,
                  int Q, LinePlan lp, const typename Cplx<T>::type* tw) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = lp.N;
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  V* a = tw_s + P;
  V* b = a + P;
  const LineGroup g{(int)threadIdx.x, (int)blockDim.x, 1};
  twiddles_async(tw_s, tw, P);
  for (int x = g.lt; x < P; x += g.tpl) a[x] = mk<V>(x < M ? count_value<T>(counts[x]) : T(0), 0);
  twiddles_wait();
  __syncthreads();
  V* z = line_fft<V, false>(a, b, lp, tw_s, g);
  for (int k = g.lt; k < P; k += g.tpl) {
    T kv = K[k < Q ? k : P - k];
    z[k] = mk<V>(z[k].x * kv, z[k].y * kv);
  }
  g.sync();
  V* other = (z == a) ? b : a;
  V* y = line_fft<V, true>(z, other, lp, tw_s, g);
  for (int m = g.lt; m < M; m += g.tpl) out[m] = y[m].x;
}

enum ColMode { COL_FWD = 0, COL_FWD_REAL = 1, COL_MID = 2, COL_INV = 3, COL_FWD_POWER = 4,
               COL_FWD_DOT = 5, COL_AUTO = 6 };

template <typename T>
struct ColsParams {
  using V = typename Cplx<T>::type;
  const V* in;     // [O][Nin][S]
  V* out;          // [O][Nout][S]
  T* out_real;     // COL_FWD_REAL: [O][S][P] (transformed axis contiguous)
  const T* K;      // COL_MID: [S][P] real spectrum, transformed axis contiguous
  int64_t S;
  int Nin, Nout;
  int Lw;          // >= 0: input row n holds lag n - Lw (wrapped); < 0: row n at position n
  int tpl;         // threads per column
  LinePlan lp;
  const V* tw;
  // COL_FWD_POWER: out_real = w(k) |2^-32 z|^2 with k = s mod Qw the
  // last-axis frequency and w = 1 at k = 0 and k = Plw/2, else 2.
  // COL_FWD_DOT: partial[blockIdx.x] += sum over the block of W * Re z.
  int Qw, Plw;
  const T* W;
  double* partial;
  // COL_AUTO: z <- |s_pre z|^2 s_post between the forward and inverse
  // transforms (the counts' power spectrum, for their autocorrelation).
  T s_pre, s_post;
};

__device__ __forceinline__ int half_weight(int64_t s, int Q, int Plast) {
  const int k = (int)(s % Q);
  return (k == 0 || 2 * k == Plast) ? 1 : 2;
}

// Block-wide sum of one double per thread, written by thread 0.
__device__ __forceinline__ void block_sum_to(double v, double* out) {
  __shared__ double warp_part[32];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) warp_part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += warp_part[w];
    *out = t;
  }
}

// W adjacent columns (s0 .. s0+W-1) of outer slab o, one line group each.
template <typename T, int MODE>
__device__ __forceinline__ void cols_body_slab(const ColsParams<T>& p, int64_t slab,
                                               int64_t vbx) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = p.lp.N;
  // Passes whose columns are Hermitian (the kernel spectrum's last pass: k is
  // real and even, so every column transforms to a real line) transform two
  // columns per FFT: F(x1 + i x2) = F(x1) + i F(x2) with both real.
  constexpr bool PAIRED = MODE == COL_FWD_REAL || MODE == COL_FWD_DOT;
  const int W = (PAIRED ? 2 : 1) * (blockDim.x / p.tpl);
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  // Line t owns lines[t LS ..): its buffer, then its scratch.  LS = 2P + 1
  // puts the lines of one position in different banks.
  const int LS = 2 * P + 1;
  V* lines = tw_s + P;
  int li;
  const LineGroup g = line_group(p.tpl, li);
  twiddles_async(tw_s, p.tw, P);
  const int64_t o = slab;
  const int64_t s0 = vbx * W;
  const V* in = p.in + o * (int64_t)p.Nin * p.S;
  if constexpr (PAIRED) {
    // line t holds columns s0 + 2t (real part) and s0 + 2t + 1 (imaginary)
    const int npair = W / 2;
    for (int idx0 = threadIdx.x; idx0 < P * npair; idx0 += kLoadBatch * blockDim.x) {
      V v1[kLoadBatch], v2[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int idx = idx0 + u * blockDim.x;
        const int pos = idx / npair, t = idx - pos * npair;
        const int n = source_row(pos, P, p.Lw, p.Nin);
        const int64_t s = s0 + 2 * t;
        const bool ok = idx < P * npair && n < p.Nin;
        v1[u] = (ok && s < p.S) ? __ldcg(in + (int64_t)n * p.S + s) : mk<V>(0, 0);
        v2[u] = (ok && s + 1 < p.S) ? __ldcg(in + (int64_t)n * p.S + s + 1) : mk<V>(0, 0);
      }
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int idx = idx0 + u * blockDim.x;
        const int pos = idx / npair, t = idx - pos * npair;
        if (idx < P * npair) lines[t * LS + pos] = mk<V>(v1[u].x - v2[u].y, v1[u].y + v2[u].x);
      }
    }
    twiddles_wait();
    __syncthreads();
    const int64_t s1 = s0 + 2 * li;
    V* a = lines + li * LS;
    double acc = 0.0;
    if (s1 < p.S) {
      const V* z = line_fft<V, false>(a, a + P, p.lp, tw_s, g);
      const bool two = s1 + 1 < p.S;
      if (MODE == COL_FWD_REAL) {
        T* d1 = p.out_real + (o * p.S + s1) * P;
        for (int k = g.lt; k < P; k += g.tpl) {
          d1[k] = z[k].x;
          if (two) d1[P + k] = z[k].y;
        }
      } else {
        const T* W1 = p.W + s1 * P;
        T part = 0;
        for (int k0 = g.lt; k0 < P; k0 += kLoadBatch * g.tpl) {
          T w1[kLoadBatch], w2[kLoadBatch];
#pragma unroll
          for (int u = 0; u < kLoadBatch; ++u) {
            const int k = k0 + u * g.tpl;
            w1[u] = k < P ? __ldg(W1 + k) : T(0);
            w2[u] = (k < P && two) ? __ldg(W1 + P + k) : T(0);
          }
#pragma unroll
          for (int u = 0; u < kLoadBatch; ++u) {
            const int k = k0 + u * g.tpl;
            if (k < P) part += w1[u] * z[k].x + w2[u] * z[k].y;
          }
        }
        acc = (double)part;
      }
    }
    if (MODE == COL_FWD_DOT) block_sum_to(acc, p.partial + blockIdx.x);
    return;
  }
  for (int idx0 = threadIdx.x; idx0 < P * W; idx0 += kLoadBatch * blockDim.x) {
    V v[kLoadBatch];
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int idx = idx0 + u * blockDim.x;
      const int pos = idx / W, t = idx - pos * W;
      const int n = source_row(pos, P, p.Lw, p.Nin);
      const int64_t s = s0 + t;
      v[u] = (idx < P * W && n < p.Nin && s < p.S) ? __ldcg(in + (int64_t)n * p.S + s) : mk<V>(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int idx = idx0 + u * blockDim.x;
      const int pos = idx / W, t = idx - pos * W;
      if (idx < P * W) lines[t * LS + pos] = v[u];
    }
  }
  twiddles_wait();
  __syncthreads();
  const int64_t s = s0 + li;
  V* a = lines + li * LS;
  V* b = a + P;
  V* z = a;
  if (s < p.S) {
    // COL_MID: the first kLoadBatch values of the column's K per thread are
    // loaded before the forward transform, which hides their latency.
    T kpre[kLoadBatch];
    const T* Kc = p.K + s * P;
    if (MODE == COL_MID) {
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int k = g.lt + u * g.tpl;
        kpre[u] = k < P ? __ldcg(Kc + k) : T(0);
      }
    }
    if (MODE == COL_INV)
      z = line_fft<V, true>(a, b, p.lp, tw_s, g);
    else
      z = line_fft<V, false>(a, b, p.lp, tw_s, g);
    if (MODE == COL_MID) {
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int k = g.lt + u * g.tpl;
        if (k < P) z[k] = mk<V>(z[k].x * kpre[u], z[k].y * kpre[u]);
      }
      for (int k0 = g.lt + kLoadBatch * g.tpl; k0 < P; k0 += kLoadBatch * g.tpl) {
        T kv[kLoadBatch];
#pragma unroll
        for (int u = 0; u < kLoadBatch; ++u) {
          const int k = k0 + u * g.tpl;
          kv[u] = k < P ? __ldcg(Kc + k) : T(0);
        }
#pragma unroll
        for (int u = 0; u < kLoadBatch; ++u) {
          const int k = k0 + u * g.tpl;
          if (k < P) z[k] = mk<V>(z[k].x * kv[u], z[k].y * kv[u]);
        }
      }
      g.sync();
      V* other = (z == a) ? b : a;
      z = line_fft<V, true>(z, other, p.lp, tw_s, g);
    }
    if (MODE == COL_AUTO) {
      for (int k = g.lt; k < P; k += g.tpl) {
        const T re = z[k].x * p.s_pre, im = z[k].y * p.s_pre;
        z[k] = mk<V>((re * re + im * im) * p.s_post, T(0));
      }
      g.sync();
      V* other = (z == a) ? b : a;
      z = line_fft<V, true>(z, other, p.lp, tw_s, g);
    }
    if (MODE == COL_FWD_POWER) {
      T* dst = p.out_real + (o * p.S + s) * P;
      const T w = (T)half_weight(s, p.Qw, p.Plw);
      const T sc = (T)2.3283064365386963e-10;  // 2^-32
      for (int k = g.lt; k < P; k += g.tpl) {
        const T re = z[k].x * sc, im = z[k].y * sc;
        dst[k] = w * (re * re + im * im);
      }
    }
  }
  if (MODE == COL_FWD_POWER) return;
  // Every line's result sits in the same buffer of its pair, told by the
  // number of stages run (not by this thread's z: the group of a column
  // beyond S ran none, and its threads store other columns too).
  const int nfft = (MODE == COL_MID || MODE == COL_AUTO) ? 2 : 1;
  const int zoff = (nfft * p.lp.nst) & 1 ? P : 0;
  __syncthreads();
  const int nout = (MODE == COL_FWD) ? P : p.Nout;
  for (int idx = threadIdx.x; idx < nout * W; idx += blockDim.x) {
    const int pos = idx / W, t = idx - pos * W;
    const int64_t ss = s0 + t;
    if (ss >= p.S) continue;
    p.out[(o * nout + pos) * p.S + ss] = lines[t * LS + zoff + pos];
  }
}

template <typename T, int MODE>
__device__ __forceinline__ void cols_body(const ColsParams<T>& p) {
  cols_body_slab<T, MODE>(p, blockIdx.y, blockIdx.x);
}

// Column passes with many columns: a block holds kSimdW adjacent columns
// position-major in shared memory (element (pos, c) at pos kSimdW + c).
// Thread t works on column t mod kSimdW; the kSimdW threads of a group run
// the same butterfly on every column, so index arithmetic and twiddles are
// uniform and each group's shared and global accesses are one contiguous
// row segment of kSimdW elements.  The kernel spectrum of such a pass is
// stored [P][S] (columns contiguous).
constexpr int kSimdW = 16;
// Column kernels launch with up to this many threads (SIMD blocks: kSimdW
// lanes per butterfly group times 16 to 32 groups).
constexpr int kColsMaxThreads = 512;

template <typename V, int R, bool INV>
__device__ __forceinline__ void simd_stage(const V* __restrict__ in, V* __restrict__ out,
                                           const Stage& s, const V* __restrict__ tw, int c, int g,
                                           int ng) {
  for (int j = g; j < s.nb; j += ng) {
    V x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = in[(j + r * s.nb) * kSimdW + c];
    int base;
    if (s.Ns > 1) {
      const unsigned q = __umulhi((unsigned)j, s.magic);
      const int k = j - (int)q * s.Ns;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        V w = tw[r * k * s.twstep];
        if (INV) w = cconj(w);
        x[r] = cmul(x[r], w);
      }
      base = (int)q * s.Ns * R + k;
    } else {
      base = j * R;
    }
    SmallDFT<V, R, INV>::run(x);
#pragma unroll
    for (int r = 0; r < R; ++r) out[(base + r * s.Ns) * kSimdW + c] = x[r];
  }
}

template <typename V, bool INV>
__device__ V* simd_fft(V* a, V* b, const LinePlan& lp, const V* __restrict__ tw, int c, int g,
                       int ng) {
  for (int s = 0; s < lp.nst; ++s) {
    const Stage& st = lp.st[s];
    switch (st.R) {
      case 2: simd_stage<V, 2, INV>(a, b, st, tw, c, g, ng); break;
      case 3: simd_stage<V, 3, INV>(a, b, st, tw, c, g, ng); break;
      case 4: simd_stage<V, 4, INV>(a, b, st, tw, c, g, ng); break;
      case 5: simd_stage<V, 5, INV>(a, b, st, tw, c, g, ng); break;
      case 7: simd_stage<V, 7, INV>(a, b, st, tw, c, g, ng); break;
      default: simd_stage<V, 8, INV>(a, b, st, tw, c, g, ng); break;
    }
    __syncthreads();
    V* t = a;
    a = b;
    b = t;
  }
  return a;
}

template <typename T, int MODE>
__device__ __forceinline__ void cols_simd_body_slab(const ColsParams<T>& p, int64_t slab) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int P = p.lp.N;
  V* tw_s = reinterpret_cast<V*>(smem_raw);
  V* bufA = tw_s + P;
  V* bufB = bufA + P * kSimdW;
  const int c = threadIdx.x % kSimdW, g = threadIdx.x / kSimdW, ng = blockDim.x / kSimdW;
  twiddles_async(tw_s, p.tw, P);
  const int64_t o = slab;
  const V* in = p.in + o * (int64_t)p.Nin * p.S;
  // Hermitian columns (see cols_body_slab): a block takes 2 kSimdW columns,
  // column c and c + kSimdW share one FFT as real and imaginary parts.
  constexpr bool PAIRED = MODE == COL_FWD_REAL || MODE == COL_FWD_DOT;
  if constexpr (PAIRED) {
    const int64_t sA = (int64_t)blockIdx.x * 2 * kSimdW + c, sB = sA + kSimdW;
    for (int pos0 = g; pos0 < P; pos0 += kLoadBatch * ng) {
      V va[kLoadBatch], vb[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int pos = pos0 + u * ng;
        const int n = source_row(pos, P, p.Lw, p.Nin);
        const bool ok = pos < P && n < p.Nin;
        va[u] = (ok && sA < p.S) ? in[(int64_t)n * p.S + sA] : mk<V>(0, 0);
        vb[u] = (ok && sB < p.S) ? in[(int64_t)n * p.S + sB] : mk<V>(0, 0);
      }
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int pos = pos0 + u * ng;
        if (pos < P) bufA[pos * kSimdW + c] = mk<V>(va[u].x - vb[u].y, va[u].y + vb[u].x);
      }
    }
    twiddles_wait();
    __syncthreads();
    const V* z = simd_fft<V, false>(bufA, bufB, p.lp, tw_s, c, g, ng);
    if (MODE == COL_FWD_DOT) {
      T part = 0;
      for (int pos0 = g; pos0 < P; pos0 += kLoadBatch * ng) {
        T wa[kLoadBatch], wb[kLoadBatch];
#pragma unroll
        for (int u = 0; u < kLoadBatch; ++u) {
          const int pos = pos0 + u * ng;
          wa[u] = (pos < P && sA < p.S) ? __ldg(p.W + (int64_t)pos * p.S + sA) : T(0);
          wb[u] = (pos < P && sB < p.S) ? __ldg(p.W + (int64_t)pos * p.S + sB) : T(0);
        }
#pragma unroll
        for (int u = 0; u < kLoadBatch; ++u) {
          const int pos = pos0 + u * ng;
          if (pos < P) {
            const V v = z[pos * kSimdW + c];
            part += wa[u] * v.x + wb[u] * v.y;
          }
        }
      }
      block_sum_to((double)part, p.partial + blockIdx.x);
    } else {
      for (int pos = g; pos < P; pos += ng) {
        const V v = z[pos * kSimdW + c];
        if (sA < p.S) p.out_real[(o * P + pos) * p.S + sA] = v.x;
        if (sB < p.S) p.out_real[(o * P + pos) * p.S + sB] = v.y;
      }
    }
    return;
  }
  const int64_t s = (int64_t)blockIdx.x * kSimdW + c;
  const bool col_ok = s < p.S;
  // kLoadBatch independent loads in flight per thread before any is stored
  for (int pos0 = g; pos0 < P; pos0 += kLoadBatch * ng) {
    V v[kLoadBatch];
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int pos = pos0 + u * ng;
      const int n = source_row(pos, P, p.Lw, p.Nin);
      v[u] = (pos < P && n < p.Nin && col_ok) ? in[(int64_t)n * p.S + s] : mk<V>(0, 0);
    }
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int pos = pos0 + u * ng;
      if (pos < P) bufA[pos * kSimdW + c] = v[u];
    }
  }
  twiddles_wait();
  __syncthreads();
  // COL_MID: this thread's first kLoadBatch values of K, loaded before the
  // forward transform.
  T kpre[kLoadBatch];
  if (MODE == COL_MID) {
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int pos = g + u * ng;
      kpre[u] = (pos < P && col_ok) ? __ldg(p.K + (int64_t)pos * p.S + s) : T(0);
    }
  }
  V* z = (MODE == COL_INV) ? simd_fft<V, true>(bufA, bufB, p.lp, tw_s, c, g, ng)
                           : simd_fft<V, false>(bufA, bufB, p.lp, tw_s, c, g, ng);
  if (MODE == COL_MID) {
#pragma unroll
    for (int u = 0; u < kLoadBatch; ++u) {
      const int pos = g + u * ng;
      if (pos < P) {
        V v = z[pos * kSimdW + c];
        z[pos * kSimdW + c] = mk<V>(v.x * kpre[u], v.y * kpre[u]);
      }
    }
    for (int pos0 = g + kLoadBatch * ng; pos0 < P; pos0 += kLoadBatch * ng) {
      T kv[kLoadBatch];
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int pos = pos0 + u * ng;
        kv[u] = (pos < P && col_ok) ? __ldg(p.K + (int64_t)pos * p.S + s) : T(0);
      }
#pragma unroll
      for (int u = 0; u < kLoadBatch; ++u) {
        const int pos = pos0 + u * ng;
        if (pos < P) {
          V v = z[pos * kSimdW + c];
          z[pos * kSimdW + c] = mk<V>(v.x * kv[u], v.y * kv[u]);
        }
      }
    }
    __syncthreads();
    V* other = (z == bufA) ? bufB : bufA;
    z = simd_fft<V, true>(z, other, p.lp, tw_s, c, g, ng);
  }
  if (MODE == COL_AUTO) {
    for (int pos = g; pos < P; pos += ng) {
      const V v = z[pos * kSimdW + c];
      const T re = v.x * p.s_pre, im = v.y * p.s_pre;
      z[pos * kSimdW + c] = mk<V>((re * re + im * im) * p.s_post, T(0));
    }
    __syncthreads();
    V* other = (z == bufA) ? bufB : bufA;
    z = simd_fft<V, true>(z, other, p.lp, tw_s, c, g, ng);
  }
  if (!col_ok) return;
  if (MODE == COL_FWD_POWER) {
    const T w = (T)half_weight(s, p.Qw, p.Plw);
    const T sc = (T)2.3283064365386963e-10;  // 2^-32
    for (int pos = g; pos < P; pos += ng) {
      const V v = z[pos * kSimdW + c];
      const T re = v.x * sc, im = v.y * sc;
      p.out_real[(o * P + pos) * p.S + s] = w * (re * re + im * im);
    }
    return;
  }
  const int nout = (MODE == COL_FWD) ? P : p.Nout;
  for (int pos = g; pos < nout; pos += ng) p.out[(o * nout + pos) * p.S + s] = z[pos * kSimdW + c];
}

template <typename T, int MODE>
__device__ __forceinline__ void cols_simd_body(const ColsParams<T>& p) {
  cols_simd_body_slab<T, MODE>(p, blockIdx.y);
}

template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_fwd_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_FWD>(p);
  else
    cols_body<T, COL_FWD>(p);
}
template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_kgen_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_FWD>(p);
  else
    cols_body<T, COL_FWD>(p);
}
template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_kgen_real_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_FWD_REAL>(p);
  else
    cols_body<T, COL_FWD_REAL>(p);
}
template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_mid_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_MID>(p);
  else
    cols_body<T, COL_MID>(p);
}
template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_power_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_FWD_POWER>(p);
  else
    cols_body<T, COL_FWD_POWER>(p);
}
template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_auto_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_AUTO>(p);
  else
    cols_body<T, COL_AUTO>(p);
}



// Batched kernel spectra (Eq. 6 and Eq. 10 for many matrices at once): one
// chunk holds up to kBatch matrices; blockIdx.y picks the matrix.
constexpr int kBatch = 64;

template <typename T>
struct BatchKGen {
  int nb;
  KGen<T> gen[kBatch];
  int rows[kBatch];       // rows of the matrix's lag grid (2 L_0 + 1; 1 for d = 1)
  int64_t off[kBatch];    // its first row in the chunk's scratch (complex elements)
};

template <typename T>
__global__ void __launch_bounds__(256) kde_rows_kgen_batch_kernel(BatchKGen<T> bk, RowsParams<T> p) {
  const int b = blockIdx.y;
  if (b >= bk.nb) return;
  // this matrix's parameters in shared memory (a per-thread copy indexed at
  // run time would live in local memory)
  __shared__ RowsParams<T> q;
  __shared__ KGen<T> gen;
  if (threadIdx.x == 0) {
    q = p;
    q.nrows = bk.rows[b];
    if (p.out_real)
      q.out_real = p.out_real + (int64_t)b * p.Q;
    else
      q.out = p.out + bk.off[b];
    gen = bk.gen[b];
  }
  __syncthreads();
  rows_kgen_body<T>(gen, q, blockIdx.x);
}

// Axis-0 pass of the batched spectra, fused with the dot product against the
// count spectrum W: no kernel spectrum is written.  Partials are laid out
// [matrix][column block].
template <typename T, bool SIMD>
__global__ void __launch_bounds__(256) kde_cols_kgen_dot_kernel(BatchKGen<T> bk, ColsParams<T> p) {
  const int b = blockIdx.y;
  if (b >= bk.nb) return;
  __shared__ ColsParams<T> q;
  if (threadIdx.x == 0) {
    q = p;
    q.in = p.in + bk.off[b];
    q.Nin = bk.rows[b];
    q.Lw = bk.gen[b].L[0];
    q.partial = p.partial + (int64_t)b * gridDim.x;
  }
  __syncthreads();
  // the bodies index the outer slab by blockIdx.y; here there is one slab
  if (SIMD)
    cols_simd_body_slab<T, COL_FWD_DOT>(q, 0);
  else
    cols_body_slab<T, COL_FWD_DOT>(q, 0, blockIdx.x);
}

// d = 1: dot of the real spectrum of matrix b with W.
template <typename T>
__global__ void __launch_bounds__(256) kde_dot1d_kernel(int nb, const T* __restrict__ K, int Q,
                                                        const T* __restrict__ W,
                                                        double* __restrict__ partial) {
  const int b = blockIdx.x;
  if (b >= nb) return;
  T part = 0;
  for (int k = threadIdx.x; k < Q; k += blockDim.x) part += W[k] * K[(int64_t)b * Q + k];
  block_sum_to((double)part, partial + b);
}

// Pair sums S_b = scale * sum of the matrix's partials (fixed order, FP64),
// then LSCV_i = S(2H_i) / n^2 - 2 (S(H_i) - n K_{H_i}(0)) / (n (n - 1)) for
// matrices ordered H_0, 2H_0, H_1, 2H_1, ...
struct LscvReduce {
  int nb, nparts;
  double scale, n;
  double K0[kBatch / 2];
};

__global__ void __launch_bounds__(32) kde_lscv_reduce_kernel(LscvReduce r, const double* __restrict__ partial,
                                                             double* __restrict__ S_out,
                                                             double* __restrict__ lscv_out) {
  const int i = blockIdx.x;  // candidate within the chunk
  if (2 * i + 1 >= r.nb) return;
  double s[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double* pp = partial + (int64_t)(2 * i + h) * r.nparts;
    double v = 0.0;
    for (int j = threadIdx.x; j < r.nparts; j += 32) v += pp[j];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    s[h] = __shfl_sync(0xffffffffu, v, 0) * r.scale;
  }
  if (threadIdx.x == 0) {
    if (S_out) {
      S_out[2 * i] = s[0];
      S_out[2 * i + 1] = s[1];
    }
    lscv_out[i] = s[1] / (r.n * r.n) - 2.0 * (s[0] - r.n * r.K0[i]) / (r.n * (r.n - 1.0));
  }
}

// Binned pair sums from the counts' autocorrelation R (P_0 x P_1, lag
// (l_0, l_1) at (l_0 mod P_0, l_1 mod P_1)):
//   S(A) = sum_{|l_k| <= L_k} K_A(delta o l) R(l).
// K_A and R are even, so the sum runs over the half plane l_0 > 0, or
// l_0 = 0 and l_1 > 0, twice, plus the lag 0 once.
//
// Along lag row l_0 >= 0 the Gaussian is C exp(e) in the completed squares
// of KGen (d = 2, column lag m = l_1, or |l_1| in Wand's layout):
//   e = D_0 l_0^2 + D_1 (m + b l_0)^2,  b = B_10 = b_hi + b_lo,
// so per row e_0 = D_0 l_0^2 and b l_0 are formed once.  D_0 and D_1 are
// stored times log2(e) (scaled in FP64 on the host), so each term is one
// exp2 of the exponent in base-2 units.
template <typename T>
struct AcGen {
  int L0, L1, wand;
  int u0, nu;  // this matrix's work units [u0, u0 + nu), kAcRows lag rows each
  int set;     // whose autocorrelation: R + set * (P_0 P_1)
  T D0, D1, b_hi, b_lo, C;
};

// Up to kAcChunk candidates (2 kAcChunk matrices) per launch; their
// parameters and work units are uploaded to the workspace.  A work unit is
// kAcRows lag rows of one matrix (the last of a matrix fewer).
//
// FP32 sums.  The terms are FP32; how they are added is fixed here, for every
// kernel below, so that a candidate's score does not depend on how many
// datasets are scored with it or on how the work is spread:
//   chain   the lags l_1 = c (mod 8) of one row inside one window [S w, S (w +
//           1)), ascending, in FP32: S = 2^ac_shift(first row, L_0, L_1), S / 8 terms;
//   group   the 4 x 8 chains of four rows (first row a multiple of four), in
//           order of 8 (row mod 4) + c, as a pair of FP32 (AcPair: the sum and
//           the sum of its rounding errors);
//   unit    the groups of its two sets of four rows, windows ascending;
//   matrix  its units, every eighth in order, the eight sums as a tree
//           (kde_lscv_ac_reduce_kernel).
// From the chains on nothing is lost to FP32: LSCV subtracts two such sums,
// and rows of small far terms vanish in one long chain.  FP64 additions would
// do, but run at 2 lanes a clock and SM; a pair costs four to eight FP32 ones.  Error
// of the additions alone, rms over random bandwidths (x 1e-9), with chains
// through eight rows and a FP32 tree / with a warp's row sums added in FP32 and
// the lanes in FP64 (what the widths below are held against) / now: supports
// of 39 x 39 lags 31 / 4.9 / 3.2, 120 x 120 22 / 2.4 / 1.8, 7 x 2000 1000 / 39
// / 5, 27 x 70 36 / 4.4 / 4.1, 7 x 32 43 / 5.3 / 5.1, 10 x 10 45 / 8.3 / 5.6; over
// 60 random shapes 0.39 of the second on average.
constexpr int kAcChunk = 1024;
constexpr int kAcRows = 8;
constexpr int kAcGroup = 4;       // rows of a group
constexpr int kAcWindow = 128;    // widest window
// Width of the windows, as its log2 (nothing is divided): 64 lags, chains of
// eight terms; 128 lags for supports above 256, where a row had as many terms
// to a lane before (60 x 165 lags 3.1 / 2.2 with 64, 3.7 with 128; 60 x 400 6.1 /
// 1.6, 3.1); and short ones, but at most sixteen a side, in the first unit, which
// holds the largest terms, of a support of few rows, where it is nearly all
// there is (5 x 48 lags 5.2 / 8.1 with 64, 4.3 with 16).
__host__ __device__ constexpr int ac_shift(int row0, int L0, int L1) {
  int b = row0 == 0 && L0 < 24 ? 4 : L1 > 256 ? 7 : 6;
  while (b < 7 && (16 << b) < L1) ++b;
  return b;
}
static_assert(kAcWindow == 1 << 7, "");
// Windows that hold lags -L1 .. L1: ac_first .. L1 >> b.
__host__ __device__ constexpr int ac_first(int L1, int b) { return -((L1 + (1 << b) - 1) >> b); }
__host__ __device__ constexpr int ac_windows(int L1, int b) { return (L1 >> b) - ac_first(L1, b) + 1; }

// A sum as value + error, |error| about half an ulp of the value.
struct AcPair {
  float s, e;
};
// The exact error of s = a + b rounded (Knuth's two-sum).
__device__ __forceinline__ float sum_error(float a, float b, float s) {
  const float bb = __fsub_rn(s, a);
  return __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ AcPair ac_add(AcPair a, AcPair b) {
  AcPair r;
  r.s = __fadd_rn(a.s, b.s);
  r.e = __fadd_rn(__fadd_rn(a.e, b.e), sum_error(a.s, b.s, r.s));
  return r;
}
// The same two at a time (component by component).
struct AcPair2 {
  float2 s, e;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 sum_error2(float2 a, float2 b, float2 s) {
  const float2 bb = sub2(s, a);
  return __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
}
__device__ __forceinline__ AcPair2 ac_add2(AcPair2 a, AcPair2 b) {
  AcPair2 r;
  r.s = __fadd2_rn(a.s, b.s);
  r.e = __fadd2_rn(__fadd2_rn(a.e, b.e), sum_error2(a.s, b.s, r.s));
  return r;
}

// K_A at lag (l0, l1) over 2 C: every lag of the half plane counts twice,
// the lag 0 once; zero outside the support and on the other half of row 0.
template <typename T>
struct AcRow {
  T t_hi, t_lo, e0;
};
template <typename T>
__device__ __forceinline__ AcRow<T> ac_row(const AcGen<T>& g, int l0) {
  const T tl = (T)l0;
  AcRow<T> r;
  r.t_hi = g.b_hi * tl;
  r.t_lo = prod_lo(g.b_hi, g.b_lo, tl, r.t_hi);
  r.e0 = g.D0 * tl * tl;
  return r;
}
// 2^x by the hardware's approximation, with results below 2^-126 (1e-38 of
// the lag 0 term) flushed to zero instead of scaled through.
__device__ __forceinline__ float ac_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Two terms in packed arithmetic: lags l.x, l.y (as floats: an integer
// conversion would take the exponential's unit) with the parameters D1, t_hi,
// t_lo, e0 of each.
__device__ __forceinline__ float2 ac_term2(float2 l, float2 D1, float2 t_hi, float2 t_lo, float2 e0) {
  const float2 v = __fadd2_rn(__fadd2_rn(l, t_hi), t_lo);
  const float2 e = __ffma2_rn(__fmul2_rn(D1, v), v, e0);
  return make_float2(ac_ex2(e.x), ac_ex2(e.y));
}

// A lane's row of a group: its parameters and its lags [lo, lo + span].
struct AcLane {
  float2 D1, th, tl, e0;
  const float* x;   // lag 0 of the row in shared memory
  int lo;
  unsigned span;
};
__device__ __forceinline__ AcLane ac_lane(const AcGen<float>& g, int l0, const float* x) {
  AcLane a;
  const AcRow<float> r = ac_row(g, l0);
  a.D1 = make_float2(g.D1, g.D1);
  a.th = make_float2(r.t_hi, r.t_hi);
  a.tl = make_float2(r.t_lo, r.t_lo);
  a.e0 = make_float2(r.e0, r.e0);
  a.x = x;
  // none in a row beyond the support, half of them in row 0
  a.lo = l0 > g.L0 ? KDE_MAX_P : l0 == 0 ? 0 : -g.L1;
  a.span = l0 > g.L0 ? 0u : (unsigned)(g.L1 - a.lo);
  return a;
}
// This lane's chain of the window of S lags from w0 on, for the group of rows
// r0 .. r0 + 3 of matrix g.
__device__ __forceinline__ float ac_chain(const AcGen<float>& g, const AcLane& a, int r0, int w0,
                                          int S, int c) {
  const unsigned sign = g.wand ? 0x7FFFFFFFu : 0xFFFFFFFFu;
  float acc = 0.f;
  auto terms = [&](float2 f) {
    const float2 l = make_float2(__uint_as_float(__float_as_uint(f.x) & sign),
                                 __uint_as_float(__float_as_uint(f.y) & sign));
    return ac_term2(l, a.D1, a.th, a.tl, a.e0);
  };
  const float2 step = make_float2(16.f, 16.f);
  const int i0 = max(0, (-g.L1 - w0) >> 3), i1 = min(S - 1, g.L1 - w0) >> 3;
  if (r0 > 0 && r0 + kAcGroup - 1 <= g.L0) {   // whole rows: only the ends can lie outside
    int l = w0 + 8 * i0 + c;
    const float* x = a.x + l;
    float2 f = make_float2((float)l, (float)(l + 8));
    int i = i0;
    auto pair = [&](bool whole) {
      const float2 k = terms(f);
      if (whole || (l >= -g.L1 && l <= g.L1)) acc = fmaf(k.x, x[0], acc);
      if (whole || (i < i1 && l + 8 <= g.L1)) acc = fmaf(k.y, x[8], acc);
      f = __fadd2_rn(f, step);
      l += 16;
      x += 16;
      i += 2;
    };
    const int last = w0 + 8 * i1 + 7 > g.L1 ? i1 - 1 : i1;
    if (w0 + 8 * i0 < -g.L1) pair(false);
#pragma unroll 4
    while (i < last) pair(true);
    while (i <= i1) pair(false);
    return acc;
  }
  int l = w0 + 8 * i0 + c;
  float2 f = make_float2((float)l, (float)(l + 8));
  for (int i = i0; i <= i1; i += 2, l += 16) {
    float2 k = terms(f);
    if (r0 == 0 && (threadIdx.x & 24) == 0) {   // row 0: its lag 0 counts once, the others twice
      if (l == 0) k.x *= 0.5f;
      if (l + 8 == 0) k.y *= 0.5f;
    }
    if ((unsigned)(l - a.lo) <= a.span) acc = fmaf(k.x, a.x[l], acc);
    if (i < i1 && (unsigned)(l + 8 - a.lo) <= a.span) acc = fmaf(k.y, a.x[l + 8], acc);
    f = __fadd2_rn(f, step);
  }
  return acc;
}

// A group's sum from its chains v[0] .. v[31].  The error is taken as for |sum|
// >= |chain|; where the first few chains grow it falls short by what one FP32
// addition of them rounds (no larger errors in the sums measured above).
__device__ __forceinline__ AcPair ac_group_sum(const float* v) {
  AcPair p{v[0], 0.f};
#pragma unroll
  for (int r = 1; r < 32; ++r) {
    const float b = v[r], s = __fadd_rn(p.s, b);
    p.e = __fadd_rn(p.e, __fadd_rn(__fsub_rn(p.s, s), b));
    p.s = s;
  }
  return p;
}

// A block's groups: those of unit row0 of nm <= 32 matrices (gs) dealt out to
// its warps in runs, their sums into sums in order (matrix, set of four rows,
// window), matrix m's at off[m].  A warp leaves the chains of `held` <= 32 groups
// in its turn of shared memory and a lane then adds each group's: shuffles for
// each took a third of the kernel.  tile: lag (row0, 0).
constexpr int kAcTurn1 = 33;   // pitch of the chains
// off, by one warp; complete after the block's next barrier.
__device__ __forceinline__ void ac_offsets(const AcGen<float>* gs, int nm, int row0, int* off) {
  const int lane = threadIdx.x & 31;
  int v = 0;
  if (lane < nm && row0 <= gs[lane].L0)
    v = (kAcRows / kAcGroup) * ac_windows(gs[lane].L1, ac_shift(row0, gs[lane].L0, gs[lane].L1));
#pragma unroll
  for (int d = 1; d < 32; d *= 2) {
    const int u = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += u;
  }
  if (lane < nm) off[lane + 1] = v;
  if (lane == 0) off[0] = 0;
}
__device__ __forceinline__ void ac_groups(const AcGen<float>* gs, const int* off, int nm, int row0,
                                          const float* tile, int pitch, float* turn, int held,
                                          AcPair* sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int end = off[nm] * (warp + 1) / warps, rs = lane >> 3, c = lane & 7;
  int t = off[nm] * warp / warps, m = 0, w = 0, b = 0, last = -1, r0 = 0;
  turn += warp * held * kAcTurn1;
  AcLane a{};
  AcGen<float> g{};
  while (t < end) {
    const int n = min(held, end - t);
    for (int k = 0; k < n; ++k, ++w) {
      if (w > last) {   // the next set of four rows, or where the run begins
        while (off[m + 1] <= t + k) ++m;
        g = gs[m];
        b = ac_shift(row0, g.L0, g.L1);
        const int first = ac_first(g.L1, b), j = t + k - off[m];
        last = g.L1 >> b;
        const int nw = last - first + 1, h = j >= nw;
        w = first + j - h * nw;
        r0 = row0 + kAcGroup * h;
        a = ac_lane(g, r0 + rs, tile + (kAcGroup * h + rs) * pitch);
      }
      turn[k * kAcTurn1 + lane] = r0 <= g.L0 ? ac_chain(g, a, r0, w << b, 1 << b, c) : 0.f;
    }
    __syncwarp();
    if (lane < n) sums[t + lane] = ac_group_sum(turn + lane * kAcTurn1);
    __syncwarp();
    t += n;
  }
}

// The groups' sums, behind the turns of the block's warps.
__device__ __forceinline__ AcPair* ac_sums(float* turn, int held) {
  return reinterpret_cast<AcPair*>(turn + (((int)(blockDim.x >> 5) * held * kAcTurn1 + 1) & ~1));
}

// Lag rows row0 .. row0 + nrow - 1 of R, lags -L1 .. L1, into tile by the
// whole block; complete for the block after ac_staged.  Row r starts at r
// pitch; the pitch of 8 (mod 32) words keeps a group's four rows on different
// banks.
__host__ __device__ constexpr int ac_pitch(int L1) { return (2 * L1 + 1 + 23) / 32 * 32 + 8; }
__device__ __forceinline__ void ac_stage(float* tile, const float* __restrict__ R, int P1, int row0,
                                         int nrow, int L1) {
  const int W = 2 * L1 + 1, pitch = ac_pitch(L1);
  for (int r = threadIdx.x >> 5; r < nrow; r += blockDim.x >> 5) {
    const float* Rrow = R + (size_t)(row0 + r) * P1;
    uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile + r * pitch + (threadIdx.x & 31));
    for (int i = threadIdx.x & 31; i < W; i += 32, dst += 128)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst),
                   "l"(__cvta_generic_to_global(Rrow + (i < L1 ? i - L1 + P1 : i - L1)))
                   : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void ac_staged() {
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  __syncthreads();
}

// FP64: a block a work unit, a warp a lag row.  The terms are bound by the
// FP64 pipe (about twenty instructions of it each), so what counts is that
// every SM has rows: with a warp a whole unit and its sixteen to a block, as
// the FP32 kernel has them, 16 candidates of 460-lag supports took 723 us
// against 398.
__global__ void __launch_bounds__(256) kde_lscv_ac64_kernel(const AcGen<double>* __restrict__ gens,
                                                            const int2* __restrict__ units,
                                                            const double* __restrict__ Rall, int P1,
                                                            int64_t set_stride,
                                                            double* __restrict__ partial) {
  const int2 u = units[blockIdx.x];
  const AcGen<double> g = gens[u.x];
  const int lane = threadIdx.x & 31, l0 = u.y + (threadIdx.x >> 5);
  double acc = 0.0;
  if (l0 <= g.L0) {
    const double* R = Rall + (int64_t)(g.set + blockIdx.y) * set_stride + (int64_t)l0 * P1;
    const AcRow<double> r = ac_row(g, l0);
#pragma unroll 4
    for (int l1 = (l0 == 0 ? 0 : -g.L1) + lane; l1 <= g.L1; l1 += 32) {
      const double v = ((double)(g.wand ? abs(l1) : l1) + r.t_hi) + r.t_lo;
      acc = fma(exp2(fma(g.D1 * v, v, r.e0)), __ldg(R + (l1 < 0 ? l1 + P1 : l1)), acc);
    }
    // every lag of the half plane counts twice, the lag 0 (K = C) once
    if (l0 == 0 && lane == 0) acc -= 0.5 * __ldg(R);
  }
  block_sum_to(acc, partial + (int64_t)(g.u0 + u.y / kAcRows) * gridDim.y + blockIdx.y);
}

// A block takes up to `sub` work units (matrix, first row) of one dataset and
// first row, a part of blocks[..] = (first unit, count <= kAcBlock): partial[u nsets + y] with u
// the unit's place among its matrix's units, for the autocorrelation g.set +
// y, y = blockIdx.y.  The units' lag rows are staged in shared memory once
// (the first unit's L_1 is the largest); read from the L2 as they are used,
// one load's latency for 32 terms was most of the kernel.  The block's groups
// are dealt out to its warps, their sums left in shared memory and added
// there in order, so that a few wide supports keep every warp at work too.
// The 2048 matrices of 1024 candidates at 512^2 take 31 us (24 with chains
// through eight rows and a tree of shuffles, whose additions err ten times as
// far): 72% of the issue slots, integer and comparison work 59% of its pipe,
// exponentials 10%, shared memory 19%.
constexpr int kAcBlock = 16;
// Warps of a block: twice as many where the staged rows leave room for one
// block an SM.
constexpr int kAcThreads = 512;
__host__ __device__ constexpr int ac_threads(int L1) {
  return 2 * kAcRows * ac_pitch(L1) * (int)sizeof(float) > 110 * 1024 ? kAcThreads : kAcThreads / 2;
}
// Groups of a unit at most, over supports up to L1.
__host__ __device__ constexpr int ac_unit_groups(int L1) {
  return (kAcRows / kAcGroup) * (L1 <= 256 ? ac_windows(L1, 4) : 33);
}
// Groups whose chains a warp holds at a time, with `matrices` units a block.
__host__ __device__ constexpr int ac_turn(int L1, int matrices, int threads) {
  const int n = (matrices * ac_unit_groups(L1) * 32 + threads - 1) / threads;
  return n < 32 ? n : 32;
}
__host__ __device__ constexpr size_t ac_block_smem(int L1, int matrices, int threads) {
  return (size_t)kAcRows * ac_pitch(L1) * sizeof(float) +
         (size_t)(threads / 32) * ac_turn(L1, matrices, threads) * kAcTurn1 * sizeof(float) +
         (size_t)matrices * ac_unit_groups(L1) * sizeof(AcPair) + sizeof(AcPair);
}
static_assert(ac_windows(KDE_MAX_P / 2 - 1, 7) <= 33 && ac_windows(256, ac_shift(0, 0, 256)) <= 33 &&
                  ac_windows(512, ac_shift(0, 0, 512)) <= 33 && ac_windows(1024, ac_shift(0, 0, 1024)) <= 33,
              "windows of a row");
static_assert(ac_block_smem(KDE_MAX_P / 2 - 1, kAcBlock, kAcThreads) + 4096 <= kSmemMax,
              "the widest support's rows and groups fit in shared memory");

__global__ void __launch_bounds__(kAcThreads) kde_lscv_ac_kernel(
    const AcGen<float>* __restrict__ gens, const int2* __restrict__ units,
    const int2* __restrict__ blocks, const float* __restrict__ Rall, int P1, int64_t set_stride,
    int sub, int held, AcPair* __restrict__ partial) {
  extern __shared__ __align__(16) float tile[];
  __shared__ AcGen<float> gs[kAcBlock];
  __shared__ int off[kAcBlock + 1];
  const int parts = (kAcBlock + sub - 1) / sub, part = blockIdx.x % parts;
  int2 blk = blocks[blockIdx.x / parts];
  blk.y = min(sub, blk.y - part * sub);
  if (blk.y <= 0) return;
  units += blk.x + part * sub;
  const int row0 = units[0].y, tid = threadIdx.x;
  if (tid < blk.y) gs[tid] = gens[units[tid].x];
  __syncthreads();
  const float* __restrict__ R = Rall + (int64_t)(gs[0].set + blockIdx.y) * set_stride;
  const int L1 = gs[0].L1, pitch = ac_pitch(L1);
  // rows below the support of the block's longest matrix (never past R)
  int L0 = 0;
  for (int i = 0; i < blk.y; ++i) L0 = max(L0, gs[i].L0);
  ac_stage(tile, R, P1, row0, min(kAcRows, L0 + 1 - row0), L1);
  float* turn = tile + kAcRows * pitch;
  AcPair* sums = ac_sums(turn, held);
  if (tid < 32) ac_offsets(gs, blk.y, row0, off);
  ac_staged();
  ac_groups(gs, off, blk.y, row0, tile + L1, pitch, turn, held, sums);
  __syncthreads();
  if (tid < blk.y) {
    AcPair v{0.f, 0.f};
#pragma unroll 4
    for (int j = off[tid]; j < off[tid + 1]; ++j) v = ac_add(v, sums[j]);
    partial[(int64_t)(gs[tid].u0 + row0 / kAcRows) * gridDim.y + blockIdx.y] = v;
  }
}

// Many datasets scored against one candidate set.  A kernel value serves
// every dataset, so the sums are a matrix product (matrices x lags) (lags x
// datasets).  A warp takes the work units of kAcQuad matrices with the same
// L_1 on one first row, a lane one chain of a group: per lag it forms the four
// kernel values once and sums them against kAcSets datasets, whose lags a
// block stages in shared memory kAcWindow lags of four rows at a time
// (datasets innermost, so that a lane's kAcSets values are four 16-byte loads;
// the pitch of 20 words keeps them free of bank conflicts) for its 16 warps,
// the next tile's copies in flight.  After a window each warp turns its 64 x
// 32 chains through shared memory, so that a lane adds the 32 chains of two
// sums.  A lane outside the support reads a slot of zeros, so that a value
// that does not count is never touched.  256 datasets x 2016 matrices of 5 to
// 108 lags (1.8 G terms, 49 us at the FP32 rate): 392 us, 3172 one by one.  Its
// shared memory moves as much for the chains' ends as for the terms, half of
// its rate with the four warps a scheduler that 64 sums a lane leave.  Tried: a
// thread 4 x 4 or 8 x 4 sums with the kernel values formed in shared memory,
// chains ending in registers (446 us: a third of its instructions are the ends
// of short chains, and an item of 190 lags alone takes 310).
constexpr int kAcQuad = 4, kAcSets = 16, kAcPitch = 20;
constexpr int kAcWarps = 16;
constexpr int kAcTurn = kAcQuad * kAcSets + 4;   // pitch of the turned chains
constexpr int kAcSlab = 256;     // datasets per launch
// Fewer datasets are scored one by one, and so are few work units: an item of
// the product takes as long for one dataset as for sixteen (18 us + 0.4 a lag of
// its widest support), and few items leave SMs idle, where a (unit, dataset)
// pair one by one takes 2.1 ns + 0.004 a lag.  One by one / product, us with
// the reduction: 343 candidates up to 30 lags (2e3 units) 32 / 36 with 7 / 8
// datasets, 32 up to 60 lags (340 units) 32 / 47 with 24, 46 / 47 with 64, 32 up
// to 190 lags (1100 units) 52 / 94 with 12, 78 / 95 with 24, 4 of them 45 / 69
// with 64.
constexpr int kAcMinSets = 8;
bool ac_product(int ns, int nunits, int nitems, int L1, int sms) {
  const int64_t blocks = (int64_t)nitems * ((ns + kAcSets - 1) / kAcSets);
  return ns >= kAcMinSets && (int64_t)nunits * ns * (2.1 + 0.004 * L1) >
                                 (double)((blocks + sms - 1) / sms) * (18000.0 + 400.0 * L1);
}
constexpr int kAcTile = kAcGroup * kAcWindow * kAcPitch;
constexpr size_t kAcSetsSmem =
    sizeof(float) * (2 * kAcTile + 2 * kAcPitch + (size_t)kAcWarps * 32 * kAcTurn);
static_assert(kAcSetsSmem <= kSmemMax, "tiles and turned chains fit in shared memory");

// The matrices of one warp: the same L_1 and windows, falling L_0 (m[0]'s the
// largest).
struct AcGroup {
  int m[kAcQuad];   // matrix or -1
  int L0, L1;
};

// Lags max(w0, -Lw) .. min(w0 + kAcWindow - 1, Lw) of lag rows t0 .. t0 + nrow - 1 of
// nset datasets into a tile (one committed group of 4-byte asynchronous
// copies; no copy and no value for datasets beyond).
__device__ __forceinline__ void ac_stage_sets(float* tile, const float* __restrict__ R, int P1,
                                              int64_t set_stride, int t0, int nrow, int nset,
                                              int w0, int Lw) {
  const int lane = threadIdx.x & 31, b = max(w0, -Lw), e = min(w0 + kAcWindow - 1, Lw);
  for (int q = threadIdx.x >> 5; q < nrow * nset; q += kAcWarps) {
    const int r = q / nset, d = q - r * nset;
    const float* Rrow = R + (int64_t)d * set_stride + (int64_t)(t0 + r) * P1;
    uint32_t dst = (uint32_t)__cvta_generic_to_shared(
        tile + (r * kAcWindow + b - w0 + lane) * kAcPitch + d);
    for (int l1 = b + lane; l1 <= e; l1 += 32, dst += 32 * kAcPitch * 4)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(dst),
                   "l"(__cvta_generic_to_global(Rrow + (l1 < 0 ? l1 + P1 : l1)))
                   : "memory");
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// ac_group_sum for two sums at a time (v: their columns, rows kAcTurn apart).
__device__ __forceinline__ AcPair2 ac_group_sum2(const float* v) {
  AcPair2 p{*reinterpret_cast<const float2*>(v), make_float2(0.f, 0.f)};
#pragma unroll
  for (int r = 1; r < 32; ++r) {
    const float2 b = *reinterpret_cast<const float2*>(v + r * kAcTurn), s = __fadd2_rn(p.s, b);
    p.e = __fadd2_rn(p.e, __fadd2_rn(sub2(p.s, s), b));
    p.s = s;
  }
  return p;
}

__global__ void __launch_bounds__(32 * kAcWarps, 1) kde_lscv_ac_sets_kernel(
    const AcGen<float>* __restrict__ gens, const AcGroup* __restrict__ groups,
    const int3* __restrict__ items, const float* __restrict__ Rall, int P1, int64_t set_stride,
    int ns, AcPair* __restrict__ partial) {
  extern __shared__ __align__(16) float tiles[];   // 2 x [row][lag][kAcPitch]
  float* zero = tiles + 2 * kAcTile;               // a lag's datasets: zeros,
  float* half = zero + kAcPitch;                   // and half of lag (0, 0)
  const int3 it = items[blockIdx.x];              // first group, groups, first row
  const int s0 = blockIdx.y * kAcSets, nset = min(kAcSets, ns - s0);
  const int Lw = groups[it.x].L1, row0 = it.z;   // L_1 falls along the groups
  int Lmax = 0;
  for (int i = 0; i < it.y; ++i) Lmax = max(Lmax, groups[it.x + i].L0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, rs = lane >> 3, c = lane & 7;
  float* turn = half + kAcPitch + warp * 32 * kAcTurn;
  const bool act = warp < it.y && groups[it.x + (warp < it.y ? warp : 0)].L0 >= row0;
  const AcGroup gr = groups[it.x + (act ? warp : 0)];
  float2 acc[kAcQuad][kAcSets / 2];
#pragma unroll
  for (int m = 0; m < kAcQuad; ++m)
#pragma unroll
    for (int d = 0; d < kAcSets / 2; ++d) acc[m][d] = make_float2(0.f, 0.f);
  const float* R = Rall + (int64_t)s0 * set_stride;
  // datasets beyond the last read as zeros
  for (int i = threadIdx.x; i < 2 * kAcTile + 2 * kAcPitch; i += blockDim.x) tiles[i] = 0.f;
  __syncthreads();
  const int nw = ac_windows(Lw, 7), first = ac_first(Lw, 7);
  const int ntile = nw * ((min(kAcRows, Lmax + 1 - row0) + kAcGroup - 1) / kAcGroup);
  auto stage = [&](int t) {
    if (t < ntile) {
      const int h = t / nw, r0 = row0 + kAcGroup * h;
      ac_stage_sets(tiles + (t & 1) * kAcTile, R, P1, set_stride, r0, min(kAcGroup, Lmax + 1 - r0),
                    nset, (first + t - h * nw) * kAcWindow, Lw);
    } else {
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
  };
  stage(0);
  AcPair2 sum{make_float2(0.f, 0.f), make_float2(0.f, 0.f)};   // sums 2 lane, 2 lane + 1
  float2 D1[2], th[2], tl[2], e0[2];
  int lo = 0;
  unsigned span = 0, sign = 0;
  const int shift = ac_shift(row0, gr.L0, gr.L1), S = 1 << shift;
  for (int t = 0; t < ntile; ++t) {
    const int h = t / nw, w0 = (first + t - h * nw) * kAcWindow, r0 = row0 + kAcGroup * h;
    const float* tile = tiles + (t & 1) * kAcTile;
    stage(t + 1);
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    if (r0 == 0 && w0 == 0) {
      if (threadIdx.x < kAcSets) half[threadIdx.x] = 0.5f * tile[threadIdx.x];
      __syncthreads();
    }
    const int l0 = r0 + rs;
    if (act && t == h * nw) {   // the lane's row of each matrix
      lo = l0 > gr.L0 ? KDE_MAX_P : l0 == 0 ? 0 : -gr.L1;
      span = l0 > gr.L0 ? 0u : (unsigned)(gr.L1 - lo);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        AcGen<float> g[2];
        AcRow<float> a[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int m = gr.m[2 * q + j];
          g[j] = gens[m >= 0 ? m : gr.m[0]];
          a[j] = ac_row(g[j], l0);
          if (m < 0 || l0 > g[j].L0) a[j].e0 = -INFINITY;   // no term
        }
        D1[q] = make_float2(g[0].D1, g[1].D1);
        th[q] = make_float2(a[0].t_hi, a[1].t_hi);
        tl[q] = make_float2(a[0].t_lo, a[1].t_lo);
        e0[q] = make_float2(a[0].e0, a[1].e0);
        sign = g[0].wand ? 0x7FFFFFFFu : 0xFFFFFFFFu;
      }
    }
    if (act && r0 <= gr.L0) {
      // the tile's windows, the support's first to its last
      const int v0 = max(w0, ac_first(gr.L1, shift) * S), v1 = min(w0 + kAcWindow - 1, gr.L1);
      for (int v = v0; v <= v1; v += S) {
        const int i0 = max(0, (-gr.L1 - v) >> 3), i1 = min(S - 1, gr.L1 - v) >> 3;
        int l = v + 8 * i0 + c;
        float f = (float)l;
        const float* x = tile + (rs * kAcWindow + l - w0) * kAcPitch;
        for (int i = i0; i <= i1; ++i, l += 8, f += 8.f, x += 8 * kAcPitch) {
          const float lf = __uint_as_float(__float_as_uint(f) & sign);
          float2 k[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) k[q] = ac_term2(make_float2(lf, lf), D1[q], th[q], tl[q], e0[q]);
          const float* xs = (unsigned)(l - lo) <= span ? x : zero;
          if (l == 0 && l0 == 0) xs = half;
          const float4* xv = reinterpret_cast<const float4*>(xs);
          const float km[kAcQuad] = {k[0].x, k[0].y, k[1].x, k[1].y};
#pragma unroll
          for (int q = 0; q < kAcSets / 4; ++q) {
            const float4 y = xv[q];
#pragma unroll
            for (int m = 0; m < kAcQuad; ++m) {
              const float2 kk = make_float2(km[m], km[m]);
              acc[m][2 * q] = __ffma2_rn(kk, make_float2(y.x, y.y), acc[m][2 * q]);
              acc[m][2 * q + 1] = __ffma2_rn(kk, make_float2(y.z, y.w), acc[m][2 * q + 1]);
            }
          }
        }
        // turn: this lane's chains into a row, then two columns of 32 back
        float4* row = reinterpret_cast<float4*>(turn + lane * kAcTurn);
#pragma unroll
        for (int m = 0; m < kAcQuad; ++m)
#pragma unroll
          for (int q = 0; q < kAcSets / 4; ++q) {
            const float2 a = acc[m][2 * q], b = acc[m][2 * q + 1];
            row[m * (kAcSets / 4) + q] = make_float4(a.x, a.y, b.x, b.y);
            acc[m][2 * q] = acc[m][2 * q + 1] = make_float2(0.f, 0.f);
          }
        __syncwarp();
        sum = ac_add2(sum, ac_group_sum2(turn + 2 * lane));
        __syncwarp();
      }
    }
    __syncthreads();
  }
  if (!act) return;
  const int m = groups[it.x + warp].m[(2 * lane) / kAcSets];
  if (m < 0) return;
  const AcGen<float>& g = gens[m];
  if (row0 > g.L0) return;
  AcPair* out = partial + (int64_t)(g.u0 + row0 / kAcRows) * ns + s0;
  const int d = (2 * lane) % kAcSets;
  if (d < nset) out[d] = AcPair{sum.s.x, sum.e.x};
  if (d + 1 < nset) out[d + 1] = AcPair{sum.s.y, sum.e.y};
}

// {n, 1 / n^2, 2 / (n (n - 1))}: the LSCV's factors, formed once per dataset
// on the host (an FP64 division costs more than the rest of a score's
// reduction).
struct NTerms {
  double v[3];
};

// A work unit's sum over 2 C as it is stored, and such sums added.
template <typename T>
using AcPart = std::conditional_t<std::is_same<T, float>::value, AcPair, double>;
__device__ __forceinline__ double ac_add(double a, double b) { return a + b; }
__device__ __forceinline__ double ac_value(double v) { return v; }
__device__ __forceinline__ double ac_value(AcPair v) { return (double)v.s + (double)v.e; }

// S(H), S(2H) per (candidate, dataset) as the sums of their units' partials,
// and the LSCV.  Class c of a matrix's units takes every eighth from c on, in
// order; the classes' sums are added as a tree.  With many scores a thread
// takes a score; with few a warp takes a class of 32 scores, as one thread
// waited for one load after another (64 candidates of 1800 lags 85 us, now
// 15).  The n terms are the dataset's (nk_set), or nk_all, or with nk_all.v[0]
// = 0 the candidate's (kn: {K_H(0), n terms}).  Outputs at y nH_all + i.
constexpr int kAcClasses = 8;
template <typename T, bool MANY>
__global__ void __launch_bounds__(256) kde_lscv_ac_reduce_kernel(
    const AcGen<T>* __restrict__ gens, const double* __restrict__ kn,
    const NTerms* __restrict__ nk_set, NTerms nk_all, const AcPart<T>* __restrict__ partial, int nh,
    int ns, int64_t nH_all, double* __restrict__ S_out, double* __restrict__ lscv_out) {
  constexpr int kScores = MANY ? 256 : 32;
  const int lane = threadIdx.x % kScores, p = threadIdx.x / kScores;
  const int64_t t = (int64_t)blockIdx.x * kScores + lane;
  const bool in = t < (int64_t)nh * ns;
  const int i = in ? (int)(t / ns) : 0, y = (int)(t - (int64_t)i * ns);
  const AcGen<T>*g0 = gens + 2 * i, *g1 = g0 + 1;
  const int nu0 = in ? g0->nu : 0, nu1 = in ? g1->nu : 0;
  const AcPart<T>*p0 = partial + (int64_t)g0->u0 * ns + y, *p1 = partial + (int64_t)g1->u0 * ns + y;
  AcPart<T> v[2] = {};
  if constexpr (MANY) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const AcPart<T>* ph = h ? p1 : p0;
      const int nu = h ? nu1 : nu0;
      AcPart<T> c[kAcClasses] = {};
      for (int j = 0; j < nu; j += kAcClasses) {
        AcPart<T> a[kAcClasses];   // loads in flight
#pragma unroll
        for (int k = 0; k < kAcClasses; ++k) a[k] = j + k < nu ? ph[(int64_t)(j + k) * ns] : AcPart<T>{};
#pragma unroll
        for (int k = 0; k < kAcClasses; ++k) c[k] = ac_add(c[k], a[k]);
      }
#pragma unroll
      for (int off = kAcClasses / 2; off > 0; off >>= 1)
#pragma unroll
        for (int k = 0; k < off; ++k) c[k] = ac_add(c[k], c[k + off]);
      v[h] = c[0];
    }
  } else {
    __shared__ AcPart<T> part[2][kAcClasses][kScores];
    for (int j = p; j < max(nu0, nu1); j += 8 * kAcClasses) {
      AcPart<T> a[8], b[8];   // loads in flight
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int u = j + k * kAcClasses;
        a[k] = u < nu0 ? p0[(int64_t)u * ns] : AcPart<T>{};
        b[k] = u < nu1 ? p1[(int64_t)u * ns] : AcPart<T>{};
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        v[0] = ac_add(v[0], a[k]);
        v[1] = ac_add(v[1], b[k]);
      }
    }
    part[0][p][lane] = v[0];
    part[1][p][lane] = v[1];
#pragma unroll
    for (int off = kAcClasses / 2; off > 0; off >>= 1) {
      __syncthreads();
      if (p < off)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          v[h] = ac_add(v[h], part[h][p + off][lane]);
          part[h][p][lane] = v[h];
        }
    }
    if (p) return;
  }
  if (!in) return;
  const double s0 = 2.0 * (double)g0->C * ac_value(v[0]), s1 = 2.0 * (double)g1->C * ac_value(v[1]);
  double nk[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    nk[k] = nk_set ? nk_set[y].v[k] : nk_all.v[0] > 0.0 ? nk_all.v[k] : kn[4 * (int64_t)i + 1 + k];
  const int64_t o = y * nH_all + i;
  if (S_out) {
    S_out[2 * o] = s0;
    S_out[2 * o + 1] = s1;
  }
  lscv_out[o] = s1 * nk[1] - nk[2] * (s0 - nk[0] * kn[4 * (int64_t)i]);
}

// S(A) from a matrix's class sums, stride apart.
__device__ __forceinline__ double ac_class_sum(const AcGen<float>& g, const AcPair* c, int64_t stride) {
  AcPair v[kAcClasses];
#pragma unroll
  for (int k = 0; k < kAcClasses; ++k) v[k] = c[k * stride];
#pragma unroll
  for (int off = kAcClasses / 2; off > 0; off >>= 1)
#pragma unroll
    for (int k = 0; k < off; ++k) v[k] = ac_add(v[k], v[k + off]);
  return g.L0 < 0 ? nan("") : 2.0 * (double)g.C * ac_value(v[0]);
}

// ---------------------------------------------------------------------------
// Candidates of the learned proposal built and scored on the device: for
// dataset s, candidate j < J is the network's theta_s clipped to a box plus
// offset j, candidate J the reference theta_s; theta = (a, beta, c) stands
// for H = R R^T with R = [[e^a, 0], [beta e^c, e^c]].  Each candidate gives
// the two matrices A = H and A = 2H of the LSCV criterion.
// ---------------------------------------------------------------------------
struct ThetaArgs {
  int nsets, J;
  const float* theta;     // nsets x 3 (device)
  const double* n;        // nsets
  const double* ref;      // nsets x 3
  const double* off;      // J x 3
  double box_lo[3], box_hi[3];
  double tau, delta[2];
  int M[2], P[2];
  int wand, per_axis;
  AcGen<float>* gens;     // [nsets][J + 1][2]; L0 < 0 marks a candidate that does not fit
  double* K0;             // [nsets][J + 1]: K_H(0)
};

// One thread per matrix: the same FP64 steps as the host path (H from
// theta, support by Eq. 15, Cholesky factor, completed-square constants),
// rounded to the lag sums' FP32 parameters.  Blocks of one warp: FP64 bound,
// so the warps are spread over every SM.
__global__ void __launch_bounds__(32) kde_theta_gen_kernel(ThetaArgs t) {
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t per = 2 * (int64_t)(t.J + 1);
  if (m >= (int64_t)t.nsets * per) return;
  const int s = (int)(m / per), r = (int)(m % per), j = r >> 1, h = r & 1;
  double th[3];
  for (int k = 0; k < 3; ++k) {
    if (j < t.J) {
      const double v = (double)t.theta[3 * s + k];
      th[k] = fmin(fmax(v, t.box_lo[k]), t.box_hi[k]) + t.off[3 * j + k];
    } else {
      th[k] = t.ref[3 * s + k];
    }
  }
  const double ea = exp(th[0]), ec = exp(th[2]), b = th[1] * ec, sc = h ? 2.0 : 1.0;
  const double A00 = sc * (ea * ea), A01 = sc * (ea * b), A11 = sc * (b * b + ec * ec);
  const double mid = 0.5 * (A00 + A11), hd = 0.5 * (A00 - A11);
  const double lam = mid + sqrt(hd * hd + A01 * A01);
  int L[2];
  bool ok = isfinite(lam) && A00 > 0.0;
  const double Akk[2] = {A00, A11};
  for (int k = 0; k < 2; ++k) {
    const double half = t.per_axis ? t.tau * sqrt(Akk[k]) : t.tau * sqrt(fabs(lam));
    const double c = ceil(half / t.delta[k]);
    L[k] = c >= (double)(t.M[k] - 1) ? t.M[k] - 1 : (int)c;
    ok = ok && t.M[k] + L[k] <= t.P[k];
  }
  const double r00 = sqrt(A00), r10 = A01 / r00, r11 = sqrt(A11 - r10 * r10);
  ok = ok && r11 > 0.0;
  const double i00 = 1.0 / r00, i11 = 1.0 / r11, i10 = -(r10 * i00) / r11;
  const double D0 = -0.5 * t.delta[0] * t.delta[0] * i00 * i00;
  const double D1 = -0.5 * t.delta[1] * t.delta[1] * i11 * i11;
  const double B = i10 * t.delta[0] / (i11 * t.delta[1]);
  const double det = (r00 * r11) * (r00 * r11);
  const double C = (1.0 / 6.283185307179586476925287) / sqrt(det);
  const double log2e = 1.4426950408889634073599246810;
  AcGen<float> g{};
  g.L0 = ok ? L[0] : -1;
  g.L1 = L[1];
  g.wand = t.wand;
  g.set = s;
  g.D0 = (float)(D0 * log2e);
  g.D1 = (float)(D1 * log2e);
  g.b_hi = (float)B;
  g.b_lo = (float)(B - (double)g.b_hi);
  g.C = (float)C;
  t.gens[m] = g;
  if (h == 0) t.K0[m >> 1] = C;
}

// A block takes up to nc <= kThetaCands candidates of one dataset (two matrices
// each) and every nr-th unit of eight lag rows (nr divides kAcClasses): S(A) =
// sum over the support of K_A(delta o l) R(l), the rows staged in shared memory
// a unit at a time, their groups dealt out to the warps and added as
// kde_lscv_ac_kernel's are, the units in the classes of
// kde_lscv_ac_reduce_kernel (classes: [class][matrix] over 2 C; with nr = 1 the
// block adds them, S).  NaN for a matrix that does not fit the plan.  Few
// datasets take fewer candidates and rows a block, so that every SM has work:
// one dataset of 28 candidates 78 us with seven and all rows a block, 6 now.
// 256 datasets of 28 candidates of 12 to 130 lags (116 M terms) take 165 us: a
// group has six terms a lane on average, and its setup and sum cost about as
// much as they do.
constexpr int kThetaCands = 7;
constexpr int kThetaThreads = 128;
// Blocks of nsets x cands candidates: nc to a block (as many as leave ten
// blocks an SM with the rows split eight ways), nr blocks to their rows.
struct ThetaSplit {
  int nc, nr;
};
ThetaSplit theta_split(int64_t nsets, int64_t cands, int sms) {
  const int64_t want = 10 * (int64_t)sms;
  ThetaSplit p{1, 1};
  while (p.nc < kThetaCands && nsets * cands * kAcClasses >= (p.nc + 1) * want) ++p.nc;
  const int64_t blocks = nsets * ((cands + p.nc - 1) / p.nc);
  while (p.nr < kAcClasses && blocks * p.nr < want) p.nr *= 2;
  return p;
}
// L1max: an upper bound of the supports along axis 1.
__global__ void __launch_bounds__(kThetaThreads) kde_lscv_theta_sums_kernel(
    const AcGen<float>* __restrict__ gens, int per, int nc, const float* __restrict__ Rall, int P1,
    int64_t set_stride, int L1max, int held, int64_t nmat, AcPair* __restrict__ classes,
    double* __restrict__ S) {
  extern __shared__ __align__(16) float tile[];
  __shared__ AcGen<float> gs[2 * kThetaCands];
  __shared__ int off[2 * kThetaCands + 1];
  __shared__ AcPair cls[2 * kThetaCands][kAcClasses];
  float* turn = tile + kAcRows * ac_pitch(L1max);
  AcPair* sums = ac_sums(turn, held);
  const int tid = threadIdx.x;
  const int ngroups = (per + 2 * nc - 1) / (2 * nc), set = blockIdx.x / ngroups;
  const int first = 2 * nc * (blockIdx.x - set * ngroups);
  const int nm = min(2 * nc, per - first);
  const int64_t mat = (int64_t)set * per + first;
  const float* __restrict__ R = Rall + (int64_t)set * set_stride;
  if (tid < nm) {
    gs[tid] = gens[mat + tid];
    for (int k = 0; k < kAcClasses; ++k) cls[tid][k] = AcPair{0.f, 0.f};
  }
  __syncthreads();
  int L0 = -1, L1 = 0;
  for (int m = 0; m < nm; ++m)
    if (gs[m].L0 >= 0) {
      L0 = max(L0, gs[m].L0);
      L1 = max(L1, gs[m].L1);
    }
  for (int row0 = kAcRows * blockIdx.y; row0 <= L0; row0 += kAcRows * gridDim.y) {
    ac_stage(tile, R, P1, row0, min(kAcRows, L0 + 1 - row0), L1);
    if (tid < 32) ac_offsets(gs, nm, row0, off);
    ac_staged();
    ac_groups(gs, off, nm, row0, tile + L1, ac_pitch(L1), turn, held, sums);
    __syncthreads();
    if (tid < nm) {
      AcPair v{0.f, 0.f};
#pragma unroll 4
      for (int j = off[tid]; j < off[tid + 1]; ++j) v = ac_add(v, sums[j]);
      AcPair& c = cls[tid][row0 / kAcRows % kAcClasses];
      c = ac_add(c, v);
    }
    __syncthreads();   // off is written again
  }
  if (tid >= nm) return;
  if (gridDim.y == 1) {
    S[mat + tid] = ac_class_sum(gs[tid], cls[tid], 1);
  } else {
    for (int k = blockIdx.y; k < kAcClasses; k += gridDim.y) classes[k * nmat + mat + tid] = cls[tid][k];
  }
}

// One warp per dataset: LSCV of its J + 1 candidates (optionally stored; S, or
// with classes not null the sums' classes),
// the first index of the smallest among the first J (a candidate that does
// not fit counts as +inf) and out[s] = {that index, its LSCV, the reference
// candidate's LSCV, that candidate's theta}.
__global__ void __launch_bounds__(32) kde_lscv_theta_pick_kernel(ThetaArgs t,
                                                                 const double* __restrict__ S,
                                                                 const AcPair* __restrict__ classes,
                                                                 int64_t nmat,
                                                                 double* __restrict__ lscv,
                                                                 double* __restrict__ out) {
  const int J = t.J;
  const double* __restrict__ n_all = t.n;
  const double* __restrict__ K0 = t.K0;
  const int s = blockIdx.x;
  const double n = n_all[s];
  double best = HUGE_VAL;
  int bi = J;   // no candidate fits
  double ref = HUGE_VAL;
  for (int j = threadIdx.x; j <= J; j += 32) {
    const int64_t c = (int64_t)s * (J + 1) + j;
    const double s1 = classes ? ac_class_sum(t.gens[2 * c], classes + 2 * c, nmat) : S[2 * c];
    const double s2 = classes ? ac_class_sum(t.gens[2 * c + 1], classes + 2 * c + 1, nmat) : S[2 * c + 1];
    double v = s2 / (n * n) - 2.0 * (s1 - n * K0[c]) / (n * (n - 1.0));
    if (isnan(v)) v = HUGE_VAL;
    if (lscv) lscv[c] = v;
    if (j == J) ref = v;
    else if (v < best) {   // j increases per lane, so the first smallest is kept
      best = v;
      bi = j;
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const double ov = __shfl_down_sync(0xffffffffu, best, off);
    const int oi = __shfl_down_sync(0xffffffffu, bi, off);
    if (ov < best || (ov == best && oi < bi)) {
      best = ov;
      bi = oi;
    }
    ref = fmin(ref, __shfl_down_sync(0xffffffffu, ref, off));
  }
  if (threadIdx.x == 0) {
    double th[3] = {0.0, 0.0, 0.0};
    if (bi < J)
      for (int k = 0; k < 3; ++k) {
        const double v = (double)t.theta[3 * s + k];
        th[k] = fmin(fmax(v, t.box_lo[k]), t.box_hi[k]) + t.off[3 * bi + k];
      }
    double* o = out + 6 * (int64_t)s;
    o[0] = (double)bi;
    o[1] = best;
    o[2] = ref;
    o[3] = th[0];
    o[4] = th[1];
    o[5] = th[2];
  }
}

template <typename T, bool SIMD>
__global__ void __launch_bounds__(kColsMaxThreads) kde_cols_inv_kernel(ColsParams<T> p) {
  if (SIMD)
    cols_simd_body<T, COL_INV>(p);
  else
    cols_body<T, COL_INV>(p);
}

// ---------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------
LinePlan line_plan(const kde_plan_info& info, int k) {
  LinePlan lp{};
  lp.N = (int)info.P[k];
  lp.nst = info.nstages[k];
  int Ns = 1;
  for (int s = 0; s < lp.nst; ++s) {
    Stage& st = lp.st[s];
    st.R = info.radix[k][s];
    st.Ns = Ns;
    st.nb = lp.N / st.R;
    st.twstep = lp.N / (Ns * st.R);
    st.magic = (unsigned)((1ull << 32) / (unsigned)Ns + 1ull);
    Ns *= st.R;
  }
  return lp;
}

template <typename T>
const typename Cplx<T>::type* twiddles(const kde_plan_s* plan, int k) {
  return reinterpret_cast<const typename Cplx<T>::type*>((const char*)plan->tw_dev + plan->tw_offset[k]);
}

static int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
      sms = 152;
  }
  return sms;
}

// Launch shape for `lines` lines of length P: threads per line (tpl) grows
// with the work per line and shrinks as lines multiply, aiming at about 16
// resident warps per SM; blocks hold up to 256 threads (lines * tpl) within
// shared memory (twiddles plus two buffers per line).
struct LineShape {
  int tpl, lpb;
};

template <typename T>
LineShape line_shape(int64_t lines, int P, int lpb_min) {
  const size_t cb = sizeof(typename Cplx<T>::type);
  const int64_t target_warps = 16LL * num_sms();
  int64_t per_line = (target_warps + lines - 1) / std::max<int64_t>(1, lines);
  int tpl = 32;
  // about one radix-8 butterfly (P/8 per stage) per thread at most, and
  // room for lpb_min lines in a 256-thread block
  const int tpl_max = std::max(32, std::min(256 / lpb_min, ((P / 8 + 31) / 32) * 32));
  while (tpl * 2 <= tpl_max && tpl / 32 < per_line) tpl *= 2;
  int lpb = std::max(1, 256 / tpl);
  const int lpb_smem = (int)((kSmemMax / cb - P) / (2 * (size_t)P + 1));
  lpb = std::max(1, std::min(lpb, lpb_smem));
  // keep at least two blocks per SM where the line count allows
  while (lpb > lpb_min && (lines + lpb - 1) / lpb < 2 * num_sms()) lpb /= 2;
  lpb = std::max(lpb, std::min(lpb_min, lpb_smem));
  return {tpl, lpb};
}

template <typename T>
size_t line_smem(int P, int W) {
  return ((size_t)(1 + 2 * W) * P + W) * sizeof(typename Cplx<T>::type);
}

// Row kernels take the launch shape in their parameters (p.tpl).
template <typename T, typename Kern, typename Params, typename... Args>
kde_status launch_rows(Kern* fn, const char* name, int64_t nrows, Params& p, cudaStream_t st,
                       Args... args) {
  const int P = p.lp.N;
  const int64_t pairs = (nrows + 1) / 2;
  const LineShape sh = line_shape<T>(pairs, P, 1);
  p.tpl = sh.tpl;
  cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
  LaunchScope ls(name, st);
  fn<<<(unsigned)((pairs + sh.lpb - 1) / sh.lpb), sh.tpl * sh.lpb, line_smem<T>(P, sh.lpb), st>>>(
      args..., p);
  e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, name);
}

// Column passes with at least this many 16-column tiles per SM, and whose
// tiles fit twice per SM, use the SIMD-across-columns body.
template <typename T>
bool simd_cols(int variant, int64_t columns, int P) {
  const size_t smem = (size_t)(1 + 2 * kSimdW) * P * sizeof(typename Cplx<T>::type);
  if (variant == KDE_COLS_LINES || smem > 100 * 1024) return false;
  return variant == KDE_COLS_SIMD || columns >= (int64_t)4 * kSimdW * num_sms();
}

// Threads of a SIMD column block: kSimdW lanes per butterfly group and the
// number of groups ng in 16..32 that leaves the fewest idle lanes over the
// plan's stages (a stage of nb butterflies takes ceil(nb / ng) rounds; for
// P = 280 = 8 7 5 the stages hold 35, 40, 56 butterflies: 82% of the lanes
// busy with 16 groups, 94% with 20), the larger ng on a tie.
static int simd_threads(const LinePlan& lp) {
  int best_ng = 16;
  double best = -1.0;
  for (int ng = 16; ng <= kColsMaxThreads / kSimdW; ng += 4) {
    int64_t work = 0, slots = 0;
    for (int s = 0; s < lp.nst; ++s) {
      const int nb = lp.st[s].nb;
      work += nb;
      slots += (int64_t)((nb + ng - 1) / ng) * ng;
    }
    const double u = (double)work / (double)slots;
    if (u > best + 1e-12 || (u > best - 1e-12 && ng > best_ng)) {
      best = u;
      best_ng = ng;
    }
  }
  return best_ng * kSimdW;
}

template <typename T>
using ColsKernel = void (*)(ColsParams<T>);

template <typename T>
kde_status launch_cols(ColsKernel<T> fn_lines, ColsKernel<T> fn_simd, ColsParams<T> p, int64_t O,
                       int variant, cudaStream_t st, const char* name, bool paired = false) {
  const int P = p.lp.N;
  const int per = paired ? 2 : 1;  // columns per transformed line
  cudaError_t e;
  if (simd_cols<T>(variant, p.S * O, P)) {
    if ((e = allow_smem(fn_simd)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    const size_t smem = (size_t)(1 + 2 * kSimdW) * P * sizeof(typename Cplx<T>::type);
    dim3 grid((unsigned)((p.S + per * kSimdW - 1) / (per * kSimdW)), (unsigned)O);
    LaunchScope ls(name, st);
    fn_simd<<<grid, simd_threads(p.lp), smem, st>>>(p);
  } else {
    const LineShape sh = line_shape<T>((p.S + per - 1) / per * O, P, 2);
    p.tpl = sh.tpl;
    const int W = sh.lpb * per;  // columns per block
    if ((e = allow_smem(fn_lines)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    dim3 grid((unsigned)((p.S + W - 1) / W), (unsigned)O);
    LaunchScope ls(name, st);
    fn_lines<<<grid, sh.tpl * sh.lpb, line_smem<T>(P, sh.lpb), st>>>(p);
  }
  e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, name);
}

#define KDE_COLS(kern) kern<T, false>, kern<T, true>

// Kernel-grid parameters of K_A (no 1/n, 2^-32 or 1/prod P folded in).
template <typename T>
kde_status kgen_for(const kde_plan_info& I, const double* A, double detA, const int64_t* L,
                    int wand, KGen<T>* g) {
  double D[3], B[3];
  kde_status st = gauss_factor(I.d, A, I.delta, D, B);
  if (st != KDE_OK) return st;
  *g = KGen<T>{};
  g->d = I.d;
  g->wand = wand;
  for (int k = 0; k < I.d; ++k) {
    g->L[k] = (int)L[k];
    g->D[k] = (T)D[k];
  }
  for (int e = 0; e < 3; ++e) {
    g->Bh[e] = (T)B[e];
    g->Bl[e] = (T)(B[e] - (double)g->Bh[e]);
  }
  g->C = (T)(std::pow(6.283185307179586476925287, -0.5 * I.d) / std::sqrt(detA));
  return KDE_OK;
}

// FP64 2-D kernel grids with small supports: both passes as direct sums over
// the lags, spread over the chip.  An FP64 line transform is one warp's (or a
// few) dependent stages whatever the support; the sums are (L_0 + 1) Q L_1 and
// P_0 Q L_0 terms.  Transforms against sums, both passes (us, graph of ten,
// GB300): 32^2, L = 3 17.4 / 2.7; 128^2, L = 15 23.8 / 4.5; 256^2, L = 30 26.4
// / 11.9; 400^2, L = 24 (2.2 M terms) 34 / 22; 256^2, L = 64 (3.1 M) 27 / 27.
//
// Rows: block l_0 forms T(l_0, q) = sum_{l_1} k e^{-2 pi i q l_1 / P_1} for the
// lags l_0 >= 0, a thread a frequency: with s, d = k(l_0, l_1) +- k(l_0, -l_1),
// Re T = k(l_0, 0) + sum s cos, Im T = -sum d sin.  Nothing here reads what the
// kernels before it write, so only the store waits for them.
__global__ void __launch_bounds__(128) kde_rows_kgen_sums_kernel(KGen<double> gen, int P, int Q,
                                                                 const double2* __restrict__ tw,
                                                                 double2* __restrict__ out) {
  extern __shared__ __align__(16) double2 ks[];   // (s, d) of lag l_1 >= 1; ks[0].x = k(l_0, 0)
  pdl_trigger();
  const int l0 = blockIdx.x, L1 = gen.L[1];
  for (int l1 = threadIdx.x; l1 <= L1; l1 += blockDim.x) {
    const int p[KDE_MAX_D] = {l0, l1, 0}, m[KDE_MAX_D] = {l0, -l1, 0};
    const double kp = kernel_value(gen, p), km = kernel_value(gen, m);
    ks[l1] = l1 ? make_double2(kp + km, kp - km) : make_double2(kp, 0.0);
  }
  __syncthreads();
  const int q = blockIdx.y * blockDim.x + threadIdx.x;
  double re = ks[0].x, im = 0.0;
  if (q < Q) {
    int m = 0;
#pragma unroll 4
    for (int l1 = 1; l1 <= L1; ++l1) {
      m += q;
      if (m >= P) m -= P;
      const double2 w = __ldg(tw + m), k = ks[l1];
      re = fma(k.x, w.x, re);
      im = fma(k.y, w.y, im);
    }
  }
  pdl_wait();
  if (q < Q) out[(int64_t)l0 * Q + q] = make_double2(re, im);
}

// Columns: block q forms K(w, q) = T(0, q) + 2 Re sum_{l_0 >= 1} T(l_0, q)
// e^{-2 pi i w l_0 / P_0}, a thread a frequency (T(-l_0) is T(l_0)'s
// conjugate); stored at w sw + q sq.
__global__ void __launch_bounds__(128) kde_cols_kgen_sums_kernel(const double2* __restrict__ in, int L0,
                                                                 int P, int Q,
                                                                 const double2* __restrict__ tw,
                                                                 double* __restrict__ K, int64_t sw,
                                                                 int64_t sq) {
  extern __shared__ __align__(16) double2 t_sm[];
  pdl_trigger();
  pdl_wait();
  const int q = blockIdx.x;
  for (int l = threadIdx.x; l <= L0; l += blockDim.x) t_sm[l] = in[(int64_t)l * Q + q];
  __syncthreads();
  const int w = blockIdx.y * blockDim.x + threadIdx.x;
  if (w >= P) return;
  double s = 0.0;
  int m = 0;
#pragma unroll 4
  for (int l = 1; l <= L0; ++l) {
    m += w;
    if (m >= P) m -= P;
    const double2 e = __ldg(tw + m), t = t_sm[l];
    s = fma(t.x, e.x, fma(-t.y, e.y, s));
  }
  K[w * sw + q * sq] = t_sm[0].x + 2.0 * s;
}

// Terms up to which each pass is the shorter as sums.
constexpr int64_t kKgenSums = 3 << 20;

template <typename T>
kde_status kernel_grid_impl(kde_plan_s* plan, int64_t n, void* Kspec, void* ws, cudaStream_t st) {
  using V = typename Cplx<T>::type;
  const kde_plan_info& I = plan->info;
  const int d = I.d;
  KGen<T> gen;
  kde_status st0 = kgen_for<T>(I, plan->H, I.det_H, I.L, plan->layout_mode == KDE_LAYOUT_WAND, &gen);
  if (st0 != KDE_OK) return st0;
  double prodP = 1.0;
  for (int k = 0; k < d; ++k) prodP *= (double)I.P[k];
  const double two_pi = 6.283185307179586476925287;
  double C = std::pow(two_pi, -0.5 * d) / std::sqrt(I.det_H) / ((double)n * 4294967296.0 * prodP);
  gen.C = (T)C;
  if constexpr (std::is_same<T, float>::value) {
    if (I.engine == KDE_ENGINE_TWO_PHASE) return fx_kernel_grid(plan, gen, Kspec, ws, st);
  }
  const int dl = d - 1;
  RowsParams<T> rp{};
  rp.Q = (int)I.Q;
  rp.Min = 0;
  rp.lp = line_plan(I, dl);
  rp.tw = twiddles<T>(plan, dl);
  if (d == 1) {
    bool taken = false;
    const kde_status s1 = line1d_kernel_grid<T>(plan, gen, (T*)Kspec, st, &taken);
    if (s1 != KDE_OK || taken) return s1;
    rp.nrows = 1;
    rp.out_real = (T*)Kspec;
    return launch_rows<T>(kde_rows_r2c_kgen_kernel<T>, "kde_rows_r2c_kgen_kernel", 1, rp, st, gen);
  }
  V* t1 = (V*)ws;
  if constexpr (std::is_same<T, double>::value) {
    if (d == 2 && (I.L[0] + 1) * I.Q * I.L[1] <= kKgenSums && I.P[0] * I.Q * I.L[0] <= kKgenSums) {
      const int Q = (int)I.Q, P0 = (int)I.P[0], L0 = (int)I.L[0];
      cudaError_t e;
      {
        LaunchScope ls("kde_rows_kgen_sums_kernel", st);
        e = launch_pdl(kde_rows_kgen_sums_kernel, dim3((unsigned)(L0 + 1), (unsigned)((Q + 127) / 128)),
                       dim3(128), (size_t)(I.L[1] + 1) * sizeof(double2), st, gen, (int)I.P[1], Q,
                       twiddles<T>(plan, 1), t1);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return cuda_fail(e, "kde_rows_kgen_sums_kernel");
      }
      // the layout the middle pass reads (launch_cols)
      const bool simd = simd_cols<T>(plan->cols_variant, I.Q, P0);
      LaunchScope ls("kde_cols_kgen_sums_kernel", st);
      e = launch_pdl(kde_cols_kgen_sums_kernel, dim3((unsigned)Q, (unsigned)((P0 + 127) / 128)),
                     dim3(128), (size_t)(L0 + 1) * sizeof(double2), st, (const double2*)t1, L0, P0, Q,
                     twiddles<T>(plan, 0), (double*)Kspec, simd ? (int64_t)Q : (int64_t)1,
                     simd ? (int64_t)1 : (int64_t)P0);
      if (e == cudaSuccess) e = cudaGetLastError();
      return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_cols_kgen_sums_kernel");
    }
  }
  int64_t rows = 1;
  for (int k = 0; k < d - 1; ++k) rows *= 2 * I.L[k] + 1;
  rp.nrows = rows;
  rp.out = t1;
  kde_status s = launch_rows<T>(kde_rows_r2c_kgen_kernel<T>, "kde_rows_r2c_kgen_kernel", rows, rp,
                                st, gen);
  if (s != KDE_OK) return s;
  if (d == 2) {
    ColsParams<T> cp{};
    cp.in = t1;
    cp.out_real = (T*)Kspec;
    cp.S = I.Q;
    cp.Nin = (int)(2 * I.L[0] + 1);
    cp.Lw = (int)I.L[0];
    cp.lp = line_plan(I, 0);
    cp.tw = twiddles<T>(plan, 0);
    return launch_cols<T>(KDE_COLS(kde_cols_kgen_real_kernel), cp, 1, plan->cols_variant, st,
                          "kde_cols_kgen_real_kernel", true);
  }
  // d == 3: axis 1 (wrapped) into t2, then axis 0 (wrapped) to the real spectrum.
  V* t2 = t1 + rows * I.Q;
  ColsParams<T> c1{};
  c1.in = t1;
  c1.out = t2;
  c1.S = I.Q;
  c1.Nin = (int)(2 * I.L[1] + 1);
  c1.Lw = (int)I.L[1];
  c1.lp = line_plan(I, 1);
  c1.tw = twiddles<T>(plan, 1);
  s = launch_cols<T>(KDE_COLS(kde_cols_kgen_kernel), c1, 2 * I.L[0] + 1, plan->cols_variant, st, "kde_cols_kgen_kernel");
  if (s != KDE_OK) return s;
  ColsParams<T> c0{};
  c0.in = t2;
  c0.out_real = (T*)Kspec;
  c0.S = I.P[1] * I.Q;
  c0.Nin = (int)(2 * I.L[0] + 1);
  c0.Lw = (int)I.L[0];
  c0.lp = line_plan(I, 0);
  c0.tw = twiddles<T>(plan, 0);
  return launch_cols<T>(KDE_COLS(kde_cols_kgen_real_kernel), c0, 1, plan->cols_variant, st,
                        "kde_cols_kgen_real_kernel", true);
}

// First pass: counts rows -> half spectra, by the FFT engine or (plans
// with dft_tc) by the tensor-core DFT-matrix product.
template <typename T>
kde_status counts_rows(kde_plan_s* plan, const long long* cnt, int64_t rows, RowsParams<T>& rp,
                       cudaStream_t st) {
  if (plan->dft_tc && sizeof(T) == sizeof(float)) return dft_tc_rows(plan, cnt, rows, rp.out, st);
  return launch_rows<T>(kde_rows_r2c_counts_kernel<T>, "kde_rows_r2c_counts_kernel", rows, rp, st,
                        cnt);
}

template <typename T>
kde_status fft_eval_impl(kde_plan_s* plan, const int64_t* counts, const void* Kspec, void* density,
                         void* ws, cudaStream_t st) {
  using V = typename Cplx<T>::type;
  const kde_plan_info& I = plan->info;
  const int d = I.d;
  const int dl = d - 1;
  const long long* cnt = reinterpret_cast<const long long*>(counts);
  if constexpr (std::is_same<T, float>::value) {
    if (I.engine == KDE_ENGINE_TWO_PHASE)
      return fx_fft_eval(plan, cnt, (const float*)Kspec, (float*)density, ws, st);
  }
  if (d == 1) {
    bool taken = false;
    const kde_status s1 = line1d_eval<T>(plan, cnt, (const T*)Kspec, (T*)density, st, &taken);
    if (s1 != KDE_OK || taken) return s1;
    const int P = (int)I.P[0];
    auto* fn = kde_line1d_kernel<T>;
    cudaError_t e = allow_smem(fn);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    LaunchScope ls("kde_line1d_kernel", st);
    fn<<<1, 256, line_smem<T>(P, 1), st>>>(cnt, (const T*)Kspec, (T*)density, (int)I.M[0], (int)I.Q,
                                          line_plan(I, 0), twiddles<T>(plan, 0));
    e = cudaGetLastError();
    return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_line1d_kernel");
  }
  V* A = (V*)ws;  // [M_0 .. M_{d-2}][Q]
  int64_t rows = 1;
  for (int k = 0; k < d - 1; ++k) rows *= I.M[k];
  RowsParams<T> rp{};
  rp.nrows = rows;
  rp.Min = (int)I.M[dl];
  rp.in_stride = I.M[dl];
  rp.Q = (int)I.Q;
  rp.out = A;
  rp.lp = line_plan(I, dl);
  rp.tw = twiddles<T>(plan, dl);
  kde_status s = counts_rows<T>(plan, cnt, rows, rp, st);
  if (s != KDE_OK) return s;
  if (d == 2) {
    ColsParams<T> cp{};
    cp.in = A;
    cp.out = A;
    cp.K = (const T*)Kspec;
    cp.S = I.Q;
    cp.Nin = (int)I.M[0];
    cp.Nout = (int)I.M[0];
    cp.Lw = -1;
    cp.lp = line_plan(I, 0);
    cp.tw = twiddles<T>(plan, 0);
    s = launch_cols<T>(KDE_COLS(kde_cols_mid_kernel), cp, 1, plan->cols_variant, st, "kde_cols_mid_kernel");
    if (s != KDE_OK) return s;
  } else {
    V* B = A + rows * I.Q;  // [M_0][P_1][Q]
    ColsParams<T> c1{};
    c1.in = A;
    c1.out = B;
    c1.S = I.Q;
    c1.Nin = (int)I.M[1];
    c1.Lw = -1;
    c1.lp = line_plan(I, 1);
    c1.tw = twiddles<T>(plan, 1);
    s = launch_cols<T>(KDE_COLS(kde_cols_fwd_kernel), c1, I.M[0], plan->cols_variant, st, "kde_cols_fwd_kernel");
    if (s != KDE_OK) return s;
    ColsParams<T> c0{};
    c0.in = B;
    c0.out = B;
    c0.K = (const T*)Kspec;
    c0.S = I.P[1] * I.Q;
    c0.Nin = (int)I.M[0];
    c0.Nout = (int)I.M[0];
    c0.Lw = -1;
    c0.lp = line_plan(I, 0);
    c0.tw = twiddles<T>(plan, 0);
    s = launch_cols<T>(KDE_COLS(kde_cols_mid_kernel), c0, 1, plan->cols_variant, st, "kde_cols_mid_kernel");
    if (s != KDE_OK) return s;
    ColsParams<T> ci{};
    ci.in = B;
    ci.out = A;
    ci.S = I.Q;
    ci.Nin = (int)I.P[1];
    ci.Nout = (int)I.M[1];
    ci.Lw = -1;
    ci.lp = line_plan(I, 1);
    ci.tw = twiddles<T>(plan, 1);
    s = launch_cols<T>(KDE_COLS(kde_cols_inv_kernel), ci, I.M[0], plan->cols_variant, st, "kde_cols_inv_kernel");
    if (s != KDE_OK) return s;
  }
  C2RParams<T> cr{};
  cr.in = A;
  cr.out = (T*)density;
  cr.nrows = rows;
  cr.Mout = (int)I.M[dl];
  cr.Q = (int)I.Q;
  cr.lp = line_plan(I, dl);
  cr.tw = twiddles<T>(plan, dl);
  return launch_rows<T>(kde_rows_c2r_kernel<T>, "kde_rows_c2r_kernel", rows, cr, st);
}

// ---------------------------------------------------------------------------
// Count spectrum and batched pair sums (bandwidth selection by LSCV).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) kde_power1d_kernel(const typename Cplx<T>::type* __restrict__ X,
                                                          T* __restrict__ W, int Q, int P) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < Q; k += gridDim.x * blockDim.x) {
    const T sc = (T)2.3283064365386963e-10;  // 2^-32
    const T re = X[k].x * sc, im = X[k].y * sc;
    W[k] = (T)half_weight(k, Q, P) * (re * re + im * im);
  }
}

// W = w(k) |2^-32 C|^2 on the half spectrum, in the kernel spectrum's order.
template <typename T>
kde_status power_spectrum_impl(kde_plan_s* plan, const int64_t* counts, void* Wout, void* ws,
                               cudaStream_t st) {
  using V = typename Cplx<T>::type;
  const kde_plan_info& I = plan->info;
  const int d = I.d, dl = d - 1;
  const long long* cnt = reinterpret_cast<const long long*>(counts);
  V* A = (V*)ws;
  int64_t rows = 1;
  for (int k = 0; k < d - 1; ++k) rows *= I.M[k];
  RowsParams<T> rp{};
  rp.nrows = rows;
  rp.Min = (int)I.M[dl];
  rp.in_stride = I.M[dl];
  rp.Q = (int)I.Q;
  rp.out = A;
  rp.lp = line_plan(I, dl);
  rp.tw = twiddles<T>(plan, dl);
  kde_status s = counts_rows<T>(plan, cnt, rows, rp, st);
  if (s != KDE_OK) return s;
  if (d == 1) {
    LaunchScope ls("kde_power1d_kernel", st);
    kde_power1d_kernel<T><<<(unsigned)((I.Q + 255) / 256), 256, 0, st>>>(A, (T*)Wout, (int)I.Q,
                                                                         (int)I.P[0]);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_power1d_kernel");
  }
  const V* src = A;
  int64_t S = I.Q;
  if (d == 3) {
    V* B = A + rows * I.Q;
    ColsParams<T> c1{};
    c1.in = A;
    c1.out = B;
    c1.S = I.Q;
    c1.Nin = (int)I.M[1];
    c1.Lw = -1;
    c1.lp = line_plan(I, 1);
    c1.tw = twiddles<T>(plan, 1);
    s = launch_cols<T>(KDE_COLS(kde_cols_fwd_kernel), c1, I.M[0], plan->cols_variant, st,
                       "kde_cols_fwd_kernel");
    if (s != KDE_OK) return s;
    src = B;
    S = I.P[1] * I.Q;
  }
  ColsParams<T> c0{};
  c0.in = src;
  c0.out_real = (T*)Wout;
  c0.S = S;
  c0.Nin = (int)I.M[0];
  c0.Lw = -1;
  c0.lp = line_plan(I, 0);
  c0.tw = twiddles<T>(plan, 0);
  c0.Qw = (int)I.Q;
  c0.Plw = (int)I.P[dl];
  return launch_cols<T>(KDE_COLS(kde_cols_power_kernel), c0, 1, plan->cols_variant, st,
                        "kde_cols_power_kernel");
}

// Scratch for one chunk of kBatch matrices: lag-grid rows (at most
// 2 (P_0 - M_0) + 1 per matrix, since every accepted matrix has
// M_0 + L_0 <= P_0) and the partial sums.
size_t lscv_workspace(const kde_plan_info& I) {
  const size_t cb = (I.precision == KDE_F32) ? 8 : 16;
  const int64_t rows_max = (I.d == 1) ? 1 : 2 * (I.P[0] - I.M[0]) + 1;
  int64_t S = I.Q;
  if (I.d == 3) S = I.P[1] * I.Q;
  // lag rows of the last axis for d = 2; d = 1 keeps one real spectrum row
  const size_t t1 = (size_t)kBatch * rows_max * I.Q * cb;
  const size_t parts = (size_t)kBatch * (size_t)(S + 1) * sizeof(double);
  return ((t1 + 255) & ~(size_t)255) + parts;
}

template <typename T>
kde_status lscv_impl(kde_plan_s* plan, int64_t n, int nH, const double* Hs, const void* Wsp,
                     double* S_out, double* lscv_out, void* ws, cudaStream_t st) {
  using V = typename Cplx<T>::type;
  const kde_plan_info& I = plan->info;
  const int d = I.d;
  double prodP = 1.0;
  for (int k = 0; k < d; ++k) prodP *= (double)I.P[k];
  const size_t cb = sizeof(V);
  const int64_t rows_max = (d == 1) ? 1 : 2 * (I.P[0] - I.M[0]) + 1;
  const size_t t1_bytes = ((size_t)kBatch * rows_max * I.Q * cb + 255) & ~(size_t)255;
  V* T1 = (V*)ws;
  double* partial = (double*)((char*)ws + t1_bytes);
  int64_t S = I.Q;
  const int chunk_h = kBatch / 2;
  for (int h0 = 0; h0 < nH; h0 += chunk_h) {
    const int nh = std::min(chunk_h, nH - h0);
    BatchKGen<T> bk{};
    LscvReduce red{};
    bk.nb = 2 * nh;
    int64_t off = 0;
    int max_rows = 1;
    for (int i = 0; i < nh; ++i) {
      const double* H = Hs + (size_t)(h0 + i) * d * d;
      for (int h = 0; h < 2; ++h) {
        double A[9], Ainv[9], detA;
        int64_t L[KDE_MAX_D];
        for (int e = 0; e < d * d; ++e) A[e] = (h ? 2.0 : 1.0) * H[e];
        kde_status st2 = kde::matrix_support(plan, A, Ainv, &detA, L);
        if (st2 != KDE_OK) return st2;
        const int b = 2 * i + h;
        st2 = kgen_for<T>(I, A, detA, L, plan->layout_mode == KDE_LAYOUT_WAND, &bk.gen[b]);
        if (st2 != KDE_OK) return st2;
        bk.rows[b] = (d == 1) ? 1 : (int)(2 * L[0] + 1);
        bk.off[b] = off;
        off += (int64_t)bk.rows[b] * I.Q;
        max_rows = std::max(max_rows, bk.rows[b]);
        if (h == 0) red.K0[i] = std::pow(6.283185307179586476925287, -0.5 * d) / std::sqrt(detA);
      }
    }
    const int dl = d - 1;
    RowsParams<T> rp{};
    rp.Q = (int)I.Q;
    rp.lp = line_plan(I, dl);
    rp.tw = twiddles<T>(plan, dl);
    if (d == 1)
      rp.out_real = (T*)T1;
    else
      rp.out = T1;
    {
      const int P = rp.lp.N;
      const int64_t pairs = (max_rows + 1) / 2;
      const LineShape sh = line_shape<T>(pairs * bk.nb, P, 1);
      rp.tpl = sh.tpl;
      auto* fn = kde_rows_kgen_batch_kernel<T>;
      cudaError_t e = allow_smem(fn);
      if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
      LaunchScope ls("kde_rows_kgen_batch_kernel", st);
      dim3 grid((unsigned)((pairs + sh.lpb - 1) / sh.lpb), (unsigned)bk.nb);
      fn<<<grid, sh.tpl * sh.lpb, line_smem<T>(P, sh.lpb), st>>>(bk, rp);
      if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_rows_kgen_batch_kernel");
    }
    int nparts;
    if (d == 1) {
      nparts = 1;
      LaunchScope ls("kde_dot1d_kernel", st);
      kde_dot1d_kernel<T><<<bk.nb, 256, 0, st>>>(bk.nb, (const T*)T1, (int)I.Q, (const T*)Wsp, partial);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return cuda_fail(e, "kde_dot1d_kernel");
    } else {
      ColsParams<T> cp{};
      cp.in = T1;
      cp.S = S;
      cp.lp = line_plan(I, 0);
      cp.tw = twiddles<T>(plan, 0);
      cp.W = (const T*)Wsp;
      cp.partial = partial;
      const int P = cp.lp.N;
      cudaError_t e;
      if (simd_cols<T>(plan->cols_variant, S, P)) {
        auto* fn = kde_cols_kgen_dot_kernel<T, true>;
        if ((e = allow_smem(fn)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
        nparts = (int)((S + 2 * kSimdW - 1) / (2 * kSimdW));
        LaunchScope ls("kde_cols_kgen_dot_kernel", st);
        fn<<<dim3((unsigned)nparts, (unsigned)bk.nb), 256,
             (size_t)(1 + 2 * kSimdW) * P * sizeof(V), st>>>(bk, cp);
      } else {
        const LineShape sh = line_shape<T>((S + 1) / 2 * bk.nb, P, 2);
        cp.tpl = sh.tpl;
        const int Wc = 2 * sh.lpb;
        auto* fn = kde_cols_kgen_dot_kernel<T, false>;
        if ((e = allow_smem(fn)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
        nparts = (int)((S + Wc - 1) / Wc);
        LaunchScope ls("kde_cols_kgen_dot_kernel", st);
        fn<<<dim3((unsigned)nparts, (unsigned)bk.nb), sh.tpl * sh.lpb, line_smem<T>(P, sh.lpb), st>>>(bk, cp);
      }
      if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_cols_kgen_dot_kernel");
    }
    red.nb = bk.nb;
    red.nparts = nparts;
    red.scale = 1.0 / prodP;
    red.n = (double)n;
    {
      LaunchScope ls("kde_lscv_reduce_kernel", st);
      kde_lscv_reduce_kernel<<<nh, 32, 0, st>>>(red, partial, S_out ? S_out + 2 * h0 : nullptr,
                                                lscv_out + h0);
      cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return cuda_fail(e, "kde_lscv_reduce_kernel");
    }
  }
  return KDE_OK;
}

// ---------------------------------------------------------------------------
// LSCV from the counts' autocorrelation (d = 2): R = F^{-1}|F(c)|^2 once per
// grid, then S(A) = sum over the support of K_A(delta o l) R(l) for every
// candidate -- no transform per candidate.
// ---------------------------------------------------------------------------
// Workspace: the autocorrelation's spectra, or (lag sums) the uploaded
// kernel parameters, K_H(0) and the FP64 partials of one chunk.
// At most this many work units per chunk: a unit holds kAcRows rows or more
// (the last of a matrix fewer), and L_0 < P_0 - M_0 + 1 for every matrix.
size_t ac_units_max(const kde_plan_info& I) {
  return (size_t)2 * kAcChunk * (size_t)((I.P[0] + kAcRows - 1) / kAcRows + 1);
}
// Uploaded per chunk: 2 nh AcGen, nh x {K_H(0), n, 1/n^2, 2/(n (n-1))}, then
// the work units and the blocks' (first unit, count).
size_t ac_upload_bytes(const kde_plan_info& I) {
  return ((size_t)2 * kAcChunk * sizeof(AcGen<double>) + (size_t)4 * kAcChunk * sizeof(double) +
          2 * ac_units_max(I) * sizeof(int2) + 255) & ~(size_t)255;
}

size_t ac_workspace(const kde_plan_info& I) {
  const size_t cb = (I.precision == KDE_F32) ? 8 : 16;
  const size_t spec = ((size_t)(I.M[0] + I.P[0]) * I.Q * cb + 255) & ~(size_t)255;
  return std::max(spec, ac_upload_bytes(I) + ac_units_max(I) * sizeof(double));
}

template <typename T>
kde_status autocorr_impl(kde_plan_s* plan, const int64_t* counts, void* Rout, void* ws,
                         cudaStream_t st, int64_t nsets = 1, void* ws_B = nullptr) {
  using V = typename Cplx<T>::type;
  const kde_plan_info& I = plan->info;
  // nsets grids one after another: counts [nsets][M_0][M_1], R [nsets][P_0][P_1]
  V* A = (V*)ws;                                       // [nsets][M_0][Q] half spectra of the rows
  V* B = ws_B ? (V*)ws_B : A + nsets * I.M[0] * I.Q;   // [nsets][P_0][Q] after the axis-0 pass
  if constexpr (std::is_same<T, float>::value) {
    if (I.engine == KDE_ENGINE_TWO_PHASE && !plan->dft_tc)
      return fx_autocorr(plan, reinterpret_cast<const long long*>(counts), (float*)Rout, A, B,
                         nsets, st);
  }
  RowsParams<T> rp{};
  rp.nrows = nsets * I.M[0];
  rp.Min = (int)I.M[1];
  rp.in_stride = I.M[1];
  rp.Q = (int)I.Q;
  rp.out = A;
  rp.lp = line_plan(I, 1);
  rp.tw = twiddles<T>(plan, 1);
  kde_status s = counts_rows<T>(plan, reinterpret_cast<const long long*>(counts), nsets * I.M[0],
                                rp, st);
  if (s != KDE_OK) return s;
  ColsParams<T> cp{};
  cp.in = A;
  cp.out = B;
  cp.S = I.Q;
  cp.Nin = (int)I.M[0];
  cp.Nout = (int)I.P[0];
  cp.Lw = -1;
  cp.lp = line_plan(I, 0);
  cp.tw = twiddles<T>(plan, 0);
  // counts are in units of 2^-32; the inverse transforms are unnormalised
  cp.s_pre = (T)2.3283064365386963e-10;
  cp.s_post = (T)(1.0 / ((double)I.P[0] * (double)I.P[1]));
  s = launch_cols<T>(KDE_COLS(kde_cols_auto_kernel), cp, nsets, plan->cols_variant, st,
                     "kde_cols_auto_kernel");
  if (s != KDE_OK) return s;
  C2RParams<T> cr{};
  cr.in = B;
  cr.out = (T*)Rout;
  cr.nrows = nsets * I.P[0];
  cr.Mout = (int)I.P[1];
  cr.Q = (int)I.Q;
  cr.lp = line_plan(I, 1);
  cr.tw = twiddles<T>(plan, 1);
  return launch_rows<T>(kde_rows_c2r_kernel<T>, "kde_rows_c2r_kernel", nsets * I.P[0], cr, st);
}

NTerms n_terms(double n) { return NTerms{{n, 1.0 / (n * n), 2.0 / (n * (n - 1.0))}}; }

// The matrices by dataset (already grouped), falling L_1, then falling L_0.
template <typename T>
std::vector<int> ac_order(const std::vector<AcGen<T>>& gens) {
  static_assert(KDE_MAX_P <= 4096, "supports fit in 12 bits");
  std::vector<int64_t> key(gens.size());
  for (size_t i = 0; i < gens.size(); ++i)
    key[i] = (int64_t)(4095 - gens[i].L1) << 44 | (int64_t)(4095 - gens[i].L0) << 32 | (int64_t)i;
  for (size_t i = 0, j = 0; i < key.size(); i = j) {
    for (j = i; j < key.size() && gens[j].set == gens[i].set;) ++j;
    std::sort(key.begin() + i, key.begin() + j);
  }
  std::vector<int> order(gens.size());
  for (size_t i = 0; i < key.size(); ++i) order[i] = (int)(key[i] & 0xFFFFFFFF);
  return order;
}

// Work units and blocks of a chunk, and its largest supports.
struct AcShape {
  int nunits, nblocks, L0, L1;
};

// Host side of one chunk of lag-sum candidates: candidates c = c0 ..
// c0 + nh - 1 of set c / nH, bandwidth Hs[c], sample count ns[c / nH] (ns may
// be NULL: n is then given at launch).  Fills `up` with the device image
// AcGen[2 nh], {K0, n, 1/n^2, 2/(n (n-1))}[nh], work units (by dataset, first
// row and falling L_1), blocks; returns their shape and, with gens_out, the
// parameters.
template <typename T>
kde_status ac_build_chunk(kde_plan_s* plan, int64_t c0, int nh, int nH, const double* Hs,
                          const int64_t* ns, std::vector<unsigned char>& up, AcShape* shape,
                          std::vector<AcGen<T>>* gens_out = nullptr) {
  const kde_plan_info& I = plan->info;
  const int d = I.d;
  std::vector<AcGen<T>> gens(2 * nh, AcGen<T>{});
  std::vector<double> kn(4 * nh, 0.0);
  std::vector<int2> units;
  size_t nunits = 0;
  for (int i = 0; i < nh; ++i) {
    const int64_t c = c0 + i;
    const double* H = Hs + (size_t)c * d * d;
    for (int h = 0; h < 2; ++h) {
      double A[9], Ainv[9], detA;
      int64_t L[KDE_MAX_D];
      for (int e = 0; e < d * d; ++e) A[e] = (h ? 2.0 : 1.0) * H[e];
      kde_status st2 = kde::matrix_support(plan, A, Ainv, &detA, L);
      if (st2 != KDE_OK) return st2;
      KGen<T> kg;
      st2 = kgen_for<T>(I, A, detA, L, plan->layout_mode == KDE_LAYOUT_WAND, &kg);
      if (st2 != KDE_OK) return st2;
      double Dd[3], Bd[3];
      st2 = gauss_factor(I.d, A, I.delta, Dd, Bd);
      if (st2 != KDE_OK) return st2;
      const double log2e = 1.4426950408889634073599246810;  // 1 / ln 2
      AcGen<T>& g = gens[2 * i + h];
      g.L0 = kg.L[0];
      g.L1 = kg.L[1];
      g.wand = kg.wand;
      g.set = (int)(c / nH);
      g.D0 = (T)(Dd[0] * log2e);
      g.D1 = (T)(Dd[1] * log2e);
      g.b_hi = kg.Bh[0];
      g.b_lo = kg.Bl[0];
      g.C = kg.C;
      g.u0 = (int)nunits;
      g.nu = g.L0 / kAcRows + 1;
      nunits += g.nu;
      if (h == 0) {
        kn[4 * i] = std::pow(6.283185307179586476925287, -0.5 * d) / std::sqrt(detA);
        const NTerms nt = ns ? n_terms((double)ns[c / nH]) : NTerms{};
        for (int k = 0; k < 3; ++k) kn[4 * i + 1 + k] = nt.v[k];
      }
    }
  }
  if (nunits > ac_units_max(I)) return fail(KDE_ERR_UNSUPPORTED, "lag-sum work units overflow");
  // matrices by dataset and falling L_1, then each dataset's rows in turn
  const std::vector<int> order = ac_order(gens);
  units.reserve(nunits);
  if (sizeof(T) == 8) {   // a block a unit: the longest rows first
    for (int m : order)
      for (int r = 0; r <= gens[m].L0; r += kAcRows) units.push_back(make_int2(m, r));
  }
  for (size_t i = 0, j = 0; sizeof(T) == 4 && i < order.size(); i = j) {
    int L0 = 0;
    for (j = i; j < order.size() && gens[order[j]].set == gens[order[i]].set; ++j)
      L0 = std::max(L0, gens[order[j]].L0);
    for (int r = 0; r <= L0; r += kAcRows)
      for (size_t k = i; k < j; ++k)
        if (r <= gens[order[k]].L0) units.push_back(make_int2(order[k], r));
  }
  *shape = AcShape{(int)units.size(), 0, 0, 0};
  for (const auto& g : gens) {
    shape->L0 = std::max(shape->L0, g.L0);
    shape->L1 = std::max(shape->L1, g.L1);
  }
  std::vector<int2> blocks;
  for (int u = 0; u < (int)units.size(); ++u) {
    const bool same = !blocks.empty() && blocks.back().y < kAcBlock &&
                      units[blocks.back().x].y == units[u].y &&
                      gens[units[blocks.back().x].x].set == gens[units[u].x].set;
    if (same) ++blocks.back().y;
    else blocks.push_back(make_int2(u, 1));
  }
  shape->nblocks = (int)blocks.size();
  const size_t gb = gens.size() * sizeof(AcGen<T>), kb = kn.size() * sizeof(double),
               ub = units.size() * sizeof(int2), bb = blocks.size() * sizeof(int2);
  up.resize(gb + kb + ub + bb);
  std::memcpy(up.data(), gens.data(), gb);
  std::memcpy(up.data() + gb, kn.data(), kb);
  std::memcpy(up.data() + gb + kb, units.data(), ub);
  std::memcpy(up.data() + gb + kb + ub, blocks.data(), bb);
  if (gens_out) *gens_out = std::move(gens);
  return KDE_OK;
}

// Pointers into a chunk's device image.
template <typename T>
struct AcImage {
  const AcGen<T>* gens;
  const double* kn;
  const int2 *units, *blocks;
  AcImage(const void* img, int nh, int nunits)
      : gens((const AcGen<T>*)img),
        kn((const double*)((const char*)img + 2 * (size_t)nh * sizeof(AcGen<T>))),
        units((const int2*)(kn + 4 * (size_t)nh)),
        blocks(units + nunits) {}
};

template <typename T>
kde_status ac_reduce(const AcImage<T>& im, int nh, int ns, const AcPart<T>* partial,
                     const NTerms* nk_set, const NTerms& nk_all, int64_t nH_all, double* S_out,
                     double* lscv_out, cudaStream_t st) {
  LaunchScope ls("kde_lscv_ac_reduce_kernel", st);
  const int64_t scores = (int64_t)nh * ns;
  auto launch = [&](auto fn, int per) {
    fn<<<(unsigned)((scores + per - 1) / per), 256, 0, st>>>(im.gens, im.kn, nk_set, nk_all, partial,
                                                             nh, ns, nH_all, S_out, lscv_out);
  };
  if (scores >= 256 * (int64_t)num_sms()) launch(kde_lscv_ac_reduce_kernel<T, true>, 256);
  else launch(kde_lscv_ac_reduce_kernel<T, false>, 32);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_lscv_ac_reduce_kernel");
}

// Units of a block: fewer where there are few in all, so that every SM has the
// blocks that it can hold, up to four (16 candidates of 230 lags 18.1 us with
// sixteen a block, 12.8 with a lag row a warp, 13.1 now; 512 x 512, 460 lags
// 29.1, 19.4, 18.3), but 24 groups at least.
int ac_block_units(int64_t nunits, int L1) {
  const int64_t fit = 220 * 1024 / ac_block_smem(L1, kAcBlock, ac_threads(L1));
  const int64_t blocks = std::min<int64_t>(4, std::max<int64_t>(1, fit)) * num_sms();
  const int64_t least = (23 + ac_unit_groups(L1)) / ac_unit_groups(L1);
  int sub = 1;   // parts of a block are alike
  while (sub < kAcBlock && (sub < least || 2 * sub <= nunits / blocks)) sub *= 2;
  return sub;
}

// One chunk whose image (ac_build_chunk) is at `img` against ns
// autocorrelations from R on, one by one (n terms as the reduction takes
// them).  sums: nunits ns of AcPart.
template <typename T>
kde_status ac_launch_chunk(const kde_plan_info& I, const void* img, int nh, const AcShape& sh, const T* R,
                           int ns, void* sums, const NTerms* nk_set, const NTerms& nk_all,
                           int64_t nH_all, double* S_out, double* lscv_out, cudaStream_t st) {
  const AcImage<T> im(img, nh, sh.nunits);
  AcPart<T>* partial = (AcPart<T>*)sums;
  static_assert(sizeof(AcPart<T>) == sizeof(double), "the workspaces count 8 bytes a unit");
  cudaError_t e;
  const int64_t per = I.P[0] * I.P[1];
  if constexpr (std::is_same<T, double>::value) {
    LaunchScope ls("kde_lscv_ac64_kernel", st);
    kde_lscv_ac64_kernel<<<dim3((unsigned)sh.nunits, (unsigned)ns), 256, 0, st>>>(
        im.gens, im.units, R, (int)I.P[1], per, partial);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_lscv_ac64_kernel");
  } else {
    const int threads = ac_threads(sh.L1), sub = ac_block_units((int64_t)sh.nunits * ns, sh.L1);
    const size_t smem = ac_block_smem(sh.L1, sub, threads);
    const unsigned grid = (unsigned)sh.nblocks * (unsigned)((kAcBlock + sub - 1) / sub);
    if ((e = allow_smem(kde_lscv_ac_kernel)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    LaunchScope ls("kde_lscv_ac_kernel", st);
    kde_lscv_ac_kernel<<<dim3(grid, (unsigned)ns), threads, smem, st>>>(
        im.gens, im.units, im.blocks, R, (int)I.P[1], per, sub,
        ac_turn(sh.L1, sub, threads), partial);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_lscv_ac_kernel");
  }
  return ac_reduce<T>(im, nh, ns, partial, nk_set, nk_all, nH_all, S_out, lscv_out, st);
}

// Candidates c = 0 .. nsets nH - 1 of set c / nH, bandwidth Hs[c], n[c / nH]:
// per chunk, the parameters are built on the host, copied into the
// workspace and launched.
template <typename T>
kde_status lscv_ac_impl(kde_plan_s* plan, int nsets, const int64_t* ns, int nH, const double* Hs,
                        const void* R, double* S_out, double* lscv_out, void* ws,
                        cudaStream_t st) {
  const kde_plan_info& I = plan->info;
  const int64_t total = (int64_t)nsets * nH;
  double* partial = (double*)((char*)ws + ac_upload_bytes(I));
  std::vector<unsigned char> up;
  for (int64_t h0 = 0; h0 < total; h0 += kAcChunk) {
    const int nh = (int)std::min<int64_t>(kAcChunk, total - h0);
    AcShape sh{};
    kde_status s = ac_build_chunk<T>(plan, h0, nh, nH, Hs, ns, up, &sh);
    if (s != KDE_OK) return s;
    if ((s = upload_async(ws, up.data(), up.size(), st)) != KDE_OK) return s;
    s = ac_launch_chunk<T>(I, ws, nh, sh, (const T*)R, 1, partial, nullptr, NTerms{}, 0,
                           S_out ? S_out + 2 * h0 : nullptr, lscv_out + h0, st);
    if (s != KDE_OK) return s;
  }
  return KDE_OK;
}

kde_status check_ws(const kde_plan_s* plan, void* ws, size_t bytes) {
  if (plan->info.workspace_bytes == 0) return KDE_OK;
  if (!ws) return fail(KDE_ERR_WORKSPACE, "workspace is NULL");
  if (bytes < plan->info.workspace_bytes) return fail(KDE_ERR_WORKSPACE, "workspace too small");
  if (((uintptr_t)ws & 15) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 16-byte aligned");
  return KDE_OK;
}

kde_status check_device(const kde_plan_s* plan) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev != plan->device) return fail(KDE_ERR_INVALID_ARG, "plan was made on another device");
  return KDE_OK;
}

}  // namespace
}  // namespace kde

using namespace kde;

extern "C" kde_status kde_kernel_grid(kde_plan plan, int64_t n, void* Kspec, void* workspace,
                                      size_t workspace_bytes, kde_stream_t stream) {
  if (!plan || !Kspec) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (n < 1) return fail(KDE_ERR_INVALID_ARG, "n must be >= 1 (the 1/n of Eq. 2)");
  kde_status s = check_ws(plan, workspace, workspace_bytes);
  if (s != KDE_OK) return s;
  if ((s = check_device(plan)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32) return kernel_grid_impl<float>(plan, n, Kspec, workspace, st);
  return kernel_grid_impl<double>(plan, n, Kspec, workspace, st);
}

extern "C" kde_status kde_fft_eval(kde_plan plan, const int64_t* counts, const void* Kspec,
                                   void* density, void* workspace, size_t workspace_bytes,
                                   kde_stream_t stream) {
  if (!plan || !counts || !Kspec || !density) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  kde_status s = check_ws(plan, workspace, workspace_bytes);
  if (s != KDE_OK) return s;
  if ((s = check_device(plan)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32)
    return fft_eval_impl<float>(plan, counts, Kspec, density, workspace, st);
  return fft_eval_impl<double>(plan, counts, Kspec, density, workspace, st);
}

// kde_fft_eval, then the counts set to zero: inside the second pass of the
// two-phase engine (the first pass is the only reader of the counts), else
// by one more operation after the evaluation.
extern "C" kde_status kde_fft_eval_consume(kde_plan plan, int64_t* counts, const void* Kspec,
                                           void* density, void* workspace, size_t workspace_bytes,
                                           kde_stream_t stream) {
  if (!plan || !counts || !Kspec || !density) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  kde_status s = check_ws(plan, workspace, workspace_bytes);
  if (s != KDE_OK) return s;
  if ((s = check_device(plan)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  const kde_plan_info& I = plan->info;
  if (I.precision == KDE_F32 && I.engine == KDE_ENGINE_TWO_PHASE)
    return kde::fx_fft_eval(plan, reinterpret_cast<const long long*>(counts), (const float*)Kspec,
                            (float*)density, workspace, st,
                            reinterpret_cast<unsigned long long*>(counts));
  s = I.precision == KDE_F32 ? fft_eval_impl<float>(plan, counts, Kspec, density, workspace, st)
                             : fft_eval_impl<double>(plan, counts, Kspec, density, workspace, st);
  if (s != KDE_OK) return s;
  int64_t cells = 1;
  for (int k = 0; k < I.d; ++k) cells *= I.M[k];
  cudaError_t e = cudaMemsetAsync(counts, 0, (size_t)cells * sizeof(int64_t), st);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaMemsetAsync(counts)");
}

// ---------------------------------------------------------------------------
// Densities for many bandwidths on one grid (Eq. 10: C = F(c) computed once,
// K computed and applied per bandwidth).  KDE_F32 2-D plans with the
// two-phase engine; bandwidths in chunks of kMultiChunk per launch.
// ---------------------------------------------------------------------------
namespace kde {
namespace {

constexpr int kMultiChunk = 64;
// Bandwidths whose parameters go up in one copy: a copy between every two
// chunks cost 8 us of idle device each.
constexpr int kMultiUpload = 1024;

struct MultiLayout {
  int Lmax0;
  size_t off_A, off_C, off_gens, off_t1, off_S, total;
};

kde_status multi_layout(const kde_plan_s* plan, MultiLayout* m) {
  const kde_plan_info& I = plan->info;
  if (I.d != 2 || I.precision != KDE_F32 || I.engine != KDE_ENGINE_TWO_PHASE ||
      I.P[0] > fxp::kMaxNamedP || I.P[1] > fxp::kMaxNamedP)
    return fail(KDE_ERR_UNSUPPORTED,
                "batched densities need a KDE_F32 2-D plan with the two-phase engine");
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  // every accepted bandwidth has M_0 + L_0 <= P_0
  m->Lmax0 = (int)(I.P[0] - I.M[0]);
  const size_t Q = (size_t)I.Q, M0 = (size_t)I.M[0], P0 = (size_t)I.P[0];
  m->off_A = 0;
  m->off_C = up(M0 * Q * 8);
  m->off_gens = m->off_C + up(P0 * Q * 8);
  m->off_t1 = m->off_gens + up(kMultiUpload * (sizeof(KGen<float>) + sizeof(int)));
  m->off_S = m->off_t1 + up((size_t)kMultiChunk * (m->Lmax0 + 1) * Q * 8);
  m->total = m->off_S + up((size_t)kMultiChunk * M0 * Q * 8);
  return KDE_OK;
}

}  // namespace
}  // namespace kde

extern "C" kde_status kde_fft_eval_multi_workspace_bytes(kde_plan plan, size_t* bytes) {
  if (!plan || !bytes) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  MultiLayout m;
  kde_status s = multi_layout(plan, &m);
  if (s != KDE_OK) return s;
  *bytes = m.total;
  return KDE_OK;
}

extern "C" kde_status kde_fft_eval_multi(kde_plan plan, int64_t n, int nH, const double* H,
                                         const int64_t* counts, void* density, void* workspace,
                                         size_t workspace_bytes, kde_stream_t stream) {
  if (!plan || (nH > 0 && (!H || !counts || !density)))
    return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (nH < 0 || n < 1) return fail(KDE_ERR_INVALID_ARG, "need nH >= 0 and n >= 1");
  MultiLayout m;
  kde_status s = multi_layout(plan, &m);
  if (s != KDE_OK) return s;
  if (nH == 0) return KDE_OK;
  if (!workspace || workspace_bytes < m.total)
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_fft_eval_multi_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  if ((s = check_device(plan)) != KDE_OK) return s;
  const kde_plan_info& I = plan->info;
  // every bandwidth's factors and kernel-grid parameters, before any launch
  std::vector<KGen<float>> gens((size_t)nH);
  std::vector<int> L0((size_t)nH);
  double prodP = (double)I.P[0] * (double)I.P[1];
  for (int h = 0; h < nH; ++h) {
    double Ainv[9], det;
    int64_t L[KDE_MAX_D];
    if ((s = matrix_support(plan, H + 4 * h, Ainv, &det, L)) != KDE_OK) return s;
    if ((s = kgen_for<float>(I, H + 4 * h, det, L, plan->layout_mode == KDE_LAYOUT_WAND,
                             &gens[h])) != KDE_OK)
      return s;
    gens[h].C = (float)(1.0 / (6.283185307179586476925287 * std::sqrt(det)) /
                        ((double)n * 4294967296.0 * prodP));
    L0[h] = (int)L[0];
  }
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  float2* C = (float2*)(ws + m.off_C);
  if ((s = fx_count_spectrum2(plan, reinterpret_cast<const long long*>(counts),
                              (float2*)(ws + m.off_A), C, st)) != KDE_OK)
    return s;
  const size_t cells = (size_t)I.M[0] * I.M[1];
  std::vector<unsigned char> up;
  for (int u0 = 0; u0 < nH; u0 += kMultiUpload) {
    const int nu = std::min(kMultiUpload, nH - u0);
    // parameters, then supports: stream-ordered after the kernels of the last ones
    const size_t gb = (size_t)nu * sizeof(KGen<float>), lb = (size_t)nu * sizeof(int);
    up.resize(gb + lb);
    std::memcpy(up.data(), gens.data() + u0, gb);
    std::memcpy(up.data() + gb, L0.data() + u0, lb);
    if ((s = upload_async(ws + m.off_gens, up.data(), up.size(), st)) != KDE_OK) return s;
    const auto* gens_dev = (const KGen<float>*)(ws + m.off_gens);
    const int* L0_dev = (const int*)(ws + m.off_gens + gb);
    for (int h0 = 0; h0 < nu; h0 += kMultiChunk) {
      s = fx_eval_batch2(plan, C, std::min(kMultiChunk, nu - h0), gens_dev + h0, L0_dev + h0, m.Lmax0,
                         (float2*)(ws + m.off_t1), (float2*)(ws + m.off_S),
                         (float*)density + (size_t)(u0 + h0) * cells, st);
      if (s != KDE_OK) return s;
    }
  }
  return KDE_OK;
}

// ---------------------------------------------------------------------------
// kde_fft_eval_noalloc: kde_fft_eval with its scratch in a fixed device array
// instead of a caller-provided workspace, for callers that cannot allocate
// device memory at the point of the call (for example code running inside a
// framework that owns every allocation, or a real-time loop that must not
// enter the allocator).  Its size is fixed at build time and the array lives
// on every device that loads this library until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr size_t kNoAllocScratchBytes = KDE_NOALLOC_SCRATCH_BYTES;
static_assert(kNoAllocScratchBytes % 256 == 0, "the scratch array is a whole number of 256-byte blocks");
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_ptr[kMaxDevices] = {};

// Device address of g_noalloc_scratch on the current device.  In host code
// the symbol's name is only a host-side handle, so the address is looked up
// once per device with that device current and cached.
kde_status noalloc_scratch(int dev, void** out) {
  if (dev < 0 || dev >= kMaxDevices) return fail(KDE_ERR_UNSUPPORTED, "device ordinal too large");
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    g_noalloc_ptr[dev] = p;
  }
  *out = g_noalloc_ptr[dev];
  return KDE_OK;
}

}  // namespace

extern "C" size_t kde_noalloc_scratch_bytes(void) { return kNoAllocScratchBytes; }

extern "C" kde_status kde_fft_eval_noalloc(kde_plan plan, const int64_t* counts, const void* Kspec,
                                           void* density, kde_stream_t stream) {
  if (!plan || !counts || !Kspec || !density) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.workspace_bytes > kNoAllocScratchBytes)
    return fail(KDE_ERR_WORKSPACE,
                "kde_fft_eval_noalloc: the plan needs " + std::to_string(plan->info.workspace_bytes) +
                    " bytes of scratch, above the fixed " + std::to_string(kNoAllocScratchBytes) +
                    "; use kde_fft_eval with a workspace");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  void* scratch = nullptr;
  if ((s = noalloc_scratch(plan->device, &scratch)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32)
    return fft_eval_impl<float>(plan, counts, Kspec, density, scratch, st);
  return fft_eval_impl<double>(plan, counts, Kspec, density, scratch, st);
}

// ---------------------------------------------------------------------------
// Count spectrum and LSCV entry points.
// ---------------------------------------------------------------------------
extern "C" kde_status kde_power_spectrum(kde_plan plan, const int64_t* counts, void* W,
                                         void* workspace, size_t workspace_bytes,
                                         kde_stream_t stream) {
  if (!plan || !counts || !W) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  kde_status s = check_ws(plan, workspace, workspace_bytes);
  if (s != KDE_OK) return s;
  if ((s = check_device(plan)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32) return power_spectrum_impl<float>(plan, counts, W, workspace, st);
  return power_spectrum_impl<double>(plan, counts, W, workspace, st);
}

extern "C" kde_status kde_lscv_workspace_bytes(kde_plan plan, size_t* bytes) {
  if (!plan || !bytes) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.d == 3) return fail(KDE_ERR_UNSUPPORTED, "LSCV batches support d = 1, 2");
  *bytes = lscv_workspace(plan->info);
  return KDE_OK;
}

extern "C" kde_status kde_lscv(kde_plan plan, int64_t n, int nH, const double* H, const void* W,
                               double* pair_sums, double* lscv, void* workspace,
                               size_t workspace_bytes, kde_stream_t stream) {
  if (!plan || !H || !W || !lscv) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.d == 3) return fail(KDE_ERR_UNSUPPORTED, "LSCV batches support d = 1, 2");
  if (n < 2) return fail(KDE_ERR_INVALID_ARG, "LSCV needs n >= 2");
  if (nH < 0) return fail(KDE_ERR_INVALID_ARG, "nH < 0");
  if (nH == 0) return KDE_OK;
  if (!workspace || workspace_bytes < lscv_workspace(plan->info))
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32)
    return lscv_impl<float>(plan, n, nH, H, W, pair_sums, lscv, workspace, st);
  return lscv_impl<double>(plan, n, nH, H, W, pair_sums, lscv, workspace, st);
}

extern "C" kde_status kde_lscv_autocorr_workspace_bytes(kde_plan plan, size_t* bytes) {
  if (!plan || !bytes) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.d != 2) return fail(KDE_ERR_UNSUPPORTED, "autocorrelation LSCV supports d = 2");
  *bytes = ac_workspace(plan->info);
  return KDE_OK;
}

extern "C" kde_status kde_autocorrelation(kde_plan plan, const int64_t* counts, void* R,
                                          void* workspace, size_t workspace_bytes,
                                          kde_stream_t stream) {
  if (!plan || !counts || !R) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.d != 2) return fail(KDE_ERR_UNSUPPORTED, "autocorrelation LSCV supports d = 2");
  if (!workspace || workspace_bytes < ac_workspace(plan->info))
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_autocorr_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32) return autocorr_impl<float>(plan, counts, R, workspace, st);
  return autocorr_impl<double>(plan, counts, R, workspace, st);
}

// Workspace of kde_prepare2_batch: device copy of the offsets, the
// standardised samples, and the autocorrelation's two intermediates for
// every grid.
struct PrepLayout {
  size_t off_offsets, off_Z, off_A, off_B, total;
};

static PrepLayout prep_layout(const kde_plan_info& I, int64_t nsets, int64_t n_total) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t cb = I.precision == KDE_F32 ? 8 : 16;  // complex element
  PrepLayout L{};
  L.off_offsets = 0;
  L.off_Z = up((size_t)(nsets + 1) * sizeof(int64_t));
  L.off_A = L.off_Z + up((size_t)n_total * 2 * sizeof(float));
  L.off_B = L.off_A + up((size_t)nsets * I.M[0] * I.Q * cb);
  L.total = L.off_B + up((size_t)nsets * I.P[0] * I.Q * cb);
  return L;
}

static kde_status prep_check(kde_plan plan, int nsets) {
  if (!plan) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  const kde_plan_info& I = plan->info;
  if (I.d != 2) return fail(KDE_ERR_UNSUPPORTED, "batched preparation supports d = 2");
  if (I.M[0] != I.M[1] || I.M[0] < 32 || I.M[0] % 32)
    return fail(KDE_ERR_UNSUPPORTED, "batched preparation needs an M x M grid, M a multiple of 32");
  if (nsets < 0 || nsets > 65535) return fail(KDE_ERR_INVALID_ARG, "need 0 <= nsets <= 65535");
  return KDE_OK;
}

extern "C" kde_status kde_prepare2_batch_workspace_bytes(kde_plan plan, int nsets, int64_t n_total,
                                                         size_t* bytes) {
  kde_status s = prep_check(plan, nsets);
  if (s != KDE_OK) return s;
  if (!bytes || n_total < 0) return fail(KDE_ERR_INVALID_ARG, "bad argument");
  *bytes = prep_layout(plan->info, nsets, n_total).total;
  return KDE_OK;
}

extern "C" kde_status kde_prepare2_batch(kde_plan plan, int nsets, const float* X,
                                         const int64_t* offsets, int64_t* counts, double* moments,
                                         float* feat, void* R, void* workspace,
                                         size_t workspace_bytes, kde_stream_t stream) {
  kde_status s = prep_check(plan, nsets);
  if (s != KDE_OK) return s;
  if (nsets == 0) return KDE_OK;
  if (!X || !offsets || !counts || !moments || !feat || !R)
    return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (offsets[0] != 0) return fail(KDE_ERR_INVALID_ARG, "offsets[0] must be 0");
  int64_t n_max = 0;
  for (int b = 0; b < nsets; ++b) {
    const int64_t n = offsets[b + 1] - offsets[b];
    if (n < 2) return fail(KDE_ERR_INVALID_ARG, "every dataset needs at least 2 samples");
    if (n >= (int64_t(1) << 31)) return fail(KDE_ERR_INVALID_ARG, "a dataset has 2^31 samples or more");
    n_max = std::max(n_max, n);
  }
  const int64_t n_total = offsets[nsets];
  const kde_plan_info& I = plan->info;
  const PrepLayout L = prep_layout(I, nsets, n_total);
  if (!workspace || workspace_bytes < L.total)
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_prepare2_batch_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  if ((s = check_device(plan)) != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  int64_t* off_dev = (int64_t*)(ws + L.off_offsets);
  float* Z = (float*)(ws + L.off_Z);
  if ((s = upload_async(off_dev, offsets, (size_t)(nsets + 1) * sizeof(int64_t), st)) != KDE_OK)
    return s;
  if ((s = standardize2_sets(X, off_dev, nsets, Z, moments, st)) != KDE_OK) return s;
  if ((s = bin_sets_f32(Z, off_dev, nsets, n_max, 2, plan->lo, plan->hi, I.M, counts, st)) != KDE_OK)
    return s;
  if ((s = features2_sets(counts, (int)I.M[0], nsets, off_dev, moments, feat, st)) != KDE_OK) return s;
  if (I.precision == KDE_F32)
    return autocorr_impl<float>(plan, counts, R, ws + L.off_A, st, nsets, ws + L.off_B);
  return autocorr_impl<double>(plan, counts, R, ws + L.off_A, st, nsets, ws + L.off_B);
}

static kde_status lscv_ac_entry(kde_plan plan, int nsets, const int64_t* n, int nH,
                                const double* H, const void* R, double* pair_sums, double* lscv,
                                void* workspace, size_t workspace_bytes, kde_stream_t stream) {
  if (!plan || !n || !H || !R || !lscv) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (plan->info.d != 2) return fail(KDE_ERR_UNSUPPORTED, "autocorrelation LSCV supports d = 2");
  if (nsets < 0 || nH < 0) return fail(KDE_ERR_INVALID_ARG, "nsets < 0 or nH < 0");
  for (int s = 0; s < nsets; ++s)
    if (n[s] < 2) return fail(KDE_ERR_INVALID_ARG, "LSCV needs n >= 2");
  if (nsets == 0 || nH == 0) return KDE_OK;
  if (!workspace || workspace_bytes < ac_workspace(plan->info))
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_autocorr_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  if (plan->info.precision == KDE_F32)
    return lscv_ac_impl<float>(plan, nsets, n, nH, H, R, pair_sums, lscv, workspace, st);
  return lscv_ac_impl<double>(plan, nsets, n, nH, H, R, pair_sums, lscv, workspace, st);
}

extern "C" kde_status kde_lscv_autocorr(kde_plan plan, int64_t n, int nH, const double* H,
                                        const void* R, double* pair_sums, double* lscv,
                                        void* workspace, size_t workspace_bytes,
                                        kde_stream_t stream) {
  return lscv_ac_entry(plan, 1, &n, nH, H, R, pair_sums, lscv, workspace, workspace_bytes, stream);
}

extern "C" kde_status kde_lscv_autocorr_batch(kde_plan plan, int nsets, const int64_t* n, int nH,
                                              const double* H, const void* R, double* pair_sums,
                                              double* lscv, void* workspace,
                                              size_t workspace_bytes, kde_stream_t stream) {
  return lscv_ac_entry(plan, nsets, n, nH, H, R, pair_sums, lscv, workspace, workspace_bytes, stream);
}

// A candidate set prepared once: its lag-sum parameters, work units and (FP32)
// groups live on the device, so scoring it against other datasets'
// autocorrelations is two launches per chunk of 1024 candidates
// with no host work.
struct kde_lscv_cands_s {
  kde_plan_s* plan;
  int nH;
  struct Chunk {
    void* dev;         // image (ac_build_chunk), then groups and items
    int64_t c0;
    int nh;
    AcShape sh;
    AcGroup* groups;   // null: scored one by one (FP64)
    int3* items;
    int nitems;
  };
  std::vector<Chunk> chunks;
};

static void cands_free(kde_lscv_cands_s* c) {
  for (auto& ch : c->chunks) cudaFree(ch.dev);
  delete c;
}

// Groups of up to kAcQuad matrices, and items of up to kAcWarps groups and a
// first row (the widest first).
template <typename T>
static void cands_group(const std::vector<AcGen<T>>& gens, std::vector<AcGroup>& groups,
                        std::vector<int3>& items) {
  const std::vector<int> order = ac_order(gens);
  for (size_t i = 0; i < order.size();) {
    AcGroup g{};
    g.L0 = gens[order[i]].L0;
    g.L1 = gens[order[i]].L1;
    for (int k = 0; k < kAcQuad; ++k) {
      const bool same = i < order.size() && gens[order[i]].L1 == g.L1 &&
                        ac_shift(0, gens[order[i]].L0, g.L1) == ac_shift(0, g.L0, g.L1);
      g.m[k] = same ? order[i++] : -1;
    }
    groups.push_back(g);
  }
  for (size_t i = 0; i < groups.size(); i += kAcWarps) {
    const int n = (int)std::min<size_t>(kAcWarps, groups.size() - i);
    int L0 = 0;
    for (int k = 0; k < n; ++k) L0 = std::max(L0, groups[i + k].L0);
    for (int r = 0; r <= L0; r += kAcRows) items.push_back(make_int3((int)i, n, r));
  }
}

template <typename T>
static kde_status cands_build(kde_lscv_cands_s* c, const double* H) {
  std::vector<unsigned char> up;
  std::vector<AcGen<T>> gens;
  for (int64_t h0 = 0; h0 < c->nH; h0 += kAcChunk) {
    const int nh = (int)std::min<int64_t>(kAcChunk, c->nH - h0);
    kde_lscv_cands_s::Chunk ch{};
    kde_status s = ac_build_chunk<T>(c->plan, h0, nh, c->nH, H, nullptr, up, &ch.sh, &gens);
    if (s != KDE_OK) return s;
    ch.c0 = h0;
    ch.nh = nh;
    std::vector<AcGroup> groups;
    std::vector<int3> items;
    const size_t at = (up.size() + 255) & ~(size_t)255;
    size_t at_items = at;
    if (sizeof(T) == 4) {
      cands_group(gens, groups, items);
      at_items = at + groups.size() * sizeof(AcGroup);
      up.resize(at_items + items.size() * sizeof(int3));
      std::memcpy(up.data() + at, groups.data(), groups.size() * sizeof(AcGroup));
      std::memcpy(up.data() + at_items, items.data(), items.size() * sizeof(int3));
      ch.nitems = (int)items.size();
    }
    cudaError_t e = cudaMalloc(&ch.dev, up.size());
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(candidate set)");
    if (ch.nitems) {
      ch.groups = (AcGroup*)((char*)ch.dev + at);
      ch.items = (int3*)((char*)ch.dev + at_items);
    }
    c->chunks.push_back(ch);
    e = cudaMemcpy(ch.dev, up.data(), up.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(candidate set)");
  }
  return KDE_OK;
}

extern "C" kde_status kde_lscv_cands_create(kde_plan plan, int nH, const double* H,
                                            kde_lscv_cands* out) {
  if (!plan || !H || !out) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  if (plan->info.d != 2) return fail(KDE_ERR_UNSUPPORTED, "autocorrelation LSCV supports d = 2");
  if (nH < 1) return fail(KDE_ERR_INVALID_ARG, "nH must be >= 1");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  auto* c = new kde_lscv_cands_s{plan, nH, {}};
  s = plan->info.precision == KDE_F32 ? cands_build<float>(c, H) : cands_build<double>(c, H);
  if (s != KDE_OK) {
    cands_free(c);
    return s;
  }
  *out = c;
  return KDE_OK;
}

extern "C" kde_status kde_lscv_cands_destroy(kde_lscv_cands cands) {
  if (!cands) return KDE_OK;
  cands_free(cands);
  return KDE_OK;
}

extern "C" kde_status kde_lscv_autocorr_cands(kde_lscv_cands cands, int64_t n, const void* R,
                                              double* pair_sums, double* lscv, void* workspace,
                                              size_t workspace_bytes, kde_stream_t stream) {
  if (!cands || !R || !lscv) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (n < 2) return fail(KDE_ERR_INVALID_ARG, "LSCV needs n >= 2");
  kde_plan_s* plan = cands->plan;
  if (!workspace || workspace_bytes < ac_workspace(plan->info))
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_autocorr_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  double* partial = (double*)((char*)workspace + ac_upload_bytes(plan->info));
  const NTerms nk = n_terms((double)n);
  for (const auto& ch : cands->chunks) {
    double* S = pair_sums ? pair_sums + 2 * ch.c0 : nullptr;
    s = plan->info.precision == KDE_F32
            ? ac_launch_chunk<float>(plan->info, ch.dev, ch.nh, ch.sh, (const float*)R, 1, partial,
                                     nullptr, nk, 0, S, lscv + ch.c0, st)
            : ac_launch_chunk<double>(plan->info, ch.dev, ch.nh, ch.sh, (const double*)R, 1,
                                      partial, nullptr, nk, 0, S, lscv + ch.c0, st);
    if (s != KDE_OK) return s;
  }
  return KDE_OK;
}

// Scratch of kde_lscv_autocorr_cands_batch: the datasets' n terms, then for
// a slab of datasets one FP64 partial per work unit of the largest chunk.
struct CandsBatch {
  int slab;            // datasets per launch
  size_t off_part, total;
};

static CandsBatch cands_batch_layout(const kde_lscv_cands_s* c, int nsets) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  int units = 0;
  CandsBatch b{};
  for (const auto& ch : c->chunks) units = std::max(units, ch.sh.nunits);
  b.slab = std::min(nsets, kAcSlab);
  b.off_part = up((size_t)nsets * sizeof(NTerms));
  b.total = b.off_part + up((size_t)b.slab * units * sizeof(double));
  return b;
}

extern "C" kde_status kde_lscv_autocorr_cands_batch_workspace_bytes(kde_lscv_cands cands, int nsets,
                                                                    size_t* bytes) {
  if (!cands || !bytes) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (nsets < 0 || nsets > 65535) return fail(KDE_ERR_INVALID_ARG, "need 0 <= nsets <= 65535");
  *bytes = cands_batch_layout(cands, nsets).total;
  return KDE_OK;
}

// The batched sums of one chunk against ns autocorrelations from R on.
static kde_status ac_product_chunk(const kde_plan_info& I, const kde_lscv_cands_s::Chunk& ch,
                                   const float* R, int ns, AcPair* partial, const NTerms* nk_set,
                                   int64_t nH_all, double* S, double* lscv, cudaStream_t st) {
  const AcImage<float> im(ch.dev, ch.nh, ch.sh.nunits);
  cudaError_t e;
  {
    if ((e = allow_smem(kde_lscv_ac_sets_kernel)) != cudaSuccess)
      return cuda_fail(e, "cudaFuncSetAttribute");
    LaunchScope ls("kde_lscv_ac_sets_kernel", st);
    kde_lscv_ac_sets_kernel<<<dim3((unsigned)ch.nitems, (unsigned)((ns + kAcSets - 1) / kAcSets)),
                              32 * kAcWarps, kAcSetsSmem, st>>>(
        im.gens, ch.groups, ch.items, R, (int)I.P[1], (int64_t)I.P[0] * I.P[1], ns, partial);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_lscv_ac_sets_kernel");
  }
  return ac_reduce<float>(im, ch.nh, ns, partial, nk_set, NTerms{}, nH_all, S, lscv, st);
}

extern "C" kde_status kde_lscv_autocorr_cands_batch(kde_lscv_cands cands, int nsets,
                                                    const int64_t* n, const void* R,
                                                    double* pair_sums, double* lscv,
                                                    void* workspace, size_t workspace_bytes,
                                                    kde_stream_t stream) {
  if (!cands) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (nsets < 0 || nsets > 65535) return fail(KDE_ERR_INVALID_ARG, "need 0 <= nsets <= 65535");
  if (nsets == 0) return KDE_OK;
  if (!n || !R || !lscv) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  std::vector<NTerms> nd((size_t)nsets);
  for (int b = 0; b < nsets; ++b) {
    if (n[b] < 2) return fail(KDE_ERR_INVALID_ARG, "LSCV needs n >= 2");
    nd[b] = n_terms((double)n[b]);
  }
  const CandsBatch lay = cands_batch_layout(cands, nsets);
  if (!workspace || workspace_bytes < lay.total)
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_autocorr_cands_batch_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  kde_plan_s* plan = cands->plan;
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  const kde_plan_info& I = plan->info;
  cudaStream_t st = (cudaStream_t)stream;
  NTerms* nset = (NTerms*)workspace;
  void* partial = (char*)workspace + lay.off_part;
  if ((s = upload_async(nset, nd.data(), nd.size() * sizeof(NTerms), st)) != KDE_OK) return s;
  const int64_t per = I.P[0] * I.P[1], nH = cands->nH;
  for (int y = 0; y < nsets; y += lay.slab) {
    const int ns = std::min(lay.slab, nsets - y);
    for (const auto& ch : cands->chunks) {
      double* S = pair_sums ? pair_sums + 2 * (y * nH + ch.c0) : nullptr;
      double* out = lscv + y * nH + ch.c0;
      if (ch.groups && ac_product(ns, ch.sh.nunits, ch.nitems, ch.sh.L1, num_sms()))
        s = ac_product_chunk(I, ch, (const float*)R + y * per, ns, (AcPair*)partial, nset + y, nH, S, out, st);
      else if (I.precision == KDE_F32)
        s = ac_launch_chunk<float>(I, ch.dev, ch.nh, ch.sh, (const float*)R + y * per, ns, partial,
                                   nset + y, NTerms{}, nH, S, out, st);
      else
        s = ac_launch_chunk<double>(I, ch.dev, ch.nh, ch.sh, (const double*)R + y * per, ns,
                                    partial, nset + y, NTerms{}, nH, S, out, st);
      if (s != KDE_OK) return s;
    }
  }
  return KDE_OK;
}

// Workspace of kde_lscv_theta_select: the uploaded n, reference thetas and
// offsets; the candidates' parameters, K_H(0) and pair sums.
struct ThetaLayout {
  size_t off_up, off_gens, off_K0, off_S, off_cls, total;
  ThetaSplit split;
};

static ThetaLayout theta_layout(int64_t nsets, int64_t J) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const int64_t cands = nsets * (J + 1);
  ThetaLayout L{};
  L.off_up = 0;
  L.off_gens = up((size_t)(nsets + 3 * nsets + 3 * J) * sizeof(double));
  L.off_K0 = L.off_gens + up((size_t)2 * cands * sizeof(AcGen<float>));
  L.off_S = L.off_K0 + up((size_t)cands * sizeof(double));
  L.off_cls = L.off_S + up((size_t)2 * cands * sizeof(double));
  L.split = theta_split(nsets, J + 1, num_sms());
  L.total = L.off_cls + (L.split.nr > 1 ? up((size_t)2 * cands * kAcClasses * sizeof(AcPair)) : 0);
  return L;
}

extern "C" kde_status kde_lscv_theta_select_workspace_bytes(kde_plan plan, int nsets, int J,
                                                            size_t* bytes) {
  if (!plan || !bytes) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (nsets < 0 || J < 1 || (int64_t)nsets * 2 * (J + 1) >= (int64_t(1) << 31))
    return fail(KDE_ERR_INVALID_ARG, "need nsets >= 0, J >= 1 and fewer than 2^31 matrices");
  *bytes = theta_layout(nsets, J).total;
  return KDE_OK;
}

extern "C" kde_status kde_lscv_theta_select(kde_plan plan, int nsets, const int64_t* n,
                                            const float* theta, const double* box, int J,
                                            const double* offsets, const double* ref, const void* R,
                                            double* lscv, double* out, void* workspace,
                                            size_t workspace_bytes, kde_stream_t stream) {
  if (!plan) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  const kde_plan_info& I = plan->info;
  if (I.d != 2 || I.precision != KDE_F32)
    return fail(KDE_ERR_UNSUPPORTED, "device-built candidates need a KDE_F32 2-D plan");
  if (nsets < 0 || J < 1 || (int64_t)nsets * 2 * (J + 1) >= (int64_t(1) << 31))
    return fail(KDE_ERR_INVALID_ARG, "need nsets >= 0, J >= 1 and fewer than 2^31 matrices");
  if (nsets == 0) return KDE_OK;
  if (!n || !theta || !box || !offsets || !ref || !R || !out)
    return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  const ThetaLayout L = theta_layout(nsets, J);
  if (!workspace || workspace_bytes < L.total)
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than kde_lscv_theta_select_workspace_bytes");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  std::vector<double> up((size_t)(nsets + 3 * nsets + 3 * J));
  for (int s = 0; s < nsets; ++s) {
    if (n[s] < 2) return fail(KDE_ERR_INVALID_ARG, "LSCV needs n >= 2");
    up[s] = (double)n[s];
  }
  for (int i = 0; i < 3 * nsets; ++i) {
    if (!std::isfinite(ref[i])) return fail(KDE_ERR_INVALID_ARG, "non-finite reference theta");
    up[nsets + i] = ref[i];
  }
  for (int i = 0; i < 3 * J; ++i) {
    if (!std::isfinite(offsets[i])) return fail(KDE_ERR_INVALID_ARG, "non-finite offset");
    up[4 * (size_t)nsets + i] = offsets[i];
  }
  for (int k = 0; k < 6; ++k)
    if (!std::isfinite(box[k])) return fail(KDE_ERR_INVALID_ARG, "non-finite box");
  kde_status s = check_device(plan);
  if (s != KDE_OK) return s;
  cudaStream_t st = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  double* upd = (double*)(ws + L.off_up);
  if ((s = upload_async(upd, up.data(), up.size() * sizeof(double), st)) != KDE_OK) return s;
  cudaError_t e = cudaSuccess;
  ThetaArgs t{};
  t.nsets = nsets;
  t.J = J;
  t.theta = theta;
  t.n = upd;
  t.ref = upd + nsets;
  t.off = upd + 4 * (size_t)nsets;
  for (int k = 0; k < 3; ++k) {
    t.box_lo[k] = box[k];
    t.box_hi[k] = box[3 + k];
  }
  t.tau = plan->tau;
  for (int k = 0; k < 2; ++k) {
    t.delta[k] = I.delta[k];
    t.M[k] = (int)I.M[k];
    t.P[k] = (int)I.P[k];
  }
  t.wand = plan->layout_mode == KDE_LAYOUT_WAND;
  t.per_axis = plan->range_mode != KDE_RANGE_CORRECTED;
  t.gens = (AcGen<float>*)(ws + L.off_gens);
  t.K0 = (double*)(ws + L.off_K0);
  double* S = (double*)(ws + L.off_S);
  AcPair* cls = L.split.nr > 1 ? (AcPair*)(ws + L.off_cls) : nullptr;
  const int64_t nmat = (int64_t)nsets * 2 * (J + 1);
  {
    LaunchScope ls("kde_theta_gen_kernel", st);
    kde_theta_gen_kernel<<<(unsigned)((nmat + 31) / 32), 32, 0, st>>>(t);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_theta_gen_kernel");
  }
  {
    // a candidate's support that fits has L_1 <= P_1 - M_1, and never more than
    // M_1 - 1 (the padding alone can be far wider than any support)
    const int L1 = (int)std::min(I.P[1] - I.M[1], I.M[1] - 1);
    const ThetaSplit sp = L.split;
    const size_t smem = ac_block_smem(L1, 2 * sp.nc, kThetaThreads);
    if ((e = allow_smem(kde_lscv_theta_sums_kernel)) != cudaSuccess)
      return cuda_fail(e, "cudaFuncSetAttribute");
    LaunchScope ls("kde_lscv_theta_sums_kernel", st);
    kde_lscv_theta_sums_kernel<<<dim3((unsigned)((int64_t)nsets * ((J + sp.nc) / sp.nc)), (unsigned)sp.nr),
                                 kThetaThreads, smem, st>>>(
        t.gens, 2 * (J + 1), sp.nc, (const float*)R, (int)I.P[1], (int64_t)I.P[0] * I.P[1], L1,
        ac_turn(L1, 2 * sp.nc, kThetaThreads), nmat, cls, S);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_lscv_theta_sums_kernel");
  }
  {
    LaunchScope ls("kde_lscv_theta_pick_kernel", st);
    kde_lscv_theta_pick_kernel<<<nsets, 32, 0, st>>>(t, S, cls, nmat, lscv, out);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_lscv_theta_pick_kernel");
  }
  return KDE_OK;
}

// ---------------------------------------------------------------------------
// Ragged batches: many independent 2-D problems (own samples, grid, H) in one
// set of launches.  Every pass is a persistent grid-stride kernel over the
// work items of all problems (a block maps its work index to a problem by
// binary search over per-pass prefix sums), so the batch costs seven launches
// whatever its size; problems of different sizes share each launch.
// ---------------------------------------------------------------------------
namespace kde {
namespace {

// Linear binning arithmetic for the batch kernel (the rounding rules of
// kde_bin: t = (x - lo) s rounded in the samples' type, i = floor(t),
// f = t - i, the last node folded to (M-2, 1), q = round-half-even(f 2^32)
// with q = 2^32 written as (i+1, 0); part w of the unit mass gives
// floor((w q + 2^31) / 2^32) to node i+1, axis 0 first).
template <typename T>
struct BinAxisLite {
  T lo, s, top;
  int M;
};

__device__ __forceinline__ float rn_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rn_sub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float rn_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rn_mul(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ bool lite_fixed(float f, int& i, unsigned& q) {
  if (f == 1.0f) {
    i += 1;
    q = 0;
  } else {
    q = __float2uint_rn(f * 4294967296.0f);  // f 2^32 < 2^32 exactly
  }
  return true;
}
template <typename T>
__device__ __forceinline__ bool lite_position(T x, const BinAxisLite<T>& a, int& i, unsigned& q) {
  const T t = rn_mul(rn_sub(x, a.lo), a.s);
  if constexpr (sizeof(T) == 8) {
    uint64_t V = 0;
    const bool in = fixed_position((uint64_t)__double_as_longlong(t),
                                   (uint64_t)__double_as_longlong(a.top), &V);
    i = (int)(V >> 32);
    q = (unsigned)V;
    return in;
  } else {
    if (!(t >= T(0) && t <= a.top)) return false;
    const T fl = floor(t);
    i = (int)fl;
    T f = rn_sub(t, fl);
    if (i == a.M - 1) {
      i = a.M - 2;
      f = T(1);
    }
    return lite_fixed(f, i, q);
  }
}

__device__ __forceinline__ unsigned lite_mulhi(unsigned long long w, unsigned q) {
  const unsigned wl = (unsigned)w, wh = (unsigned)(w >> 32);
  return wh * q + __umulhi(wl, q) + ((wl * q) >> 31);
}

// corners (0,0), (0,1), (1,0), (1,1) (axis-0 offset first)
__device__ __forceinline__ void lite_corner_weights2(const unsigned* q, unsigned long long* w) {
  const unsigned long long one = 1ull << 32;
  const unsigned long long a1 = lite_mulhi(one, q[0]), a0 = one - a1;
  w[1] = lite_mulhi(a0, q[1]);
  w[0] = a0 - w[1];
  w[3] = lite_mulhi(a1, q[1]);
  w[2] = a1 - w[3];
}

// BP_BIN: every problem's binning (the persistent queue's items); the staged
// form splits it into problems binned by direct adds (BP_DBIN) and by
// block-private counts, in two classes of shared memory (BP_PBIN, + 1).
enum BatchPass { BP_BIN = 0, BP_KROWS, BP_KCOLS, BP_ROWS, BP_MID, BP_C2R, BP_DBIN, BP_PBIN,
                 BP_COUNT = BP_PBIN + 2 };

template <typename T>
struct BatchItem {
  using V = typename Cplx<T>::type;
  int64_t x_off, n;          // samples [x_off, x_off + n) of the concatenated X
  T lo[2], s[2], top[2];     // binning: lo, (M-1)/(hi-lo), M-1 in the samples' type
  int M[2], P[2], Q, L[2];
  int64_t counts_off;        // int64 elements
  int64_t kspec_off;         // real elements, [Q][P0] (column-major spectrum)
  int64_t A_off;             // complex elements, [M0][Q]
  int64_t T1_off;            // complex elements, [2 L0 + 1][Q]
  int64_t dens_off;          // real elements, [M0][M1]
  LinePlan lp[2];
  const V* tw[2];
  KGen<T> gen;
};

__device__ __forceinline__ int find_item(const int* __restrict__ start, int count, int w) {
  int lo = 0, hi = count - 1;  // largest i with start[i] <= w
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= w) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <typename T>
struct BatchArgs {
  const BatchItem<T>* items;
  const int* wstart;   // [BP_COUNT][count + 1] work prefix per pass
  int count;
  int tpl_rows, tpl_cols;
  const T* X;
  long long* counts;
  T* kspec;
  typename Cplx<T>::type* A;
  typename Cplx<T>::type* T1;
  T* density;
};

// Binning of every problem's samples: the same arithmetic as the direct
// method.  Work item = (problem, chunk of kBinChunk samples); a block takes
// whole work items, so each knows its problem without a per-sample search.
constexpr int kBinChunk = 8192;

// Chunk vb of problem it's samples (all threads of the block).
template <typename T>
__device__ __forceinline__ void batch_bin_item(const BatchArgs<T>& a, int it, int64_t vb) {
  {
    const BatchItem<T>& B = a.items[it];
    const int64_t c0 = vb * kBinChunk;
    const int64_t c1 = min(B.n, c0 + kBinChunk);
    // two adjacent lanes per sample: lane parity p adds the corners at
    // offset p along the last axis, so a lane pair's two words share a
    // 32-byte sector three times in four and coalesce into one request
    const int par = threadIdx.x & 1;
    const int64_t jstep = blockDim.x >> 1;
    constexpr int U = 8;  // samples whose coordinates are loaded before any is added
    unsigned long long* c = reinterpret_cast<unsigned long long*>(a.counts + B.counts_off);
    for (int64_t j0 = c0 + (threadIdx.x >> 1); j0 < c1; j0 += U * jstep) {
      T xs[U][2];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int64_t j = j0 + u * jstep;
        xs[u][0] = j < c1 ? a.X[(B.x_off + j) * 2] : T(0);
        xs[u][1] = j < c1 ? a.X[(B.x_off + j) * 2 + 1] : T(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (j0 + u * jstep >= c1) break;
        int i[2];
        unsigned q[2];
        bool in = true;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          BinAxisLite<T> ax{B.lo[k], B.s[k], B.top[k], B.M[k]};
          in &= lite_position<T>(xs[u][k], ax, i[k], q[k]);
        }
        if (!in) continue;
        unsigned long long wt[4];
        lite_corner_weights2(q, wt);
        const unsigned long long w0 = par ? wt[1] : wt[0], w1 = par ? wt[3] : wt[2];
        const int64_t base = (int64_t)i[0] * B.M[1] + i[1] + par;
        if (w0) atomicAdd(c + base, w0);
        if (w1) atomicAdd(c + base + B.M[1], w1);
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) kde_batch_bin_kernel(BatchArgs<T> a) {
  const int* wst = a.wstart + BP_DBIN * (a.count + 1);
  const int total = wst[a.count];
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    const int it = find_item(wst, a.count, w);
    batch_bin_item<T>(a, it, w - wst[it]);
  }
}

// Problems with few cells for their samples: a block's chunk summed in shared
// memory and added into the problem's counts once, as kde_bin_private_kernel
// does (the same split sums, exact for the at most 2^15 samples of a chunk).
// One block an item; 64 datasets of 10^3 to 10^6 samples on 64^2 to 1024^2
// grids: the binning 325 us by direct adds alone, 145 + 66 with these (event
// times); side by side on the plan's two streams the batch takes 656 us, one
// after the other 699 and by direct adds alone 829 (with 512 threads a block,
// 661 side by side).
constexpr int kBatchPrivCells[2] = {6144, 24576};   // 48 and 192 KB of sums
template <typename T, int kBatchPrivThreads>
__global__ void __launch_bounds__(kBatchPrivThreads)
kde_batch_bin_private_kernel(BatchArgs<T> a, int pass) {
  extern __shared__ __align__(16) unsigned priv_sm[];
  const int* wst = a.wstart + pass * (a.count + 1);
  const int it = find_item(wst, a.count, blockIdx.x);
  const BatchItem<T>& B = a.items[it];
  const int v = blockIdx.x - wst[it], nb = wst[it + 1] - wst[it];
  const int M1 = B.M[1], cells = B.M[0] * M1, words = (cells + 3) & ~3;
  const int64_t c0 = B.n * v / nb, c1 = B.n * (v + 1) / nb;
  unsigned *lo = priv_sm, *hi = priv_sm + words;
  for (int j = threadIdx.x; j < words / 2; j += kBatchPrivThreads)
    reinterpret_cast<uint4*>(priv_sm)[j] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  constexpr int U = 4;
  for (int64_t j0 = c0 + threadIdx.x; j0 < c1; j0 += U * kBatchPrivThreads) {
    T xs[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t j = j0 + u * kBatchPrivThreads;
      xs[u][0] = j < c1 ? a.X[(B.x_off + j) * 2] : T(0);
      xs[u][1] = j < c1 ? a.X[(B.x_off + j) * 2 + 1] : T(0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j0 + u * kBatchPrivThreads >= c1) break;
      int i[2];
      unsigned q[2];
      bool in = true;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        BinAxisLite<T> ax{B.lo[k], B.s[k], B.top[k], B.M[k]};
        in &= lite_position<T>(xs[u][k], ax, i[k], q[k]);
      }
      if (!in) continue;
      unsigned long long w[4];
      lite_corner_weights2(q, w);
      const int base = i[0] * M1 + i[1];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (w[c] == 0) continue;   // also a corner beyond the last node
        const int idx = base + (c >> 1) * M1 + (c & 1);
        if (!KDE_DCHECK(idx >= 0 && idx < cells, KDE_DBG_BIN_DIRECT)) continue;
        const unsigned l = (unsigned)w[c] & 0xFFFFu;
        if (l) atomicAdd(lo + idx, l);
        atomicAdd(hi + idx, (unsigned)(w[c] >> 16));
      }
    }
  }
  __syncthreads();
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(a.counts + B.counts_off);
  const int first = (int)((int64_t)cells * v / nb);   // blocks of a problem start apart
  for (int j0 = threadIdx.x; j0 < cells; j0 += kBatchPrivThreads) {
    const int j = j0 + first < cells ? j0 + first : j0 + first - cells;
    const unsigned long long s = ((unsigned long long)hi[j] << 16) + lo[j];
    if (s) atomicAdd(cnt + j, s);
  }
}

// Per-block parameters of a pass over one problem (set by one thread).
template <typename T>
struct PassShared {
  RowsParams<T> rp;
  C2RParams<T> cr;
  ColsParams<T> cp;
  KGen<T> gen;
};

template <typename T>
__device__ __forceinline__ void batch_pass_params(const BatchArgs<T>& a, int PASS, int it,
                                                  PassShared<T>& sh) {
  {
    {
      const BatchItem<T>& B = a.items[it];
      RowsParams<T>& rp = sh.rp;
      C2RParams<T>& cr = sh.cr;
      ColsParams<T>& cp = sh.cp;
      KGen<T>& gen = sh.gen;
      if (PASS == BP_KROWS || PASS == BP_ROWS) {
        RowsParams<T> r{};
        r.Q = B.Q;
        r.lp = B.lp[1];
        r.tw = B.tw[1];
        r.tpl = a.tpl_rows;
        if (PASS == BP_KROWS) {
          r.nrows = 2 * B.L[0] + 1;
          r.out = a.T1 + B.T1_off;
          gen = B.gen;
        } else {
          r.nrows = B.M[0];
          r.Min = B.M[1];
          r.in_stride = B.M[1];
          r.out = a.A + B.A_off;
        }
        rp = r;
      } else if (PASS == BP_C2R) {
        C2RParams<T> c{};
        c.in = a.A + B.A_off;
        c.out = a.density + B.dens_off;
        c.nrows = B.M[0];
        c.Mout = B.M[1];
        c.Q = B.Q;
        c.tpl = a.tpl_rows;
        c.lp = B.lp[1];
        c.tw = B.tw[1];
        cr = c;
      } else {
        ColsParams<T> c{};
        c.S = B.Q;
        c.lp = B.lp[0];
        c.tw = B.tw[0];
        c.tpl = a.tpl_cols;
        if (PASS == BP_KCOLS) {
          c.in = a.T1 + B.T1_off;
          c.out_real = a.kspec + B.kspec_off;
          c.Nin = 2 * B.L[0] + 1;
          c.Lw = B.L[0];
        } else {
          c.in = a.A + B.A_off;
          c.out = a.A + B.A_off;
          c.K = a.kspec + B.kspec_off;
          c.Nin = B.M[0];
          c.Nout = B.M[0];
          c.Lw = -1;
        }
        cp = c;
      }
    }
  }
}

template <typename T>
__device__ __forceinline__ void batch_pass_body(const BatchArgs<T>& a, int PASS, int it, int64_t vb,
                                                const PassShared<T>& sh) {
  if (PASS == BP_KROWS) rows_kgen_body<T>(sh.gen, sh.rp, vb);
  if (PASS == BP_ROWS) rows_counts_body<T>(a.counts + a.items[it].counts_off, sh.rp, vb);
  if (PASS == BP_C2R) rows_c2r_body<T>(sh.cr, vb);
  if (PASS == BP_KCOLS) cols_body_slab<T, COL_FWD_REAL>(sh.cp, 0, vb);
  if (PASS == BP_MID) cols_body_slab<T, COL_MID>(sh.cp, 0, vb);
}

template <typename T, int PASS>
__global__ void __launch_bounds__(256) kde_batch_pass_kernel(BatchArgs<T> a) {
  __shared__ PassShared<T> sh;
  __shared__ int item, base;
  const int* wst = a.wstart + PASS * (a.count + 1);
  const int total = wst[a.count];
  for (int w = blockIdx.x; w < total; w += gridDim.x) {
    if (threadIdx.x == 0) {
      const int it = find_item(wst, a.count, w);
      item = it;
      base = wst[it];
      batch_pass_params<T>(a, PASS, it, sh);
    }
    __syncthreads();
    batch_pass_body<T>(a, PASS, item, w - base, sh);
    __syncthreads();  // the next item reloads twiddles and parameters
  }
}

// ---------------------------------------------------------------------------
// The whole ragged batch as one persistent launch.  Work items of every
// problem and stage (zero the counts, kernel rows, binning, kernel spectrum,
// count rows, middle axis, output rows) form one queue, in stage order or
// problem by problem (largest first); blocks claim items with an atomic
// counter.  An item waits for the stages of its own problem it reads from
// (per-problem completion counters); in either order those precede it in
// the queue, so a claimed item only waits on items already claimed by
// running blocks: the queue always progresses.  Every
// wait is bounded: after wait_polls polls the block records the timeout in
// the status word, raises the abort flag (waiters of this launch then give
// up at once) and leaves.  The last block out resets the queue for the next
// launch.  Completion: every thread fences its writes, the block barrier,
// then one thread adds to the counter; a waiter fences after it sees the
// count, and the stages read produced data through L2 (__ldcg).
// ---------------------------------------------------------------------------
enum PersistStage { PS_ZERO = 0, PS_KROWS, PS_BIN, PS_KCOLS, PS_ROWS, PS_MID, PS_C2R, PS_COUNT };
constexpr int kZeroChunk = 1 << 16;        // int64 counts zeroed per item
constexpr unsigned kCtlWords = 4;          // next, exited, abort, status; then done[count][PS_COUNT]
constexpr unsigned kDefaultWaitPolls = 1u << 22;   // about a second of polls

template <typename T>
struct PersistArgs {
  BatchArgs<T> a;
  const int* pstart;                // [PS_COUNT][count + 1] items per problem, prefix
  const int4* queue;                // per queue position: problem, stage, item within it
  int total;                        // queue length
  unsigned* ctl;
  unsigned wait_polls;
  int withhold;                     // stage whose completions are never signalled (-1: none)
};

__device__ __forceinline__ int stage_pass(int st) {
  switch (st) {
    case PS_KROWS: return BP_KROWS;
    case PS_KCOLS: return BP_KCOLS;
    case PS_ROWS: return BP_ROWS;
    case PS_MID: return BP_MID;
    case PS_C2R: return BP_C2R;
    default: return -1;
  }
}

template <typename T>
__global__ void __launch_bounds__(256) kde_batch_persistent_kernel(PersistArgs<T> pa) {
  __shared__ PassShared<T> sh;
  __shared__ unsigned s_item;
  __shared__ int s_ok;
  const BatchArgs<T>& a = pa.a;
  unsigned* ctl = pa.ctl;
  unsigned* done = ctl + kCtlWords;
  const unsigned total = (unsigned)pa.total;
  while (true) {
    if (threadIdx.x == 0) s_item = atomicAdd(&ctl[0], 1u);
    __syncthreads();
    const unsigned item = s_item;
    if (item >= total) break;
    const int4 q = pa.queue[item];
    const int it = q.x, st = q.y;
    const int64_t vb = q.z;
    if (threadIdx.x == 0) {
      int dep[2] = {-1, -1};
      if (st == PS_BIN) dep[0] = PS_ZERO;
      if (st == PS_KCOLS) dep[0] = PS_KROWS;
      if (st == PS_ROWS) dep[0] = PS_BIN;
      if (st == PS_MID) {
        dep[0] = PS_ROWS;
        dep[1] = PS_KCOLS;
      }
      if (st == PS_C2R) dep[0] = PS_MID;
      bool ok = true;
      for (int k = 0; k < 2 && ok; ++k) {
        if (dep[k] < 0) continue;
        const int* pd = pa.pstart + dep[k] * (a.count + 1);
        const unsigned need = (unsigned)(pd[it + 1] - pd[it]);
        volatile unsigned* cnt = done + (size_t)it * PS_COUNT + dep[k];
        volatile unsigned* abort_flag = ctl + 2;
        unsigned polls = 0;
        while (*cnt < need) {
          if (*abort_flag || ++polls > pa.wait_polls) {
            ok = false;
            break;
          }
          __nanosleep(256);
        }
      }
      if (!ok) {
        atomicExch(&ctl[3], 1u);   // status: a wait gave up (kept until checked)
        atomicExch(&ctl[2], 1u);   // abort this launch
      }
      __threadfence();
      s_ok = ok;
      if (ok && stage_pass(st) >= 0) batch_pass_params<T>(a, stage_pass(st), it, sh);
    }
    __syncthreads();
    if (!s_ok) break;
    if (st == PS_ZERO) {
      const BatchItem<T>& B = a.items[it];
      const int64_t cells = (int64_t)B.M[0] * B.M[1];
      long long* c = a.counts + B.counts_off;
      for (int64_t i = vb * kZeroChunk + threadIdx.x; i < min(cells, (vb + 1) * kZeroChunk);
           i += blockDim.x)
        c[i] = 0;
    } else if (st == PS_BIN) {
      batch_bin_item<T>(a, it, vb);
    } else {
      batch_pass_body<T>(a, stage_pass(st), it, vb, sh);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && st != pa.withhold) atomicAdd(done + (size_t)it * PS_COUNT + st, 1u);
  }
  // the last block out resets the queue and the counters for the next launch
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(&ctl[1], 1u) == gridDim.x - 1) {
      for (int i = 0; i < a.count * PS_COUNT; ++i) done[i] = 0;
      ctl[0] = 0;
      ctl[2] = 0;
      __threadfence();
      ctl[1] = 0;
    }
  }
}

}  // namespace
}  // namespace kde

struct kde_batch_plan_s {
  int count;
  int precision;
  std::vector<kde_plan_s*> plans;   // per problem: info and twiddles
  void* items_dev;                  // BatchItem<T>[count]
  int* wstart_dev;                  // [BP_COUNT][count + 1]
  std::vector<int> wstart;          // host copy
  int64_t x_total, counts_elems, kspec_elems, A_elems, T1_elems, dens_elems;
  int Pmax;
  int priv_cells[2];                // largest grid of each private binning class
  int tpl_rows, tpl_cols;           // launch shape (tunable)
  int mode;                         // KDE_BATCH_PERSISTENT or KDE_BATCH_STAGED (tunable)
  int* pstart_dev;                  // [PS_COUNT][count + 1] items per problem (persistent queue)
  std::vector<int> pstart;
  int4* queue_dev;                  // the persistent queue (problem, stage, item)
  int queue_len, queue_cap;
  int queue_order;                  // KDE_BATCH_QUEUE_STAGES or KDE_BATCH_QUEUE_PROBLEMS
  unsigned* ctl_dev;                // queue control words and completion counters
  unsigned wait_polls;
  int withhold;
  size_t workspace_bytes;
  std::vector<int64_t> n;           // samples per problem
  std::vector<kde_batch_item> items;  // the problems, for re-planning by the tuner
  kde_opts opts;
  int pad_policy;                   // KDE_BATCH_PAD_SMALLEST or KDE_BATCH_PAD_FEWEST_STAGES
  int radix_order;                  // 0: largest radix first, 1: smallest first
  // the kernel-grid passes need no samples: they run on this stream beside
  // the binning (fork and join events on the caller's stream)
  cudaStream_t side;
  cudaEvent_t fork, zeroed, join;
};

namespace kde {
namespace {

constexpr int kBatchLines = 2;  // lines per block in the batch passes

template <typename T>
kde_status batch_upload(kde_batch_plan_s* bp, const kde_batch_item* items) {
  using V = typename Cplx<T>::type;
  std::vector<BatchItem<T>> h(bp->count);
  int64_t x = 0, cnt = 0, ks = 0, A = 0, T1 = 0, de = 0;
  for (int i = 0; i < bp->count; ++i) {
    const kde_plan_s* pl = bp->plans[i];
    const kde_plan_info& I = pl->info;
    BatchItem<T>& B = h[i];
    B.x_off = x;
    B.n = items[i].n;
    for (int k = 0; k < 2; ++k) {
      const double sk = (double)(I.M[k] - 1) / (pl->hi[k] - pl->lo[k]);
      B.lo[k] = (T)pl->lo[k];
      B.s[k] = (T)sk;
      B.top[k] = (T)(I.M[k] - 1);
      B.M[k] = (int)I.M[k];
      B.P[k] = (int)I.P[k];
      B.L[k] = (int)I.L[k];
      B.lp[k] = line_plan(I, k);
      B.tw[k] = twiddles<T>(pl, k);
    }
    B.Q = (int)I.Q;
    B.counts_off = cnt;
    B.kspec_off = ks;
    B.A_off = A;
    B.T1_off = T1;
    B.dens_off = de;
    kde_status sg = kgen_for<T>(I, pl->H, I.det_H, I.L, pl->layout_mode == KDE_LAYOUT_WAND, &B.gen);
    if (sg != KDE_OK) return sg;
    B.gen.C = (T)(std::pow(6.283185307179586476925287, -1.0) / std::sqrt(I.det_H) /
                  ((double)items[i].n * 4294967296.0 * (double)I.P[0] * (double)I.P[1]));
    x += items[i].n;
    cnt += I.M[0] * I.M[1];
    ks += I.P[0] * I.Q;
    A += I.M[0] * I.Q;
    T1 += (2 * I.L[0] + 1) * I.Q;
    de += I.M[0] * I.M[1];
  }
  bp->x_total = x;
  bp->counts_elems = cnt;
  bp->kspec_elems = ks;
  bp->A_elems = A;
  bp->T1_elems = T1;
  bp->dens_elems = de;
  cudaError_t e = cudaMalloc(&bp->items_dev, sizeof(BatchItem<T>) * bp->count);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(batch items)");
  e = cudaMemcpy(bp->items_dev, h.data(), sizeof(BatchItem<T>) * bp->count, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(batch items)");
  const size_t cb = sizeof(V), rb = sizeof(T);
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  bp->workspace_bytes = up(cnt * 8) + up(ks * rb) + up(A * cb) + up(T1 * cb);
  return KDE_OK;
}

int64_t items_n(const kde_batch_plan_s* bp, int i) { return bp->n[i]; }

// Work items per problem and pass for the current launch shape; uploaded.
kde_status batch_work(kde_batch_plan_s* bp) {
  const int c = bp->count;
  bp->wstart.assign((size_t)BP_COUNT * (c + 1), 0);
  const int lr = kBatchLines, lc = kBatchLines;
  bp->priv_cells[0] = bp->priv_cells[1] = 0;
  for (int i = 0; i < c; ++i) {
    const kde_plan_info& I = bp->plans[i]->info;
    int w[BP_COUNT] = {};
    w[BP_BIN] = (int)((bp->plans[i] ? items_n(bp, i) : 0) + kBinChunk - 1) / kBinChunk;
    // the rule of kde_bin's private counts in 2-D; a chunk holds half as many
    // samples as the cells it flushes (at most 2^15; with four times as many
    // the two launches took 46 us each)
    const int64_t n = bp->plans[i] ? items_n(bp, i) : 0, cells = I.M[0] * I.M[1];
    if (cells <= kBatchPrivCells[1] && n >= 4096 + 8 * cells) {
      const int64_t per = std::min<int64_t>(1 << 15, std::max<int64_t>(2048, cells / 2));
      const int cls = cells > kBatchPrivCells[0];
      w[BP_PBIN + cls] = (int)((n + per - 1) / per);
      bp->priv_cells[cls] = std::max(bp->priv_cells[cls], (int)cells);
    } else {
      w[BP_DBIN] = w[BP_BIN];
    }
    w[BP_KROWS] = (int)((((2 * I.L[0] + 1) + 1) / 2 + lr - 1) / lr);
    w[BP_KCOLS] = (int)((I.Q + 2 * lc - 1) / (2 * lc));
    w[BP_ROWS] = (int)(((I.M[0] + 1) / 2 + lr - 1) / lr);
    w[BP_MID] = (int)((I.Q + lc - 1) / lc);
    w[BP_C2R] = w[BP_ROWS];
    for (int pss = 0; pss < BP_COUNT; ++pss)
      bp->wstart[(size_t)pss * (c + 1) + i + 1] = bp->wstart[(size_t)pss * (c + 1) + i] + w[pss];
  }
  // the persistent queue's stages: zeroing of the counts, then the passes
  bp->pstart.assign((size_t)PS_COUNT * (c + 1), 0);
  for (int i = 0; i < c; ++i) {
    const kde_plan_info& I = bp->plans[i]->info;
    int w[PS_COUNT];
    const int* ws = bp->wstart.data();
    auto per = [&](int pss) { return ws[(size_t)pss * (c + 1) + i + 1] - ws[(size_t)pss * (c + 1) + i]; };
    w[PS_ZERO] = (int)((I.M[0] * I.M[1] + kZeroChunk - 1) / kZeroChunk);
    w[PS_KROWS] = per(BP_KROWS);
    w[PS_BIN] = per(BP_BIN);
    w[PS_KCOLS] = per(BP_KCOLS);
    w[PS_ROWS] = per(BP_ROWS);
    w[PS_MID] = per(BP_MID);
    w[PS_C2R] = per(BP_C2R);
    for (int st = 0; st < PS_COUNT; ++st)
      bp->pstart[(size_t)st * (c + 1) + i + 1] = bp->pstart[(size_t)st * (c + 1) + i] + w[st];
  }
  // the queue: stage by stage, or problem by problem with the most work first
  std::vector<int4> q;
  auto items_of = [&](int i, int st) {
    return bp->pstart[(size_t)st * (c + 1) + i + 1] - bp->pstart[(size_t)st * (c + 1) + i];
  };
  if (bp->queue_order == KDE_BATCH_QUEUE_PROBLEMS) {
    std::vector<int> order(c);
    for (int i = 0; i < c; ++i) order[i] = i;
    std::vector<int64_t> work(c, 0);
    for (int i = 0; i < c; ++i) {
      const kde_plan_info& I = bp->plans[i]->info;
      work[i] = bp->n[i] + (int64_t)I.P[0] * I.P[1];
    }
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return work[x] > work[y]; });
    for (int i : order)
      for (int st = 0; st < PS_COUNT; ++st)
        for (int v = 0; v < items_of(i, st); ++v) q.push_back(make_int4(i, st, v, 0));
  } else {
    for (int st = 0; st < PS_COUNT; ++st)
      for (int i = 0; i < c; ++i)
        for (int v = 0; v < items_of(i, st); ++v) q.push_back(make_int4(i, st, v, 0));
  }
  cudaError_t e = cudaSuccess;
  if ((int)q.size() > bp->queue_cap) {
    if (bp->queue_dev) cudaFree(bp->queue_dev);
    bp->queue_dev = nullptr;
    bp->queue_cap = 0;
    e = cudaMalloc((void**)&bp->queue_dev, sizeof(int4) * q.size());
    if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(batch queue)");
    bp->queue_cap = (int)q.size();
  }
  bp->queue_len = (int)q.size();
  e = cudaMemcpy(bp->wstart_dev, bp->wstart.data(), sizeof(int) * bp->wstart.size(),
                 cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(bp->pstart_dev, bp->pstart.data(), sizeof(int) * bp->pstart.size(),
                   cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(bp->queue_dev, q.data(), sizeof(int4) * q.size(), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaMemcpy(batch work)");
}

template <typename T>
kde_status batch_persistent(kde_batch_plan_s* bp, const BatchArgs<T>& a0, cudaStream_t st) {
  PersistArgs<T> pa{};
  pa.a = a0;
  pa.a.tpl_cols = pa.a.tpl_rows;   // one block shape for every stage
  pa.pstart = bp->pstart_dev;
  pa.queue = bp->queue_dev;
  pa.total = bp->queue_len;
  pa.ctl = bp->ctl_dev;
  pa.wait_polls = bp->wait_polls;
  pa.withhold = bp->withhold;
  auto* fn = kde_batch_persistent_kernel<T>;
  cudaError_t e = allow_smem(fn);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
  const size_t smem = line_smem<T>(bp->Pmax, kBatchLines);
  const int threads = bp->tpl_rows * kBatchLines;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
  if (e != cudaSuccess) return cuda_fail(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
  const int grid = std::max(1, std::min(pa.total, std::max(1, per_sm) * num_sms()));
  LaunchScope ls("kde_batch_persistent_kernel", st);
  fn<<<grid, threads, smem, st>>>(pa);
  e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_batch_persistent_kernel");
}

template <typename T>
kde_status batch_eval_impl(kde_batch_plan_s* bp, const void* X, void* density, void* ws,
                           cudaStream_t st) {
  using V = typename Cplx<T>::type;
  auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
  char* w = (char*)ws;
  BatchArgs<T> a{};
  a.items = (const BatchItem<T>*)bp->items_dev;
  a.wstart = bp->wstart_dev;
  a.count = bp->count;
  a.tpl_rows = bp->tpl_rows;
  a.tpl_cols = bp->tpl_cols;
  a.X = (const T*)X;
  a.counts = (long long*)w;
  w += up(bp->counts_elems * 8);
  a.kspec = (T*)w;
  w += up(bp->kspec_elems * sizeof(T));
  a.A = (V*)w;
  w += up(bp->A_elems * sizeof(V));
  a.T1 = (V*)w;
  a.density = (T*)density;
  if (bp->mode == KDE_BATCH_PERSISTENT) return batch_persistent<T>(bp, a, st);
  // the kernel-grid passes (no samples needed) fork onto the plan's side
  // stream and join before the count rows
  cudaError_t e = cudaEventRecord(bp->fork, st);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(bp->side, bp->fork, 0);
  if (e != cudaSuccess) return cuda_fail(e, "fork (batch kernel grid)");
  e = cudaMemsetAsync(a.counts, 0, bp->counts_elems * 8, st);
  if (e == cudaSuccess) e = cudaEventRecord(bp->zeroed, st);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(batch counts)");
  const int sms = num_sms();
  const int c = bp->count;
  {
    const int total = bp->wstart[(size_t)BP_DBIN * (c + 1) + c];
    if (total > 0) {
      LaunchScope ls("kde_batch_bin_kernel", st);
      kde_batch_bin_kernel<T><<<std::min(total, sms * 8), 256, 0, st>>>(a);
      if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_batch_bin_kernel");
    }
  }
  auto run = [&](auto fn, int pass, int tpl, const char* name, cudaStream_t ss) -> kde_status {
    const int total = bp->wstart[(size_t)pass * (c + 1) + c];
    if (total == 0) return KDE_OK;
    cudaError_t e2 = allow_smem(fn);
    if (e2 != cudaSuccess) return cuda_fail(e2, "cudaFuncSetAttribute");
    const size_t smem = line_smem<T>(bp->Pmax, kBatchLines);
    const int grid = std::min(total, sms * 8);
    LaunchScope ls(name, ss);
    fn<<<grid, tpl * kBatchLines, smem, ss>>>(a);
    e2 = cudaGetLastError();
    return e2 == cudaSuccess ? KDE_OK : cuda_fail(e2, name);
  };
  kde_status s;
  if ((s = run(kde_batch_pass_kernel<T, BP_KROWS>, BP_KROWS, bp->tpl_rows, "kde_batch_krows_kernel", bp->side)) != KDE_OK) return s;
  if ((s = run(kde_batch_pass_kernel<T, BP_KCOLS>, BP_KCOLS, bp->tpl_cols, "kde_batch_kcols_kernel", bp->side)) != KDE_OK) return s;
  // the private counts' problems beside the others' binning, once zeroed
  if ((e = cudaStreamWaitEvent(bp->side, bp->zeroed, 0)) != cudaSuccess)
    return cuda_fail(e, "cudaStreamWaitEvent(batch counts)");
  for (int cls = 0; cls < 2; ++cls) {
    const int total = bp->wstart[(size_t)(BP_PBIN + cls) * (c + 1) + c];
    if (total == 0) continue;
    const size_t smem = 2 * (size_t)((bp->priv_cells[cls] + 3) & ~3) * sizeof(unsigned);
    const bool wide = smem > 100 * 1024;   // one block an SM: twice the warps
    auto* fn = wide ? kde_batch_bin_private_kernel<T, 1024> : kde_batch_bin_private_kernel<T, 512>;
    if ((e = allow_smem(fn)) != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
    LaunchScope ls("kde_batch_bin_private_kernel", bp->side);
    fn<<<total, wide ? 1024 : 512, smem, bp->side>>>(a, BP_PBIN + cls);
    if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "kde_batch_bin_private_kernel");
  }
  e = cudaEventRecord(bp->join, bp->side);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(st, bp->join, 0);
  if (e != cudaSuccess) return cuda_fail(e, "join (batch kernel grid)");
  if ((s = run(kde_batch_pass_kernel<T, BP_ROWS>, BP_ROWS, bp->tpl_rows, "kde_batch_rows_kernel", st)) != KDE_OK) return s;
  if ((s = run(kde_batch_pass_kernel<T, BP_MID>, BP_MID, bp->tpl_cols, "kde_batch_mid_kernel", st)) != KDE_OK) return s;
  return run(kde_batch_pass_kernel<T, BP_C2R>, BP_C2R, bp->tpl_rows, "kde_batch_c2r_kernel", st);
}

}  // namespace
}  // namespace kde

namespace kde {
namespace {

// Padded length of one problem's axis under a batch padding policy: the
// smallest 7-smooth size >= need, or the one with the fewest radix stages
// up to 25% longer (ties: the shorter).
int64_t batch_pad(int64_t need, int policy) {
  auto smooth = [](int64_t x) {
    for (int q : {2, 3, 5, 7})
      while (x % q == 0) x /= q;
    return x == 1;
  };
  int64_t P = need;
  while (!smooth(P)) ++P;
  if (policy != KDE_BATCH_PAD_FEWEST_STAGES) return P;
  auto stages = [](int64_t x) {
    int n = 0;
    for (int r : {8, 7, 5, 4, 3, 2})
      while (x % r == 0) {
        x /= r;
        ++n;
      }
    return n;
  };
  int64_t best = P;
  for (int64_t q = P; q <= need + need / 4; ++q)
    if (smooth(q) && stages(q) < stages(best)) best = q;
  return best;
}

// (Re)creates every problem's plan under the batch's padding policy and
// radix order (the Stockham passes run the batch; the radix plan of an axis
// is applied in the chosen order).
kde_status batch_plans(kde_batch_plan_s* bp) {
  for (auto* p : bp->plans) kde_plan_destroy(p);
  bp->plans.clear();
  bp->Pmax = 0;
  for (size_t i = 0; i < bp->items.size(); ++i) {
    const kde_batch_item& it = bp->items[i];
    kde_opts o = bp->opts;
    o.engine = KDE_ENGINE_STOCKHAM;
    kde_plan_info info{};
    kde_status s = kde_plan_info_compute(2, it.M, it.lo, it.hi, it.H, &o, &info);
    if (s != KDE_OK) return s;
    for (int k = 0; k < 2; ++k)
      o.P_min[k] = std::max(o.P_min[k], batch_pad(it.M[k] + info.L[k], bp->pad_policy));
    kde_plan p = nullptr;
    if ((s = kde_plan_create(2, it.M, it.lo, it.hi, it.H, &o, &p)) != KDE_OK) return s;
    if (bp->radix_order == 1)
      for (int k = 0; k < 2; ++k) std::reverse(p->info.radix[k], p->info.radix[k] + p->info.nstages[k]);
    bp->plans.push_back(p);
    for (int k = 0; k < 2; ++k) bp->Pmax = std::max(bp->Pmax, (int)p->info.P[k]);
  }
  return KDE_OK;
}

// Re-plans, re-uploads the problem table and the work counts.
kde_status batch_rebuild(kde_batch_plan_s* bp) {
  kde_status s = batch_plans(bp);
  if (s != KDE_OK) return s;
  if (bp->items_dev) {
    cudaFree(bp->items_dev);
    bp->items_dev = nullptr;
  }
  s = (bp->precision == KDE_F32) ? batch_upload<float>(bp, bp->items.data())
                                 : batch_upload<double>(bp, bp->items.data());
  return s == KDE_OK ? batch_work(bp) : s;
}

}  // namespace
}  // namespace kde

extern "C" kde_status kde_batch_plan_create(int count, const kde_batch_item* items,
                                            const kde_opts* opts, kde_batch_plan* out) {
  if (!out || !items || count < 1) return fail(KDE_ERR_INVALID_ARG, "bad argument");
  *out = nullptr;
  kde_batch_plan_s* bp = new (std::nothrow) kde_batch_plan_s();
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "out of host memory");
  bp->count = count;
  bp->precision = opts ? opts->precision : KDE_F32;
  bp->Pmax = 0;
  bp->tpl_rows = 64;
  bp->tpl_cols = 64;
  bp->mode = KDE_BATCH_PERSISTENT;
  bp->wait_polls = kDefaultWaitPolls;
  bp->withhold = -1;
  bp->pstart_dev = nullptr;
  bp->ctl_dev = nullptr;
  bp->queue_dev = nullptr;
  bp->queue_len = bp->queue_cap = 0;
  bp->queue_order = KDE_BATCH_QUEUE_PROBLEMS;
  bp->items_dev = nullptr;
  bp->wstart_dev = nullptr;
  bp->side = nullptr;
  bp->fork = bp->zeroed = bp->join = nullptr;
  kde_opts o{};
  o.tau = 3.7;
  if (opts) o = *opts;
  o.cols_variant = KDE_COLS_LINES;
  auto cleanup = [&](kde_status s) {
    for (auto* p : bp->plans) kde_plan_destroy(p);
    if (bp->items_dev) cudaFree(bp->items_dev);
    if (bp->wstart_dev) cudaFree(bp->wstart_dev);
    if (bp->pstart_dev) cudaFree(bp->pstart_dev);
    if (bp->ctl_dev) cudaFree(bp->ctl_dev);
    if (bp->queue_dev) cudaFree(bp->queue_dev);
    if (bp->side) cudaStreamDestroy(bp->side);
    if (bp->fork) cudaEventDestroy(bp->fork);
    if (bp->zeroed) cudaEventDestroy(bp->zeroed);
    if (bp->join) cudaEventDestroy(bp->join);
    delete bp;
    return s;
  };
  for (int i = 0; i < count; ++i) {
    if (items[i].n < 1 || items[i].n >= (int64_t(1) << 31))
      return cleanup(fail(KDE_ERR_INVALID_ARG, "every problem needs 1 <= n < 2^31"));
    bp->n.push_back(items[i].n);
    bp->items.push_back(items[i]);
  }
  bp->opts = o;
  bp->pad_policy = KDE_BATCH_PAD_SMALLEST;
  bp->radix_order = 0;
  kde_status s0 = batch_plans(bp);
  if (s0 != KDE_OK) return cleanup(s0);
  const size_t cb = (bp->precision == KDE_F32) ? 8 : 16;
  if (line_smem<float>(bp->Pmax, kBatchLines) / 8 * cb > kSmemMax)
    return cleanup(fail(KDE_ERR_UNSUPPORTED, "padded size too large for the batch passes"));
  cudaError_t e = cudaMalloc((void**)&bp->wstart_dev, sizeof(int) * BP_COUNT * (count + 1));
  if (e == cudaSuccess) e = cudaMalloc((void**)&bp->pstart_dev, sizeof(int) * PS_COUNT * (count + 1));
  const size_t ctl_bytes = sizeof(unsigned) * (kCtlWords + (size_t)PS_COUNT * count);
  if (e == cudaSuccess) e = cudaMalloc((void**)&bp->ctl_dev, ctl_bytes);
  if (e == cudaSuccess) e = cudaMemset(bp->ctl_dev, 0, ctl_bytes);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "cudaMalloc(batch work)"));
  kde_status s = (bp->precision == KDE_F32) ? batch_upload<float>(bp, items) : batch_upload<double>(bp, items);
  if (s == KDE_OK) s = batch_work(bp);
  if (s != KDE_OK) return cleanup(s);
  int lo_prio = 0, hi_prio = 0;
  cudaDeviceGetStreamPriorityRange(&lo_prio, &hi_prio);
  e = cudaStreamCreateWithPriority(&bp->side, cudaStreamNonBlocking, hi_prio);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&bp->fork, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&bp->zeroed, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&bp->join, cudaEventDisableTiming);
  if (e != cudaSuccess) return cleanup(cuda_fail(e, "side stream (batch kernel grid)"));
  *out = bp;
  return KDE_OK;
}

extern "C" kde_status kde_batch_plan_query(kde_batch_plan bp, int64_t* x_rows, int64_t* density_elems,
                                           size_t* workspace_bytes) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (x_rows) *x_rows = bp->x_total;
  if (density_elems) *density_elems = bp->dens_elems;
  if (workspace_bytes) *workspace_bytes = bp->workspace_bytes;
  return KDE_OK;
}

extern "C" kde_status kde_batch_set_shape(kde_batch_plan bp, int tpl_rows, int tpl_cols) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  for (int t : {tpl_rows, tpl_cols})
    if (t != 32 && t != 64 && t != 128) return fail(KDE_ERR_INVALID_ARG, "threads per line: 32, 64 or 128");
  bp->tpl_rows = tpl_rows;
  bp->tpl_cols = tpl_cols;
  return KDE_OK;
}

extern "C" kde_status kde_batch_set_mode(kde_batch_plan bp, int mode) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (mode != KDE_BATCH_PERSISTENT && mode != KDE_BATCH_STAGED)
    return fail(KDE_ERR_INVALID_ARG, "mode: KDE_BATCH_PERSISTENT or KDE_BATCH_STAGED");
  bp->mode = mode;
  return KDE_OK;
}

extern "C" kde_status kde_batch_get_mode(kde_batch_plan bp, int* mode) {
  if (!bp || !mode) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  *mode = bp->mode;
  return KDE_OK;
}

extern "C" kde_status kde_batch_set_wait(kde_batch_plan bp, uint32_t polls, int withhold_stage) {
  if (!bp || polls == 0) return fail(KDE_ERR_INVALID_ARG, "need a plan and polls >= 1");
  if (withhold_stage < -1 || withhold_stage >= PS_COUNT)
    return fail(KDE_ERR_INVALID_ARG, "withhold_stage: -1 or a stage index 0..6");
  bp->wait_polls = polls;
  bp->withhold = withhold_stage;
  return KDE_OK;
}

extern "C" kde_status kde_batch_check(kde_batch_plan bp, kde_stream_t stream) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  unsigned flag = 0;
  cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
  if (e == cudaSuccess) e = cudaMemcpy(&flag, bp->ctl_dev + 3, sizeof(unsigned), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess && flag) e = cudaMemset(bp->ctl_dev + 3, 0, sizeof(unsigned));
  if (e != cudaSuccess) return cuda_fail(e, "kde_batch_check");
  if (flag) return fail(KDE_ERR_TIMEOUT, "a wait of the persistent batch kernel gave up; the output is invalid");
  return KDE_OK;
}

extern "C" kde_status kde_batch_eval(kde_batch_plan bp, const void* X, void* density, void* workspace,
                                     size_t workspace_bytes, kde_stream_t stream) {
  if (!bp || !density || (!X && bp->x_total > 0)) return fail(KDE_ERR_INVALID_ARG, "NULL argument");
  if (!workspace || workspace_bytes < bp->workspace_bytes)
    return fail(KDE_ERR_WORKSPACE, "workspace smaller than the batch plan needs");
  if (((uintptr_t)workspace & 255) != 0) return fail(KDE_ERR_INVALID_ARG, "workspace not 256-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  if (bp->precision == KDE_F32) return batch_eval_impl<float>(bp, X, density, workspace, st);
  return batch_eval_impl<double>(bp, X, density, workspace, st);
}

extern "C" kde_status kde_batch_plan_destroy(kde_batch_plan bp) {
  if (!bp) return KDE_OK;
  for (auto* p : bp->plans) kde_plan_destroy(p);
  cudaError_t e = cudaSuccess;
  if (bp->side) cudaStreamDestroy(bp->side);
  if (bp->fork) cudaEventDestroy(bp->fork);
  if (bp->zeroed) cudaEventDestroy(bp->zeroed);
  if (bp->join) cudaEventDestroy(bp->join);
  if (bp->items_dev) e = cudaFree(bp->items_dev);
  if (bp->wstart_dev) cudaFree(bp->wstart_dev);
  if (bp->pstart_dev) cudaFree(bp->pstart_dev);
  if (bp->ctl_dev) cudaFree(bp->ctl_dev);
  if (bp->queue_dev) cudaFree(bp->queue_dev);
  delete bp;
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "cudaFree(batch)");
}

// Tuner for a batch plan: times kde_batch_eval with CUDA events on the
// stream (one warm-up and reps timed runs each) over the padding policy
// (smallest 7-smooth length, or the fewest radix stages within 25%), the
// radix order (largest or smallest radix first), the mode (persistent or
// staged) and the threads per line (32, 64, 128; rows and columns alike in
// the persistent mode, every pair in the staged one), skipping settings
// whose workspace exceeds the caller's, and keeps the fastest.  Re-plans
// the problems (set-up, not per evaluation); synchronises the stream.
extern "C" kde_status kde_batch_tune(kde_batch_plan bp, const void* X, void* density,
                                     void* workspace, size_t workspace_bytes, kde_stream_t stream,
                                     int reps, float* best_ms) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (reps < 1) reps = 3;
  cudaStream_t st = (cudaStream_t)stream;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
    return fail(KDE_ERR_CUDA, "cudaEventCreate");
  struct Cfg {
    int pad, order, mode, tr, tc, queue;
  };
  std::vector<Cfg> cfgs;
  for (int pad : {KDE_BATCH_PAD_SMALLEST, KDE_BATCH_PAD_FEWEST_STAGES})
    for (int order : {0, 1}) {
      for (int qo : {KDE_BATCH_QUEUE_PROBLEMS, KDE_BATCH_QUEUE_STAGES})
        for (int t : {32, 64, 128}) cfgs.push_back({pad, order, KDE_BATCH_PERSISTENT, t, t, qo});
      for (int tr : {32, 64, 128})
        for (int tc : {32, 64, 128})
          cfgs.push_back({pad, order, KDE_BATCH_STAGED, tr, tc, bp->queue_order});
    }
  float best = 1e30f;
  Cfg bc = {bp->pad_policy, bp->radix_order, bp->mode, bp->tpl_rows, bp->tpl_cols, bp->queue_order};
  // workspaces of at least 64 MB serve as the L2 flush between reps
  const size_t flush_bytes =
      workspace_bytes >= ((size_t)64 << 20) ? std::min(workspace_bytes, (size_t)256 << 20) : 0;
  // the timed runs go on a stream of the tuner's own, after the caller's
  // stream has reached this call
  cudaStream_t cs = nullptr;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return fail(KDE_ERR_CUDA, "cudaStreamCreate");
  }
  cudaEventRecord(e0, st);
  cudaStreamWaitEvent(cs, e0, 0);
  kde_status s = KDE_OK;
  int cur_pad = bp->pad_policy, cur_order = bp->radix_order, cur_q = bp->queue_order;
  for (const Cfg& c : cfgs) {
    if (c.pad != cur_pad || c.order != cur_order || c.queue != cur_q) {
      bp->pad_policy = c.pad;
      bp->radix_order = c.order;
      bp->queue_order = c.queue;
      if ((s = kde::batch_rebuild(bp)) != KDE_OK) break;
      cur_pad = c.pad;
      cur_order = c.order;
      cur_q = c.queue;
    }
    if (bp->workspace_bytes > workspace_bytes) continue;
    bp->mode = c.mode;
    bp->tpl_rows = c.tr;
    bp->tpl_cols = c.tc;
    if ((s = kde_batch_eval(bp, X, density, workspace, workspace_bytes, (kde_stream_t)cs)) != KDE_OK)
      break;
    // the evaluation as it is used: captured once as a CUDA graph (no host
    // gaps between the staged launches), replayed reps times; before each
    // replay a workspace of L2's order of size is overwritten (it is
    // scratch) so that the replay starts with the caches cold, as a new
    // batch would.  Plain launches if the capture fails.
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      const kde_status sc = kde_batch_eval(bp, X, density, workspace, workspace_bytes, (kde_stream_t)cs);
      const cudaError_t ec = cudaStreamEndCapture(cs, &graph);
      if (sc != KDE_OK || ec != cudaSuccess ||
          cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        graph = nullptr;
        exec = nullptr;
        cudaGetLastError();   // a failed capture leaves no error behind
      }
    } else {
      cudaGetLastError();
    }
    float ms = 0.f;
    for (int r = 0; r < reps && s == KDE_OK; ++r) {
      if (flush_bytes) {
        cudaError_t e = cudaMemsetAsync(workspace, 0, flush_bytes, cs);
        if (e != cudaSuccess) {
          s = cuda_fail(e, "cudaMemsetAsync(workspace)");
          break;
        }
      }
      cudaEventRecord(e0, cs);
      if (exec) {
        const cudaError_t e = cudaGraphLaunch(exec, cs);
        if (e != cudaSuccess) s = cuda_fail(e, "cudaGraphLaunch(tuning run)");
      } else {
        s = kde_batch_eval(bp, X, density, workspace, workspace_bytes, (kde_stream_t)cs);
      }
      cudaEventRecord(e1, cs);
      if (s != KDE_OK) break;
      cudaError_t e = cudaEventSynchronize(e1);
      if (e != cudaSuccess) {
        s = cuda_fail(e, "tuning run");
        break;
      }
      float one = 0.f;
      cudaEventElapsedTime(&one, e0, e1);
      ms += one;
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (s != KDE_OK) break;
    ms /= reps;
    if (ms < best) {
      best = ms;
      bc = c;
    }
  }
  cudaStreamSynchronize(cs);
  cudaStreamDestroy(cs);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (s != KDE_OK) return s;
  if (bc.pad != cur_pad || bc.order != cur_order || bc.queue != cur_q) {
    bp->pad_policy = bc.pad;
    bp->radix_order = bc.order;
    bp->queue_order = bc.queue;
    if ((s = kde::batch_rebuild(bp)) != KDE_OK) return s;
  }
  bp->mode = bc.mode;
  bp->tpl_rows = bc.tr;
  bp->tpl_cols = bc.tc;
  if (best_ms) *best_ms = best;
  if ((s = kde_batch_check(bp, stream)) != KDE_OK) return s;
  return KDE_OK;
}

extern "C" kde_status kde_batch_set_queue_order(kde_batch_plan bp, int order) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (order != KDE_BATCH_QUEUE_STAGES && order != KDE_BATCH_QUEUE_PROBLEMS)
    return fail(KDE_ERR_INVALID_ARG, "order: KDE_BATCH_QUEUE_STAGES or KDE_BATCH_QUEUE_PROBLEMS");
  bp->queue_order = order;
  return kde::batch_work(bp);
}

extern "C" kde_status kde_batch_get_config(kde_batch_plan bp, int* pad_policy, int* radix_order,
                                           int64_t* P) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (pad_policy) *pad_policy = bp->pad_policy;
  if (radix_order) *radix_order = bp->radix_order | (bp->queue_order << 8);
  if (P)
    for (int i = 0; i < bp->count; ++i)
      for (int k = 0; k < 2; ++k) P[2 * i + k] = bp->plans[i]->info.P[k];
  return KDE_OK;
}

extern "C" kde_status kde_batch_get_shape(kde_batch_plan bp, int* tpl_rows, int* tpl_cols) {
  if (!bp) return fail(KDE_ERR_INVALID_ARG, "NULL plan");
  if (tpl_rows) *tpl_rows = bp->tpl_rows;
  if (tpl_cols) *tpl_cols = bp->tpl_cols;
  return KDE_OK;
}

KDE_DEBUG_READER(eval)
