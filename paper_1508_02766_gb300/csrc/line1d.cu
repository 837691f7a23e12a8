// One-dimensional problems (d = 1): the whole transform is one line, which a
// single block would work on alone.
//
// kde_line1d_kgen_kernel: the kernel spectrum as the cosine sum
//   K_q = k_0 + 2 sum_{l=1}^{L} k_l cos(2 pi q l / P)
// (k is real and even), a block for 32 frequencies.  It replaces one block's
// L + 1 exponentials and length-P transform: the sums are (L + 1) Q terms in
// all, spread over the chip, and each block repeats only the exponentials.
//
// kde_line1d_cluster_kernel: counts -> F -> x K -> F^-1 -> crop on one
// cluster of kC blocks.  P = N1 N2 as a matrix of N1 rows: columns
// x[n2 + N2 n1] (transformed over n1 in real pairs), then rows over n2, then
// K, and back.  Counts and density are real, so rows k1 and N1 - k1 are
// conjugates and only rows 0 .. N1/2 are transformed: half the arithmetic of
// the complex line, on kC SMs instead of one.  The two transposes are stores
// into the shared memory of the block that owns the row or column pair
// (distributed shared memory), each ended by a cluster barrier.
//
// What bounds them: FP64 runs at 2 lanes a clock and SM, and one SM took 72
// (evaluation) and 41 us (spectrum) for P = 2100, L = 81 in FP64 (event
// times); now 27 and 8, the latency of about ten short dependent stages and
// a launch.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "fft_engine.cuh"
#include "kde_internal.h"
#include "kgen.cuh"
#include "pdl.cuh"

namespace kde {
namespace {

namespace cg = cooperative_groups;

constexpr int kC = 8;           // blocks per cluster (16 measured level: the stages' latency, not FP64 issue, is left)
constexpr int kThreads = 256;
constexpr int kQ = 32;          // frequencies per block of the spectrum kernel

// Radix plan of one factor; twstep counts in steps of the length-P table.
struct SubPlan {
  int N, nst;
  Stage st[KDE_MAX_STAGES];
};

struct LineArgs {
  int P, M, N1, N2;
  int np;          // column pairs, ceil(N2 / 2)
  int nlA, nlB;    // column pairs and rows per block
  SubPlan a, b;    // length N1 and N2
};

// One stage of nl lines of s.nb butterflies each, line i at i ld, spread
// over the whole block.
template <typename V, int R, bool INV>
__device__ __forceinline__ void batch_stage(const V* in, V* out, int nl, int ld, const Stage& s,
                                            const V* tw) {
  for (int i = threadIdx.x; i < nl * s.nb; i += kThreads) {
    const int li = i / s.nb, j = i - li * s.nb;
    const V* src = in + li * ld;
    V x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = src[j + r * s.nb];
    int base = j * R;
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
    }
    SmallDFT<V, R, INV>::run(x);
    V* dst = out + li * ld + base;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r * s.Ns] = x[r];
  }
}

// All stages of nl lines in a (scratch b); returns the buffer of the result.
// Callers synchronise before; ends synchronised.
template <typename V, bool INV>
__device__ V* batch_fft(V* a, V* b, int nl, int ld, const SubPlan& p, const V* tw) {
  for (int s = 0; s < p.nst; ++s) {
    const Stage& st = p.st[s];
    switch (st.R) {
      case 2: batch_stage<V, 2, INV>(a, b, nl, ld, st, tw); break;
      case 3: batch_stage<V, 3, INV>(a, b, nl, ld, st, tw); break;
      case 4: batch_stage<V, 4, INV>(a, b, nl, ld, st, tw); break;
      case 5: batch_stage<V, 5, INV>(a, b, nl, ld, st, tw); break;
      case 7: batch_stage<V, 7, INV>(a, b, nl, ld, st, tw); break;
      default: batch_stage<V, 8, INV>(a, b, nl, ld, st, tw); break;
    }
    __syncthreads();
    V* t = a;
    a = b;
    b = t;
  }
  return a;
}

template <typename T>
__global__ void __launch_bounds__(kThreads)
kde_line1d_cluster_kernel(const long long* __restrict__ counts, const T* __restrict__ K,
                          T* __restrict__ out, LineArgs g,
                          const typename Cplx<T>::type* __restrict__ twg) {
  using V = typename Cplx<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x;
  const int N1 = g.N1, N2 = g.N2, H1 = N1 / 2 + 1, ldA = 2 * H1;  // ldA >= N1
  V* tw = reinterpret_cast<V*>(smem_raw);
  V* a = tw + g.P;             // column pairs [nlA][ldA]
  V* b = a + g.nlA * ldA;
  V* c = b + g.nlA * ldA;      // rows [nlB][N2]
  V* d = c + g.nlB * N2;
#pragma unroll 8
  for (int i = tid; i < g.P; i += kThreads) tw[i] = __ldg(twg + i);
  // counts and K are written by the kernels before this one
  pdl_trigger();
  pdl_wait();
  const int p0 = rank * g.nlA, npl = max(0, min(g.nlA, g.np - p0));
  const int r0 = rank * g.nlB, nrl = max(0, min(g.nlB, H1 - r0));
  for (int i = tid; i < npl * N1; i += kThreads) {
    const int n1 = i / npl, li = i - n1 * npl;
    const int col = 2 * (p0 + li), pos = col + N2 * n1;
    const T x0 = pos < g.M ? count_value<T>(counts[pos]) : T(0);
    const T x1 = (col + 1 < N2 && pos + 1 < g.M) ? count_value<T>(counts[pos + 1]) : T(0);
    a[li * ldA + n1] = mk<V>(x0, x1);
  }
  // every block of the cluster runs before any stores into its shared memory
  cl.sync();
  {
    const V* z = batch_fft<V, false>(a, b, npl, ldA, g.a, tw);
    for (int i = tid; i < npl * H1; i += kThreads) {
      const int li = i / H1, k1 = i - li * H1, n2 = 2 * (p0 + li);
      const V zk = z[li * ldA + k1], zm = z[li * ldA + (k1 ? N1 - k1 : 0)];
      const V X = mk<V>(T(0.5) * (zk.x + zm.x), T(0.5) * (zk.y - zm.y));
      const V Y = mk<V>(T(0.5) * (zk.y + zm.y), T(-0.5) * (zk.x - zm.x));
      const int owner = k1 / g.nlB;
      V* dst = cl.map_shared_rank(c, owner) + (k1 - owner * g.nlB) * N2 + n2;
      dst[0] = cmul(X, tw[n2 * k1]);
      if (n2 + 1 < N2) dst[1] = cmul(Y, tw[(n2 + 1) * k1]);
    }
  }
  cl.sync();
  {
    V* z = batch_fft<V, false>(c, d, nrl, N2, g.b, tw);
    for (int i = tid; i < nrl * N2; i += kThreads) {
      const int r = i / N2, k2 = i - r * N2, k = r0 + r + N1 * k2;
      const T kv = __ldg(K + (2 * k <= g.P ? k : g.P - k));
      z[i] = mk<V>(z[i].x * kv, z[i].y * kv);
    }
    __syncthreads();
    V* other = z == c ? d : c;
    const V* y = batch_fft<V, true>(z, other, nrl, N2, g.b, tw);
    for (int i = tid; i < nrl * N2; i += kThreads) {
      const int r = i / N2, n2 = i - r * N2, k1 = r0 + r, p = n2 >> 1, owner = p / g.nlA;
      V* dst = cl.map_shared_rank(a, owner) + (p - owner * g.nlA) * ldA + (n2 & 1) * H1 + k1;
      *dst = cmul(y[i], cconj(tw[n2 * k1]));
    }
  }
  cl.sync();
  // the pair's full lines from rows 0 .. N1/2 (the rest are conjugates)
  for (int i = tid; i < npl * N1; i += kThreads) {
    const int li = i / N1, k = i - li * N1;
    const bool lo = k < H1;
    const V* src = a + li * ldA + (lo ? k : N1 - k);
    const V Y0 = src[0], Y1 = 2 * (p0 + li) + 1 < N2 ? src[H1] : mk<V>(0, 0);
    b[li * ldA + k] = lo ? mk<V>(Y0.x - Y1.y, Y0.y + Y1.x) : mk<V>(Y0.x + Y1.y, Y1.x - Y0.y);
  }
  __syncthreads();
  const V* z = batch_fft<V, true>(b, a, npl, ldA, g.a, tw);
  for (int i = tid; i < npl * N1; i += kThreads) {
    const int n1 = i / npl, li = i - n1 * npl;
    const int col = 2 * (p0 + li), pos = col + N2 * n1;
    const V v = z[li * ldA + n1];
    if (pos < g.M) out[pos] = v.x;
    if (col + 1 < N2 && pos + 1 < g.M) out[pos + 1] = v.y;
  }
}

// Warp w of a block takes the lags l = 1 + w (mod 8) of frequencies
// q0 .. q0 + 31, one per lane; the eight sums are added in a fixed order.
template <typename T>
__global__ void __launch_bounds__(kThreads)
kde_line1d_kgen_kernel(KGen<T> gen, T* __restrict__ Kspec, int P,
                       const typename Cplx<T>::type* __restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int L = gen.L[0], Q = P / 2 + 1, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  T* cs = reinterpret_cast<T*>(smem_raw);   // cos(2 pi m / P), m <= P/2
  T* kv = cs + Q;                           // k_l, l <= L
  T* part = kv + L + 1;                     // [8][32]
  pdl_trigger();
  for (int m = tid; m < Q; m += kThreads) cs[m] = __ldg(&tw[m].x);
  for (int l = tid; l <= L; l += kThreads) {
    const int lag[KDE_MAX_D] = {l, 0, 0};
    kv[l] = kernel_value<T>(gen, lag);
  }
  __syncthreads();
  const int q = blockIdx.x * kQ + lane;
  T s = 0, e = 0;
  if (q < Q) {
    int m = (int)((int64_t)q * (w + 1) % P);
    const int step = (int)((int64_t)q * 8 % P);
    for (int l = w + 1; l <= L; l += 8) {
      const T c = cs[2 * m <= P ? m : P - m];
      if (sizeof(T) == 4) {   // Kahan: FP32 sums of many terms lose digits the transform keeps
        const T y = fma(kv[l], c, -e), t = s + y;
        e = (t - s) - y;
        s = t;
      } else {
        s = fma(kv[l], c, s);
      }
      m += step;
      if (m >= P) m -= P;
    }
  }
  part[tid] = s;
  __syncthreads();
  // Kspec may still be read by the kernels before this one
  pdl_wait();
  if (w == 0 && q < Q) {
    T t = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) t += part[i * 32 + lane];
    Kspec[q] = kv[0] + T(2) * t;
  }
}

SubPlan sub_plan(const int* radix, int nst, int N, int P) {
  SubPlan p{};
  p.N = N;
  p.nst = nst;
  int Ns = 1;
  for (int s = 0; s < nst; ++s) {
    Stage& st = p.st[s];
    st.R = radix[s];
    st.Ns = Ns;
    st.nb = N / st.R;
    st.twstep = P / (Ns * st.R);
    st.magic = (unsigned)((1ull << 32) / (unsigned)Ns + 1ull);
    Ns *= st.R;
  }
  return p;
}

// The split of the plan's radices whose products are nearest each other.
bool split_line(const kde_plan_info& I, LineArgs* g) {
  const int P = (int)I.P[0], n = I.nstages[0];
  int best = 0;
  double best_r = 0.0;
  for (int mask = 1; mask < (1 << n) - 1; ++mask) {
    int N1 = 1;
    for (int s = 0; s < n; ++s)
      if ((mask >> s) & 1) N1 *= I.radix[0][s];
    const double r = (double)std::min(N1, P / N1) / (double)std::max(N1, P / N1);
    if (r > best_r) {
      best_r = r;
      best = mask;
    }
  }
  if (!best) return false;
  int ra[KDE_MAX_STAGES], rb[KDE_MAX_STAGES], na = 0, nb = 0;
  g->N1 = 1;
  for (int s = 0; s < n; ++s) {
    if ((best >> s) & 1) {
      ra[na++] = I.radix[0][s];
      g->N1 *= I.radix[0][s];
    } else {
      rb[nb++] = I.radix[0][s];
    }
  }
  g->P = P;
  g->M = (int)I.M[0];
  g->N2 = P / g->N1;
  g->np = (g->N2 + 1) / 2;
  g->nlA = (g->np + kC - 1) / kC;
  g->nlB = (g->N1 / 2 + 1 + kC - 1) / kC;
  g->a = sub_plan(ra, na, g->N1, P);
  g->b = sub_plan(rb, nb, g->N2, P);
  return true;
}

template <typename T>
const typename Cplx<T>::type* table(const kde_plan_s* plan) {
  return reinterpret_cast<const typename Cplx<T>::type*>((const char*)plan->tw_dev + plan->tw_offset[0]);
}

// Shortest line for the cluster.  One block against the cluster (us, graph of
// ten, GB300): FP64 P = 420 16.6 / 17.2, 525 19.5 / 18.9, 810 32 / 17,
// 2160 67 / 20, 4032 118 / 26; FP32 P = 480 4.5 / 6.4, 1050 6.6 / 7.0,
// 1536 7.0 / 7.0, 2160 10.5 / 7.9, 4032 13.5 / 8.4 (three cluster barriers
// and the two transposes are about 5 us of it).
template <typename T>
constexpr int min_line() { return sizeof(T) == 8 ? 512 : 1536; }
// Widest support of the cosine sums.  Their terms grow with L, the transform's
// do not, but the two do not meet: transform against sums (us) FP64 L = 20 34 /
// 1.4 (P = 2025), L = 600 52 / 3.5 (P = 2625), L = 1025 47 / 7.4 (P = 2560), L =
// 2039 70 / 18 (P = 4096); FP32 6.2 / 1.0, 7.0 / 1.2, 7.4 / 2.5, 11.1 / 4.9.  The
// line is where the FP32 sums' error has been held against the transform's
// (level, over drawn cases); above it single supports went either way (4.1e-8 /
// 7.0e-8 at L = 1700, 5.9e-8 / 2.5e-8 at 2039).
constexpr int kMaxLags = 1024;

}  // namespace

// The cluster evaluation of a d = 1 plan; *taken = false (nothing launched)
// for lines shorter than min_line or without two factors, which the one-block
// kernel takes.
template <typename T>
kde_status line1d_eval(const kde_plan_s* plan, const long long* counts, const T* K, T* density,
                       cudaStream_t st, bool* taken) {
  using V = typename Cplx<T>::type;
  LineArgs g{};
  *taken = plan->info.P[0] >= min_line<T>() && split_line(plan->info, &g);
  if (!*taken) return KDE_OK;
  const size_t smem = sizeof(V) * ((size_t)g.P + 2 * (size_t)g.nlA * 2 * (g.N1 / 2 + 1) +
                                   2 * (size_t)g.nlB * g.N2);
  auto* fn = kde_line1d_cluster_kernel<T>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kC);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kC;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  LaunchScope ls("kde_line1d_cluster_kernel", st);
  e = cudaLaunchKernelEx(&cfg, fn, counts, K, density, g, table<T>(plan));
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_line1d_cluster_kernel");
}

// The cosine-sum spectrum of a d = 1 plan; *taken = false for supports above
// kMaxLags.
template <typename T>
kde_status line1d_kernel_grid(const kde_plan_s* plan, const KGen<T>& gen, T* Kspec,
                              cudaStream_t st, bool* taken) {
  const int P = (int)plan->info.P[0], Q = P / 2 + 1;
  *taken = gen.L[0] <= kMaxLags;
  if (!*taken) return KDE_OK;
  const size_t smem = sizeof(T) * ((size_t)Q + gen.L[0] + 1 + kThreads);
  LaunchScope ls("kde_line1d_kgen_kernel", st);
  cudaError_t e = launch_pdl(kde_line1d_kgen_kernel<T>, dim3((Q + kQ - 1) / kQ), dim3(kThreads),
                             smem, st, gen, Kspec, P, table<T>(plan));
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? KDE_OK : cuda_fail(e, "kde_line1d_kgen_kernel");
}

template kde_status line1d_eval<float>(const kde_plan_s*, const long long*, const float*, float*,
                                       cudaStream_t, bool*);
template kde_status line1d_eval<double>(const kde_plan_s*, const long long*, const double*, double*,
                                        cudaStream_t, bool*);
template kde_status line1d_kernel_grid<float>(const kde_plan_s*, const KGen<float>&, float*,
                                              cudaStream_t, bool*);
template kde_status line1d_kernel_grid<double>(const kde_plan_s*, const KGen<double>&, double*,
                                               cudaStream_t, bool*);

}  // namespace kde
