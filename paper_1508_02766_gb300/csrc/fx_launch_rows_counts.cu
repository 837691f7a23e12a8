// Two-phase engine: launcher of one pass (its own translation unit so that
// the passes compile in parallel).
#include "fx3_kernels.cuh"

namespace kde {
namespace fx {

cudaError_t launch_rows_counts(const Launch& l, const RowsArgs& a, const long long* counts) {
#define KDE_FX_KERNEL(n1, n2) kde_fx_rows_fwd_kernel<0, n1, n2, SRC_COUNTS>
#define KDE_FX_CASE_PAIR(n1, n2) \
  case n1 * 64 + n2:             \
    return launch_kernel(KDE_FX_KERNEL(n1, n2), l.grid, l.threads, l.smem, l.st, a, counts, KGen<float>{});
#define KDE_FX_CASE_TRIPLE(n1, n2, n3)  \
  case n1 * 4096 + n2 * 64 + n3:       \
    return launch_kernel(kde_fx3_rows_fwd_kernel<n1, n2, n3, SRC_COUNTS, false>, l.grid, l.threads, l.smem, l.st, a, counts, KGen<float>{});
#define KDE_FX_CASE_WIDE(n1, n2, n3)  \
  case n1 * 4096 + n2 * 64 + n3:       \
    return launch_kernel(kde_fx3_rows_fwd_kernel<n1, n2, n3, SRC_COUNTS, true>, l.grid, l.threads, l.smem, l.st, a, counts, KGen<float>{});
  KDE_FX_DISPATCH(KDE_FX_KERNEL, a, counts, KGen<float>{})
#undef KDE_FX_CASE_WIDE
#undef KDE_FX_CASE_TRIPLE
#undef KDE_FX_CASE_PAIR
#undef KDE_FX_KERNEL
}

}  // namespace fx
}  // namespace kde

KDE_DEBUG_READER(fx_rows_counts)
