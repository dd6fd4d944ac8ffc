// Index checks of the QG_CHECK_BOUNDS build: qg_at compares an element's address with the registered device
// arrays (bounds_register); a miss records the first bad source line and address and reads or writes a dummy
// word instead.  The build step turns every d.<array>[i] of qg_kernels.cu into it; other accesses through a
// pointer are written QG_AT(p, i), plain p[i] in the normal build.  Every translation unit has a table of
// its own.
#pragma once

#ifdef QG_CHECK_BOUNDS
#include <cuda_runtime.h>

namespace qg {

constexpr int QG_MAX_RANGES = 8192;
struct QgRange {
  unsigned long long lo, hi;  // [lo, hi)
};

namespace {

__device__ QgRange g_qg_ranges[QG_MAX_RANGES];  // sorted by lo, disjoint
__device__ int g_qg_nranges;
__device__ int g_qg_bad_line;                 // first failing access: its source line (0: none)
__device__ unsigned long long g_qg_bad_addr;  // and its address
__device__ __align__(16) unsigned char g_qg_dummy[64];

template <typename T>
__device__ __forceinline__ T &qg_at(T *p, long long i, int line) {
  const unsigned long long a = reinterpret_cast<unsigned long long>(p + i);
  int lo = 0, hi = g_qg_nranges - 1;
  while (lo <= hi) {  // the last range starting at or below a
    const int mid = (lo + hi) >> 1;
    if (g_qg_ranges[mid].lo <= a) lo = mid + 1;
    else hi = mid - 1;
  }
  if (hi >= 0 && a + sizeof(T) <= g_qg_ranges[hi].hi) return p[i];
  if (atomicCAS(&g_qg_bad_line, 0, line) == 0) g_qg_bad_addr = a;
  return *reinterpret_cast<T *>(g_qg_dummy);
}

// This translation unit's table, and its first miss (line 0: none).
inline void check_upload(const QgRange *v, int n) {
  if (n) cudaMemcpyToSymbol(g_qg_ranges, v, sizeof(QgRange) * n);
  cudaMemcpyToSymbol(g_qg_nranges, &n, sizeof(int));
}
inline void check_first(int *line, unsigned long long *addr) {
  cudaMemcpyFromSymbol(line, g_qg_bad_line, sizeof(int));
  cudaMemcpyFromSymbol(addr, g_qg_bad_addr, sizeof(*addr));
}

}  // namespace
}  // namespace qg

#define QG_AT(p, i) qg::qg_at((p), (long long)(i), __LINE__)
#else
#define QG_AT(p, i) (p)[i]
#endif
