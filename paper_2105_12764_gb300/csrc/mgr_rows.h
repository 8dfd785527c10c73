// mgr_rows.h -- element offset of a row of a level grid within its plane.
// Plain C++ for host and device.
#pragma once

#ifdef __CUDACC__
#define MGR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MGR_HOST_DEVICE inline
#endif

namespace mgr {

// Offset of row i of a level with n rows, s apart on an axis of N rows of `pitch`
// elements: row i sits at min(i * s, N - 1), rows outside the level are read as its
// first or last.  The row is clamped before the product with the pitch: a plane has
// fewer than 2^31 elements, but the last coarse row's i * s may reach nearly 2 N
// (514 rows of 2097152: row 2 * 2 of the level of 4 rows 256 apart is row 513, and
// 4 * 256 * 2097152 = 2^31).  i * s itself stays below 2^31 (N <= 2^30).
MGR_HOST_DEVICE int level_row_offset(int i, int n, int s, int N, int pitch) {
  const int level_row = i < 0 ? 0 : i < n ? i : n - 1;
  const int row = level_row * s;
  return (row < N ? row : N - 1) * pitch;
}

}  // namespace mgr
