// mgr_rows.h -- element offsets of a strip's rows within a plane.  Plain C++ for
// host and device.
#pragma once

#ifdef __CUDACC__
#define MGR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MGR_HOST_DEVICE inline
#endif

namespace mgr {

// Row i of a level whose rows lie s apart on an axis of N rows of `pitch` elements sits
// at row min(i * s, N - 1).  Walks the coarse rows i = 2 qc of a strip, and with each the
// fine row 2 qc - 1 above it, from one before the strip's first.
//
// Offsets are unsigned and unclamped until they are used: a plane has fewer than 2^31
// elements, and a coarse row of the level has i * s < 2 (N - 1), hence an offset below
// 2^32, where 31 bits would not do (514 rows of 2097152: row 4 of the level of rows 256
// apart is row 513, and 4 * 256 * 2097152 = 2^31).  Past the end of the axis the offset
// may wrap; what is returned lies within the plane all the same.
// (Row indices clamped before a product with the pitch, for every row: the FP32 passes
// took 1 to 3% longer.)
struct StripRows {
  unsigned at, second, half, last;
  MGR_HOST_DEVICE StripRows(int first, int s, int N, int pitch) {
    half = unsigned(s) * unsigned(pitch);
    last = unsigned(N - 1) * unsigned(pitch);
    second = 2u * unsigned(first) * half;
    restart();
  }
  MGR_HOST_DEVICE int coarse() const { return int(at < last ? at : last); }
  // Where the row before the axis is read, as row 0.
  MGR_HOST_DEVICE void restart() { at = second == 0 ? 0u : second - 2u * half; }
  MGR_HOST_DEVICE void next(bool start) { at = start ? second : at + 2u * half; }  // start: from the first one
  MGR_HOST_DEVICE int fine() const {
    const unsigned f = (at > half ? at : half) - half;
    return int(f < last ? f : last);
  }
  // Where only rows of the level are used: before the axis the offset wraps.
  MGR_HOST_DEVICE void rewind() { at = second - 2u * half; }
  MGR_HOST_DEVICE void advance() { at += 2u * half; }
  MGR_HOST_DEVICE int above() const { return int(at - half < last ? at - half : last); }
};

}  // namespace mgr
