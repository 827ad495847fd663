// Passes of the far-field sum (farfield.cu) over the observation directions, and their scratch:
// host arithmetic shared by the launches and their test.
#pragma once
#include <algorithm>
#include <cstddef>

namespace ls {

constexpr int FL = 16;  // grid lines (last axis) per CTA

inline int far_tiles(int d, int n) { return (int)(((d == 2 ? (long)n : (long)n * n) + FL - 1) / FL); }

// complex scratch entries of one direction: its partial sums and its columns of the two tables
inline long far_dir_elems(int d, int n, int nrhs) {
  return (long)nrhs * far_tiles(d, n) + (long)(d - 1) * n + n / 2;
}

// Directions per pass: their scratch stays below 256 MB (64 directions at least).  A direction takes
// 24 entries and more on every grid, so a pass has at most 43 690 tiles of 16 directions: they fit
// gridDim.z.
inline int far_chunk(int d, int n, int nrhs, int nobs) {
  const long most = (16L << 20) / far_dir_elems(d, n, nrhs) / 64 * 64;
  return (int)std::min<long>(nobs, std::max<long>(64, most));
}

// complex entries of the tables and the partial sums
inline size_t far_scratch_elems(int d, int n, int nrhs, int nobs) {
  return (size_t)nrhs * d * n + (size_t)far_dir_elems(d, n, nrhs) * far_chunk(d, n, nrhs, nobs);
}

}  // namespace ls
