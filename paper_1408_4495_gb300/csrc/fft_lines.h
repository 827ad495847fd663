// Plan of the half-length line transforms (fft_lines.cuh), shared by the kernels (device) and the
// construction of their twiddle tables (host).
//
// A line of length L (2^k or 3 * 2^k) is split into two or three factors, and each thread holds E
// of its values in registers from the first butterfly to the last: between two factors the
// values change hands through shared memory once.  Large radices keep these exchanges few (the
// passes are bound by shared-memory traffic and instruction issue long before HBM): 16 x 16 x 8
// for L = 2048 exchanges twice per transform, against three times and twice the barriers for
// radix 8.  The inverse transform takes the factors in reverse order, so that it starts from the
// registers in which the forward one ends.
//
// The factor pass that starts from sub-transforms of length N (N = L first, N / R after radix R)
// multiplies output k of butterfly j (0 <= k < R, 0 <= j < N / R) by exp(-+2 pi i j k / N).  The
// table holds these factors pass after pass (all but the last), output after output, butterfly
// after butterfly: neighbouring threads read neighbouring entries.  Forward table first, then
// the inverse one.
#pragma once

#if defined(__CUDACC__)
#define LS_FL_HD __host__ __device__
#else
#define LS_FL_HD
#endif

namespace ls {

struct LinePlan {
  int nf;    // factors
  int r[3];  // radices of the forward transform
  int e;     // values per thread
};

// wide: 16-byte values (float-float, FP64) take radix 16 at most (32 values would fill 128 registers)
LS_FL_HD constexpr LinePlan line_plan(int L, bool wide) {
  return L == 16     ? LinePlan{2, {4, 4, 1}, 4}
         : L == 32   ? LinePlan{2, {8, 4, 1}, 8}
         : L == 48   ? LinePlan{2, {12, 4, 1}, 12}
         : L == 64   ? LinePlan{2, {8, 8, 1}, 8}
         : L == 96   ? (wide ? LinePlan{3, {4, 4, 6}, 12} : LinePlan{2, {12, 8, 1}, 24})
         : L == 128  ? LinePlan{2, {16, 8, 1}, 16}
         : L == 256  ? LinePlan{2, {16, 16, 1}, 16}
         : L == 512  ? (wide ? LinePlan{3, {8, 8, 8}, 8} : LinePlan{2, {32, 16, 1}, 32})
         : L == 1024 ? (wide ? LinePlan{3, {16, 8, 8}, 16} : LinePlan{2, {32, 32, 1}, 32})
         : L == 2048 ? LinePlan{3, {16, 16, 8}, 16}
         : L == 4096 ? LinePlan{3, {16, 16, 16}, 16}
                     : LinePlan{0, {1, 1, 1}, 1};
}
// radix of pass p (0, 1, ..) of the forward (inv false) or inverse transform; 1 past the last
LS_FL_HD constexpr int line_radix(int L, bool wide, bool inv, int p) {
  const LinePlan q = line_plan(L, wide);
  return p >= q.nf ? 1 : q.r[inv ? q.nf - 1 - p : p];
}
// entries of one direction's table, and of the whole one
LS_FL_HD constexpr int line_tw_dir(int L, bool wide, bool inv) {
  return line_plan(L, wide).nf == 3 ? L + L / line_radix(L, wide, inv, 0) : L;
}
LS_FL_HD constexpr int line_tw_size(int L, bool wide) {
  return line_tw_dir(L, wide, false) + line_tw_dir(L, wide, true);
}

}  // namespace ls
