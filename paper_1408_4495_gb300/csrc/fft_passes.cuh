// Kernels and launchers of the operator's FFT passes: half-length line transforms (n of L = 2n
// entries in or out) with the pad, the omega^2 m scale, the symbol multiply, the crop and the "+u"
// fused in.  The operator-level sequence that chains them is in fft.cu; each arithmetic (FP32,
// FP64, float-float) instantiates the passes in its own translation units (fft_pass_*.cu) so that
// they compile in parallel.
//
// A pass keeps its lines in registers (fft_lines.cuh): global memory to registers, two or three
// factors with one shared-memory exchange between them, registers to global memory; the symbol
// pass multiplies the spectrum in the registers where the forward transform leaves it and the
// inverse one begins.  Against Stockham passes of radix 8 that went through shared memory at every
// pass (16 store-and-load rounds with two barriers each in the L = 2048 symbol pass, now 4 with
// one): FP32, 2D n = 512, 16 vectors: rows forward / symbol / rows inverse 53 / 149 / 61 us -> 20
// / 61 / 25 us; n = 1024, 64 vectors: symbol pass 2.23 -> 1.39 ms; float-float 8.0 -> 5.0 ms.  What
// bounds them (counters at 2D n = 1024, 16 vectors): FP32 the path to L1 and shared memory (79 %
// busy, 1.4 TB/s through the symbol pass; the row passes 75 and 83 % of the memory bandwidth), float-float
// the FP32 pipe (81 % active in the symbol pass: 418 instructions a point of the padded grid, additions of 8 packed
// ones a complex number), FP64 its pipe (85 % active at n = 256).
#pragma once

#include <atomic>
#include <string>
#include <type_traits>

#include "common.cuh"
#include "fft_lines.cuh"
#include "kernels.h"
#include "pdl.cuh"
#include "prof.h"

namespace ls {

// kernel-class names of the three arithmetics
template <typename C> constexpr const char* arith_tag();
template <> constexpr const char* arith_tag<float2>() { return "c64"; }
template <> constexpr const char* arith_tag<double2>() { return "c128"; }
template <> constexpr const char* arith_tag<ffp>() { return "cff"; }

template <typename C> __device__ __forceinline__ C l_of_f64(double2 v);
template <> __device__ __forceinline__ float2 l_of_f64<float2>(double2 v) { return make_float2((float)v.x, (float)v.y); }
template <> __device__ __forceinline__ double2 l_of_f64<double2>(double2 v) { return v; }
template <> __device__ __forceinline__ ffp l_of_f64<ffp>(double2 v) { return ffp_of_f64(v); }
__device__ __forceinline__ double2 l_to_f64(double2 v) { return v; }
__device__ __forceinline__ double2 l_to_f64(ffp v) { return ffp_to_f64(v); }
// a times entry i of the real weights (float-float: one pair per weight)
__device__ __forceinline__ float2 l_weight(float2 a, const void* w, long i) {
  const float x = __ldg(static_cast<const float*>(w) + i);
  return make_float2(a.x * x, a.y * x);
}
__device__ __forceinline__ double2 l_weight(double2 a, const void* w, long i) {
  const double x = __ldg(static_cast<const double*>(w) + i);
  return make_double2(a.x * x, a.y * x);
}
__device__ __forceinline__ ffp l_weight(ffp a, const void* w, long i) {
  const float2 x = __ldg(static_cast<const float2*>(w) + i);
  return l_norm(l_mulr(a, ff(x.x, x.y)));
}

// ------------------------------------------------------------------------------------
// Row passes: lines contiguous in memory, T threads per line (one warp or less for L <= 1024 in
// FP32 and L <= 256 otherwise, which then needs no block barrier).
// ------------------------------------------------------------------------------------
template <typename C, int L> struct RowShape {
  using LAY = LineLay<C, L, 0>;
  // FP64 is bound by its pipe (two lanes an SM): small CTAs spread a small batch over more SMs
  static constexpr int NT0 = std::is_same<C, double2>::value ? 64 : 128;
  static constexpr int NT = LAY::T > NT0 ? LAY::T : NT0;
  static constexpr int NL = NT / LAY::T;
  static constexpr bool WARP = LAY::T <= 32;
  // registers per thread: 32 of values leave room in 64 (float-float temporaries take 80)
  static constexpr int REGS = LAY::E * (int)sizeof(C) / 4 > 32 ? 128 : (std::is_same<C, ffp>::value ? 80 : 64);
  static constexpr int MINB = 65536 / (NT * REGS);
  static constexpr size_t SMEM = (size_t)NL * LAY::LS * sizeof(C);
};

enum { ROW_IN_C = 0, ROW_IN_F64 = 1, ROW_IN_WAVE = 2 };

// forward: n entries of each line (IN: in the passes' arithmetic, FP64, or the plane wave
// -omega^2 m exp(i omega x . dir) from its per-axis phase tables), scaled by the weights, to the L
// entries of its transform
template <typename C, int L, int IN>
__global__ void __launch_bounds__(RowShape<C, L>::NT, RowShape<C, L>::MINB) k_row_fwd(RowPassArgs a) {
  using SH = RowShape<C, L>;
  using LAY = typename SH::LAY;
  constexpr int E = LAY::E, T = LAY::T, n = L / 2;
  constexpr int R1 = line_radix(L, LAY::WIDE, false, 0), RL = line_radix(L, LAY::WIDE, false, LAY::P.nf - 1);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int li = threadIdx.x / T, t = threadIdx.x - li * T;
  const long line = (long)blockIdx.x * SH::NL + li;
  const bool valid = line < a.lines;
  C v[E];
  if (valid) {
    const long row = line % a.pw_lines;  // row of the weights (the line within its grid)
    C px = czero_l<C>();
    const C* pl = nullptr;
    if constexpr (IN == ROW_IN_WAVE) {
      const C* ph = static_cast<const C*>(a.phase) + (line / a.pw_lines) * a.d * n;
      pl = ph + (a.d - 1) * n;
      if (a.d == 2) px = l_neg(l_ldg(ph + row));
      else px = l_neg(l_norm(l_mul(l_ldg(ph + row / n), l_ldg(ph + n + row % n))));
    }
#pragma unroll
    for (int m = 0; m < E / R1; ++m)
#pragma unroll
      for (int r = 0; r < R1 / 2; ++r) {
        const int e = t + m * T + r * (L / R1);
        C x;
        if constexpr (IN == ROW_IN_WAVE) x = l_norm(l_mul(px, l_ldg(pl + e)));
        else if constexpr (IN == ROW_IN_F64) x = l_of_f64<C>(static_cast<const double2*>(a.in)[line * a.in_ls + e]);
        else x = static_cast<const C*>(a.in)[line * a.in_ls + e];
        v[m * R1 + r] = l_weight(x, a.pw, row * n + e);
      }
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = czero_l<C>();
  }
  line_fft<C, L, -1, true, false, SH::WARP, LAY>(v, reinterpret_cast<C*>(smem_raw) + li * LAY::LS,
                                                 static_cast<const C*>(a.tw), t);
  pdl_trigger_small();
  if (!valid) return;
  C* out = static_cast<C*>(a.out) + line * a.out_ls;
#pragma unroll
  for (int m = 0; m < E / RL; ++m)
#pragma unroll
    for (int r = 0; r < RL; ++r) out[t + m * T + r * (L / RL)] = l_norm(v[m * RL + r]);
}

// inverse: L entries of each line to the first n of its transform, + addv, subtracted from subv.
// OUT64: addv, subv and out are FP64 (FP32 arithmetic: addv is rounded to FP32 first)
template <typename C, int L, bool OUT64>
__global__ void __launch_bounds__(RowShape<C, L>::NT, RowShape<C, L>::MINB) k_row_inv(RowPassArgs a) {
  using SH = RowShape<C, L>;
  using LAY = typename SH::LAY;
  constexpr int E = LAY::E, T = LAY::T;
  constexpr int R1 = line_radix(L, LAY::WIDE, true, 0), RL = line_radix(L, LAY::WIDE, true, LAY::P.nf - 1);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int li = threadIdx.x / T, t = threadIdx.x - li * T;
  const long line = (long)blockIdx.x * SH::NL + li;
  const bool valid = line < a.lines;
  C v[E];
  pdl_wait();
  const C* in = static_cast<const C*>(a.in) + line * a.in_ls;
#pragma unroll
  for (int m = 0; m < E / R1; ++m)
#pragma unroll
    for (int r = 0; r < R1; ++r) v[m * R1 + r] = valid ? in[t + m * T + r * (L / R1)] : czero_l<C>();
  line_fft<C, L, 1, false, true, SH::WARP, LAY>(v, reinterpret_cast<C*>(smem_raw) + li * LAY::LS,
                                                static_cast<const C*>(a.tw), t);
  pdl_trigger_small();
  if (!valid) return;
  // the added and subtracted entries of a butterfly are loaded together, before any store (the
  // output may be one of them)
  using A = typename std::conditional<OUT64, double2, C>::type;
  constexpr bool F32 = std::is_same<C, float2>::value;
  using B = typename std::conditional<F32, C, A>::type;  // FP32 arithmetic rounds addv as it is read
  const A* addv = static_cast<const A*>(a.addv);
  const A* subv = static_cast<const A*>(a.subv);
  A* out = static_cast<A*>(a.out) + line * a.out_ls;
#pragma unroll
  for (int m = 0; m < E / RL; ++m) {
    B add[RL / 2], sub[RL / 2];
#pragma unroll
    for (int r = 0; r < RL / 2; ++r) {
      const long i = line * a.add_ls + t + m * T + r * (L / RL);
      add[r] = czero_l<B>();
      if (addv) {
        if constexpr (OUT64 && F32) add[r] = l_of_f64<B>(addv[i]);
        else add[r] = addv[i];
      }
      if constexpr (OUT64 && !F32) sub[r] = subv ? subv[i] : czero_l<B>();
    }
#pragma unroll
    for (int r = 0; r < RL / 2; ++r) {
      const C x = v[m * RL + r];
      A o;
      if constexpr (OUT64 && F32) {
        const C y = l_add(x, add[r]);
        o = make_double2(f64_of(y.x), f64_of(y.y));
      } else if constexpr (OUT64) {
        o = l_add(l_to_f64(x), add[r]);
        if (subv) o = l_sub(sub[r], o);
      } else {
        o = l_norm(l_add(x, add[r]));
      }
      out[t + m * T + r * (L / RL)] = o;
    }
  }
}

// ------------------------------------------------------------------------------------
// Column passes: lines strided (element stride es), TC neighbouring lines per CTA (32 bytes of a
// row at least: whole sectors), threads running through the tile's lines first.
// MODE 0: forward (n in, L out); 1: inverse (L in, n out); 2: forward, symbol, inverse (n in, n out).
// ------------------------------------------------------------------------------------
template <typename C, int L> struct ColShape {
  static constexpr bool WIDE = sizeof(C) == 16;
  static constexpr int TC = std::is_same<C, double2>::value ? (L < 64 ? 8 : L <= 256 ? 4 : 2)
                            : WIDE ? (L <= 256 ? 8 : (L <= 1024 ? 4 : 2)) : (L <= 256 ? 16 : (L <= 1024 ? 8 : 4));
  using LAY = LineLay<C, L, TC>;
  static constexpr int NT = TC * LAY::T;
  static constexpr int REGS = LAY::E * (int)sizeof(C) / 4 > 32 ? 128 : (std::is_same<C, ffp>::value ? 80 : 64);
  static constexpr int WT = NT < 32 ? 32 : NT;  // whole warps
  static constexpr int MINB = 65536 / (WT * REGS) < 1 ? 1 : 65536 / (WT * REGS);
  static constexpr bool WARP = NT <= 32;
  static constexpr size_t SMEM = (size_t)TC * LAY::LS * sizeof(C);
  static_assert(L % TC == 0 && NT <= 1024, "column tiles divide every inner extent (L or L^2)");
};

template <typename C, int L, int MODE>
__global__ void __launch_bounds__(ColShape<C, L>::NT, ColShape<C, L>::MINB) k_col_pass(ColPassArgs a) {
  using SH = ColShape<C, L>;
  using LAY = typename SH::LAY;
  constexpr int E = LAY::E, T = LAY::T, TC = SH::TC, n = L / 2;
  constexpr int F1 = line_radix(L, LAY::WIDE, false, 0), FL = line_radix(L, LAY::WIDE, false, LAY::P.nf - 1);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int c = threadIdx.x % TC, t = threadIdx.x / TC;
  const int tiles = (int)(a.inner / TC);
  const long o = blockIdx.x / tiles;
  const int c0 = (int)(blockIdx.x - o * tiles) * TC + c;
  const C* in = static_cast<const C*>(a.in) + o * a.in_os + c0;
  C* out = static_cast<C*>(a.out) + o * a.out_os + c0;
  const C* tw = static_cast<const C*>(a.tw);
  C* s = reinterpret_cast<C*>(smem_raw) + c * LAY::LS;
  C v[E];
  pdl_wait();
  if constexpr (MODE != 1) {
#pragma unroll
    for (int m = 0; m < E / F1; ++m)
#pragma unroll
      for (int r = 0; r < F1 / 2; ++r) v[m * F1 + r] = in[(t + m * T + r * (L / F1)) * a.in_es];
    line_fft<C, L, -1, true, false, SH::WARP, LAY>(v, s, tw, t);
  } else {
#pragma unroll
    for (int m = 0; m < E / FL; ++m)
#pragma unroll
      for (int r = 0; r < FL; ++r) v[m * FL + r] = in[(t + m * T + r * (L / FL)) * a.in_es];
  }
  if constexpr (MODE == 0) {
    pdl_trigger_small();
#pragma unroll
    for (int m = 0; m < E / FL; ++m)
#pragma unroll
      for (int r = 0; r < FL; ++r) out[(t + m * T + r * (L / FL)) * a.out_es] = l_norm(v[m * FL + r]);
  }
  if constexpr (MODE == 2) {
    // the symbol is even in every axis: entry e of the line reads row min(e, L - e) of the
    // quadrant at the line's (folded) position on the other axes
    const int n1 = n + 1;
    int base, es;
    if (a.d == 2) {
      base = c0 <= n ? c0 : L - c0;
      es = n1;
    } else {
      const int k1 = c0 / L, k2 = c0 % L;
      base = (k1 <= n ? k1 : L - k1) * n1 + (k2 <= n ? k2 : L - k2);
      es = n1 * n1;
    }
    const C* sym = static_cast<const C*>(a.sym) + base;
#pragma unroll
    for (int m = 0; m < E / FL; ++m)
#pragma unroll
      for (int r = 0; r < FL; ++r) {
        const int e = t + m * T + r * (L / FL);
        v[m * FL + r] = l_norm(l_mul(v[m * FL + r], l_ldg(sym + (e <= n ? e : L - e) * es)));
      }
    line_sync<SH::WARP>();  // the forward transform's last reads before the inverse one's stores
  }
  if constexpr (MODE != 0) {
    line_fft<C, L, 1, false, true, SH::WARP, LAY>(v, s, tw, t);
    pdl_trigger_small();
#pragma unroll
    for (int m = 0; m < E / F1; ++m)
#pragma unroll
      for (int r = 0; r < F1 / 2; ++r) out[(t + m * T + r * (L / F1)) * a.out_es] = l_norm(v[m * F1 + r]);
  }
}

// ------------------------------------------------------------------------------------
// Host dispatch
// ------------------------------------------------------------------------------------
template <typename K> void pass_smem(K kern, size_t smem, std::atomic<bool>& attr) {
  if (!attr.load(std::memory_order_acquire)) {  // set once per process; repeats are harmless
    LS_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr.store(true, std::memory_order_release);
  }
}

template <typename C, int L, int IN> void launch_row_fwd(const RowPassArgs& a, cudaStream_t st) {
  using SH = RowShape<C, L>;
  static std::atomic<bool> attr{false};
  pass_smem(k_row_fwd<C, L, IN>, SH::SMEM, attr);
  static const std::string cls = std::string("fft_row_fwd_") + arith_tag<C>();
  const long blocks = (a.lines + SH::NL - 1) / SH::NL;
  if (blocks > 0) LS_LAUNCH(cls.c_str(), st, k_row_fwd<C, L, IN><<<(unsigned)blocks, SH::NT, SH::SMEM, st>>>(a));
}
template <typename C, int L, bool OUT64> void launch_row_inv(const RowPassArgs& a, cudaStream_t st) {
  using SH = RowShape<C, L>;
  static std::atomic<bool> attr{false};
  pass_smem(k_row_inv<C, L, OUT64>, SH::SMEM, attr);
  static const std::string cls = std::string("fft_row_inv_") + arith_tag<C>();
  const long blocks = (a.lines + SH::NL - 1) / SH::NL;
  if (blocks > 0) LS_LAUNCH(cls.c_str(), st, launch_pdl(k_row_inv<C, L, OUT64>, (unsigned)blocks, SH::NT, SH::SMEM, st, a));
}
// the forms that the operator uses: FP32 vectors in FP32 or FP64, FP64 in FP64, float-float in FP64
template <typename C, int L> void launch_row_L(int sign, const RowPassArgs& a, cudaStream_t st) {
  constexpr bool FF = std::is_same<C, ffp>::value, F32 = std::is_same<C, float2>::value;
  if (sign < 0) {
    if (a.phase) {
      if constexpr (!F32) launch_row_fwd<C, L, ROW_IN_WAVE>(a, st);
      else LS_FAIL(EINVAL_, "row pass: no plane waves in FP32");
    } else if constexpr (FF) {
      launch_row_fwd<C, L, ROW_IN_F64>(a, st);
    } else if (F32 && a.io64) {
      if constexpr (F32) launch_row_fwd<C, L, ROW_IN_F64>(a, st);
    } else {
      launch_row_fwd<C, L, ROW_IN_C>(a, st);
    }
  } else if (F32 && a.io64) {
    if constexpr (F32) launch_row_inv<C, L, true>(a, st);
  } else {
    launch_row_inv<C, L, FF>(a, st);
  }
}

template <typename C, int L, int MODE> void launch_col_L(const ColPassArgs& a, cudaStream_t st) {
  using SH = ColShape<C, L>;
  static std::atomic<bool> attr{false};
  pass_smem(k_col_pass<C, L, MODE>, SH::SMEM, attr);
  static const std::string cls =
      std::string(MODE == 0 ? "fft_col_fwd_" : MODE == 1 ? "fft_col_inv_" : "fft_col_sym_") + arith_tag<C>();
  const long blocks = a.inner / SH::TC * a.outer;
  if (blocks > 0) LS_LAUNCH(cls.c_str(), st, launch_pdl(k_col_pass<C, L, MODE>, (unsigned)blocks, SH::NT, SH::SMEM, st, a));
}

#define LS_FOR_L(X) X(16) X(32) X(48) X(64) X(96) X(128) X(256) X(512) X(1024) X(2048) X(4096)

// Explicit instantiation (PREFIX empty) or instantiation declaration (PREFIX extern) of the
// launchers of one arithmetic C and one length LL: the float-float passes spread their lengths over
// several translation units, which compile in parallel.
#define LS_PASS_INST(PREFIX, C, LL)                                                \
  PREFIX template void launch_row_L<C, LL>(int, const RowPassArgs&, cudaStream_t); \
  PREFIX template void launch_col_L<C, LL, 0>(const ColPassArgs&, cudaStream_t);   \
  PREFIX template void launch_col_L<C, LL, 1>(const ColPassArgs&, cudaStream_t);   \
  PREFIX template void launch_col_L<C, LL, 2>(const ColPassArgs&, cudaStream_t);

template <typename C> void row_pass(int L, int sign, const RowPassArgs& a, cudaStream_t st) {
  switch (L) {
#define CASE(LL)                     \
  case LL:                           \
    launch_row_L<C, LL>(sign, a, st); \
    return;
    LS_FOR_L(CASE)
#undef CASE
  }
  LS_FAIL(EINVAL_, "unsupported FFT length %d", L);
}

template <typename C> void col_pass(int L, int mode, const ColPassArgs& a, cudaStream_t st) {
  switch (L) {
#define CASE(LL)                                          \
  case LL:                                                \
    if (mode == 0) launch_col_L<C, LL, 0>(a, st);         \
    else if (mode == 1) launch_col_L<C, LL, 1>(a, st);    \
    else launch_col_L<C, LL, 2>(a, st);                   \
    return;
    LS_FOR_L(CASE)
#undef CASE
  }
  LS_FAIL(EINVAL_, "unsupported FFT length %d", L);
}

}  // namespace ls
