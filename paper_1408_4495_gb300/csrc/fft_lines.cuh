// Line transforms of the FFT passes with the values in registers (plan in fft_lines.h), in FP32,
// FP64 and float-float arithmetic.
//
// Shared-memory layout of a line during a transform with factors R1, R2 (, R3): value (k1, i) at
// k1 S1 + i, i < L / R1, S1 = L / R1 + 1, and lines LS apart with LS = U / G (mod U), U the
// entries of 128 bytes, G the group of neighbouring lines (or threads) a warp touches: every
// store and load of a quarter or half warp then falls on distinct banks (checked by a model of
// all lengths and layouts).  The second exchange of a three-factor transform writes the places it
// has read, so each exchange takes one barrier.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "ffloat.cuh"
#include "fft_lines.h"

namespace ls {

// ------------------------------------------------------------------------------ arithmetic
// Float-float complex number of the passes: leading and trailing parts as (re, im) pairs, so that
// an addition runs on packed pairs (add.rn.f32x2: one instruction for both components).
struct __align__(16) ffp {
  float2 h, l;
};

#define LS_PACKED2(name, op)                                                              \
  __device__ __forceinline__ float2 name(float2 a, float2 b) {                            \
    unsigned long long x, y, r;                                                           \
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));                          \
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));                          \
    asm(op ".rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));                           \
    float2 o;                                                                             \
    asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));                         \
    return o;                                                                             \
  }
LS_PACKED2(p_add, "add")
LS_PACKED2(p_sub, "sub")
#undef LS_PACKED2
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) {
  unsigned long long x, y, z, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(z) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
  float2 o;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(o.x), "=f"(o.y) : "l"(r));
  return o;
}

// FP32 pair of a constant
struct FfConst {
  float h, l;
};
__host__ __device__ constexpr FfConst ff_const(double c) { return FfConst{(float)c, (float)(c - (double)(float)c)}; }

// l_add, l_sub: a +- b; l_addi<S>: a + S i b (S = +1 or -1); l_mul: a w; l_scale: a c
__device__ __forceinline__ float2 l_add(float2 a, float2 b) { return p_add(a, b); }
__device__ __forceinline__ float2 l_sub(float2 a, float2 b) { return p_sub(a, b); }
template <int S> __device__ __forceinline__ float2 l_addi(float2 a, float2 b) {
  return S > 0 ? make_float2(a.x - b.y, a.y + b.x) : make_float2(a.x + b.y, a.y - b.x);
}
__device__ __forceinline__ float2 l_mul(float2 a, float2 w) {
  return make_float2(fmaf(a.x, w.x, -(a.y * w.y)), fmaf(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ float2 l_neg(float2 a) { return make_float2(-a.x, -a.y); }
template <int S> __device__ __forceinline__ float2 l_rot(float2 a) {
  return S > 0 ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}
__device__ __forceinline__ float2 l_norm(float2 a) { return a; }
// a (c + i s), constants, with the constants' FP32 rounding errors made up for: they are the same
// for every line, forward and inverse, so they would add up where the other roundings average out
// (2D n = 512: error of the apply 7.4e-8 without this, 6.5e-8 with the radix-8 passes)
__device__ __forceinline__ float2 l_mulc(float2 a, double c, double s) {
  const FfConst kc = ff_const(c), ks = ff_const(s);
  const float px = fmaf(a.x, kc.l, -(a.y * ks.l)), py = fmaf(a.x, ks.l, a.y * kc.l);
  return make_float2(fmaf(a.x, kc.h, -fmaf(a.y, ks.h, -px)), fmaf(a.x, ks.h, fmaf(a.y, kc.h, py)));
}
__device__ __forceinline__ float2 l_scale(float2 a, double c) {
  const FfConst k = ff_const(c);
  return make_float2(fmaf(a.x, k.h, a.x * k.l), fmaf(a.y, k.h, a.y * k.l));
}

__device__ __forceinline__ double2 l_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 l_sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <int S> __device__ __forceinline__ double2 l_addi(double2 a, double2 b) {
  return S > 0 ? make_double2(a.x - b.y, a.y + b.x) : make_double2(a.x + b.y, a.y - b.x);
}
__device__ __forceinline__ double2 l_mul(double2 a, double2 w) {
  return make_double2(fma(a.x, w.x, -(a.y * w.y)), fma(a.x, w.y, a.y * w.x));
}
__device__ __forceinline__ double2 l_neg(double2 a) { return make_double2(-a.x, -a.y); }
template <int S> __device__ __forceinline__ double2 l_rot(double2 a) {
  return S > 0 ? make_double2(-a.y, a.x) : make_double2(a.y, -a.x);
}
__device__ __forceinline__ double2 l_norm(double2 a) { return a; }
__device__ __forceinline__ double2 l_mulc(double2 a, double c, double s) { return l_mul(a, make_double2(c, s)); }
__device__ __forceinline__ double2 l_scale(double2 a, double c) { return make_double2(a.x * c, a.y * c); }

// Float-float with the renormalisation deferred (ffloat.cuh): an addition keeps the exact TwoSum
// of the leading parts and adds the trailing parts; values are renormalised (l_norm) once per
// factor pass, when they go to shared memory.
__device__ __forceinline__ ffp l_add(ffp a, ffp b) {
  const float2 s = p_add(a.h, b.h), nb = p_sub(a.h, s);  // nb = -(s - a)
  const float2 e = p_add(p_sub(a.h, p_add(s, nb)), p_add(b.h, nb));
  return ffp{s, p_add(e, p_add(a.l, b.l))};
}
__device__ __forceinline__ ffp l_sub(ffp a, ffp b) {
  const float2 s = p_sub(a.h, b.h), nb = p_sub(a.h, s);
  const float2 e = p_add(p_sub(a.h, p_add(s, nb)), p_sub(nb, b.h));
  return ffp{s, p_add(e, p_sub(a.l, b.l))};
}
template <int S> __device__ __forceinline__ ffp l_addi(ffp a, ffp b) {
  const float2 g = make_float2((float)-S, (float)S);
  const float2 bh = make_float2(b.h.y, b.h.x), bl = make_float2(b.l.y, b.l.x);
  const float2 s = p_fma(bh, g, a.h), nb = p_sub(a.h, s);
  const float2 e = p_add(p_sub(a.h, p_add(s, nb)), p_fma(bh, g, nb));
  return ffp{s, p_add(e, p_fma(bl, g, a.l))};
}
__device__ __forceinline__ ffp l_neg(ffp a) {
  return ffp{make_float2(-a.h.x, -a.h.y), make_float2(-a.l.x, -a.l.y)};
}
template <int S> __device__ __forceinline__ ffp l_rot(ffp a) {
  return S > 0 ? ffp{make_float2(-a.h.y, a.h.x), make_float2(-a.l.y, a.l.x)}
               : ffp{make_float2(a.h.y, -a.h.x), make_float2(a.l.y, -a.l.x)};
}
__device__ __forceinline__ ff ff_re(ffp a) { return ff(a.h.x, a.l.x); }
__device__ __forceinline__ ff ff_im(ffp a) { return ff(a.h.y, a.l.y); }
__device__ __forceinline__ ffp ffp_of(ff x, ff y) { return ffp{make_float2(x.hi, y.hi), make_float2(x.lo, y.lo)}; }
__device__ __forceinline__ ffp l_mul(ffp a, ffp w) {
  const ff x = lz_add(lz_mul(ff_re(a), ff_re(w)), lz_neg(lz_mul(ff_im(a), ff_im(w))));
  const ff y = lz_add(lz_mul(ff_re(a), ff_im(w)), lz_mul(ff_im(a), ff_re(w)));
  return ffp_of(x, y);
}
__device__ __forceinline__ ffp l_norm(ffp a) {
  const float2 s = p_add(a.h, a.l);
  return ffp{s, p_sub(a.l, p_sub(s, a.h))};
}
// a times the real float-float w.  Products stay scalar: ptxas contracts a packed multiplication
// that feeds a packed addition into one FMA whatever its rounding modifier says, which would lose
// the product's own rounding that the error term belongs to.
__device__ __forceinline__ ffp l_mulr(ffp a, ff w) { return ffp_of(lz_mul(ff_re(a), w), lz_mul(ff_im(a), w)); }
__device__ __forceinline__ ffp l_mulc(ffp a, double c, double s) {
  const FfConst kc = ff_const(c), ks = ff_const(s);
  return l_mul(a, ffp{make_float2(kc.h, ks.h), make_float2(kc.l, ks.l)});
}
__device__ __forceinline__ ffp l_scale(ffp a, double c) {
  const FfConst k = ff_const(c);
  return l_mulr(a, ff(k.h, k.l));
}
__device__ __forceinline__ ffp ffp_of_f64(double2 v) { return ffp_of(ff_of_f64(v.x), ff_of_f64(v.y)); }
__device__ __forceinline__ double2 ffp_to_f64(ffp v) { return make_double2(ff_to_f64(ff_re(v)), ff_to_f64(ff_im(v))); }

template <typename C> __device__ __forceinline__ C czero_l() { return czero<C>(); }
template <> __device__ __forceinline__ ffp czero_l<ffp>() { return ffp{make_float2(0.f, 0.f), make_float2(0.f, 0.f)}; }

// read-only cached load of one complex entry
template <typename C> __device__ __forceinline__ C l_ldg(const C* p) { return __ldg(p); }
template <> __device__ __forceinline__ ffp l_ldg<ffp>(const ffp* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return ffp{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

// ------------------------------------------------------------------------------ butterflies
// cos(2 pi k / N) for N = 8, 12, 16, 32
__host__ __device__ constexpr double cos_turn(int k, int N) {
  constexpr double q32[9] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                             0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                             0.19509032201612826785, 0.0};
  constexpr double q12[4] = {1.0, 0.86602540378443864676, 0.5, 0.0};
  const int M = N == 12 ? 12 : 32, m = ((k * (M / N)) % M + M) % M;
  const int f = m > M / 2 ? M - m : m;  // cos is even
  const int g = f > M / 4 ? M / 2 - f : f;
  const double c = N == 12 ? q12[g] : q32[g];
  return f > M / 4 ? -c : c;
}
__host__ __device__ constexpr double sin_turn(int k, int N) { return cos_turn(k - N / 4, N); }

// a exp(S 2 pi i K / N)
template <int K, int N, int S, typename C> __device__ __forceinline__ C l_turn(C a) {
  constexpr int k = K % N;
  if constexpr (k == 0) return a;
  else if constexpr (4 * k == N) return l_rot<S>(a);
  else if constexpr (2 * k == N) return l_neg(a);
  else if constexpr (4 * k == 3 * N) return l_rot<-S>(a);
  else if constexpr (8 * k == N) return l_scale(l_addi<S>(a, a), 0.70710678118654752440);       // (1 + S i) a
  else if constexpr (8 * k == 3 * N) return l_scale(l_addi<-S>(a, a), -0.70710678118654752440);  // -(1 - S i) a
  else if constexpr (8 * k == 5 * N) return l_scale(l_addi<S>(a, a), -0.70710678118654752440);
  else if constexpr (8 * k == 7 * N) return l_scale(l_addi<-S>(a, a), 0.70710678118654752440);
  else return l_mulc(a, cos_turn(k, N), S * sin_turn(k, N));
}

// 4-point DFT in place; P = 1: a2 = a3 = 0 (not read); P = 2: only outputs 0 and 1 formed
template <int S, int P, typename C> __device__ __forceinline__ void l_dft4(C& a0, C& a1, C& a2, C& a3) {
  if constexpr (P == 1) {
    const C x = a0, y = a1;
    a0 = l_add(x, y);
    a2 = l_sub(x, y);
    a1 = l_addi<S>(x, y);
    a3 = l_addi<-S>(x, y);
  } else {
    const C t0 = l_add(a0, a2), t1 = l_sub(a0, a2), t2 = l_add(a1, a3), t3 = l_sub(a1, a3);
    a0 = l_add(t0, t2);
    a1 = l_addi<S>(t1, t3);
    if constexpr (P != 2) {
      a2 = l_sub(t0, t2);
      a3 = l_addi<-S>(t1, t3);
    }
  }
}
template <int S, typename C> __device__ __forceinline__ void l_dft3(C& a0, C& a1, C& a2) {
  const C t = l_add(a1, a2), d = l_scale(l_sub(a1, a2), 0.86602540378443864676);
  const C m = l_sub(a0, l_scale(t, 0.5));
  a0 = l_add(a0, t);
  a1 = l_addi<S>(m, d);
  a2 = l_addi<-S>(m, d);
}

// in-register R-point DFT, v[k] <- sum_i v[i] exp(S 2 pi i k i / R), natural order.
// P = 1: v[R/2..] are zero and not read; P = 2: only v[0 .. R/2) formed.
template <int R, int S, int P, typename C> struct LineDft;
template <int S, int P, typename C> struct LineDft<4, S, P, C> {
  static __device__ __forceinline__ void run(C* v) { l_dft4<S, P>(v[0], v[1], v[2], v[3]); }
};
template <int S, int P, typename C> struct LineDft<8, S, P, C> {
  static __device__ __forceinline__ void run(C* v) {
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    l_dft4<S, P == 1 ? 1 : 0>(e0, e1, e2, e3);
    l_dft4<S, P == 1 ? 1 : 0>(o0, o1, o2, o3);
    o1 = l_turn<1, 8, S>(o1);
    o3 = l_turn<3, 8, S>(o3);
    v[0] = l_add(e0, o0);
    v[1] = l_add(e1, o1);
    v[2] = l_addi<S>(e2, o2);
    v[3] = l_add(e3, o3);
    if constexpr (P != 2) {
      v[4] = l_sub(e0, o0);
      v[5] = l_sub(e1, o1);
      v[6] = l_addi<-S>(e2, o2);
      v[7] = l_sub(e3, o3);
    }
  }
};
template <int S, int P, typename C> struct LineDft<6, S, P, C> {
  static __device__ __forceinline__ void run(C* v) {
    static_assert(P == 0, "radix 6: neither first nor last of a half-length end");
    l_dft3<S>(v[0], v[2], v[4]);
    l_dft3<S>(v[1], v[3], v[5]);
    const C o1 = l_turn<2, 12, S>(v[3]), o2 = l_turn<4, 12, S>(v[5]), e0 = v[0], e1 = v[2], e2 = v[4], o0 = v[1];
    v[0] = l_add(e0, o0);
    v[1] = l_add(e1, o1);
    v[2] = l_add(e2, o2);
    v[3] = l_sub(e0, o0);
    v[4] = l_sub(e1, o1);
    v[5] = l_sub(e2, o2);
  }
};
// R = 4 B: 4-point DFTs over i = b + B a, then B-point ones over b; output k = k1 + 4 k2
template <int R, int S, int P, typename C> struct LineDft4B {
  static constexpr int B = R / 4;
  template <int b> static __device__ __forceinline__ void first(C* v) {
    l_dft4<S, P == 1 ? 1 : 0>(v[b], v[b + B], v[b + 2 * B], v[b + 3 * B]);
    v[b + B] = l_turn<b, R, S>(v[b + B]);
    v[b + 2 * B] = l_turn<2 * b, R, S>(v[b + 2 * B]);
    v[b + 3 * B] = l_turn<3 * b, R, S>(v[b + 3 * B]);
    if constexpr (b + 1 < B) first<b + 1>(v);
  }
  static __device__ __forceinline__ void run(C* v) {
    first<0>(v);
    C w[R];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      C* u = v + k1 * B;
      if constexpr (B == 3) l_dft3<S>(u[0], u[1], u[2]);
      else LineDft<B, S, P == 2 ? 2 : 0, C>::run(u);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) w[k1 + 4 * k2] = u[k2];
    }
#pragma unroll
    for (int k = 0; k < (P == 2 ? R / 2 : R); ++k) v[k] = w[k];
  }
};
template <int S, int P, typename C> struct LineDft<12, S, P, C> : LineDft4B<12, S, P, C> {};
template <int S, int P, typename C> struct LineDft<16, S, P, C> : LineDft4B<16, S, P, C> {};
template <int S, int P, typename C> struct LineDft<32, S, P, C> : LineDft4B<32, S, P, C> {};

// ------------------------------------------------------------------------------ lines
// GROUP: neighbouring lines of a warp's accesses (column tiles: the tile's lines, which the
// threads run through first) or 0 for line-major threads
template <typename C, int L, int GROUP> struct LineLay {
  static constexpr bool WIDE = sizeof(C) == 16;
  static constexpr LinePlan P = line_plan(L, WIDE);
  static constexpr int E = P.e, T = L / E;  // values per thread, threads per line
  static constexpr int U = 128 / (int)sizeof(C);
  static constexpr int G = GROUP > 0 ? (U / GROUP > 0 ? U / GROUP : 1) : (T < U ? T : U);
  LS_FL_HD static constexpr int s1(bool inv) { return L / line_radix(L, WIDE, inv, 0) + 1; }
  LS_FL_HD static constexpr int span(bool inv) { return line_radix(L, WIDE, inv, 0) * s1(inv); }
  LS_FL_HD static constexpr int pad(int x) { return x + ((G - x) % U + U) % U; }
  static constexpr int LS = pad(span(false) > span(true) ? span(false) : span(true));  // entries per line
};

template <bool WARP> __device__ __forceinline__ void line_sync() {
  if constexpr (WARP) __syncwarp();
  else __syncthreads();
}

// Transform of one line by its T threads: v[m R1 + r] holds entry t + m T + r L / R1 before, and
// v[m Rl + r] entry t + m T + r L / Rl after (R1, Rl the first and last radix of the direction).
// HIN: entries L/2.. are zero (r >= R1 / 2 not read); HOUT: entries L/2.. are not formed.
// s: the line's shared memory, free on entry (the caller's barrier), tw: the whole table.
// WARP: the line's threads lie in one warp.
template <typename C, int L, int S, bool HIN, bool HOUT, bool WARP, typename LAY>
__device__ __forceinline__ void line_fft(C* v, C* __restrict__ s, const C* __restrict__ tw, int t) {
  constexpr bool WIDE = LAY::WIDE, INV = S > 0;
  constexpr int NF = LAY::P.nf, E = LAY::E, T = LAY::T;
  constexpr int R1 = line_radix(L, WIDE, INV, 0), R2 = line_radix(L, WIDE, INV, 1), R3 = line_radix(L, WIDE, INV, 2);
  constexpr int S1 = LAY::s1(INV), J1 = L / R1;
  static_assert(R1 * R2 * R3 == L && E % R1 == 0 && E % R2 == 0 && (NF == 2 || E % R3 == 0), "line plan");
  const C* tw1 = tw + (INV ? line_tw_dir(L, WIDE, false) : 0);
#pragma unroll
  for (int m = 0; m < E / R1; ++m) {
    C* x = v + m * R1;
    LineDft<R1, S, HIN ? 1 : 0, C>::run(x);
    const int j = t + m * T;
    s[j] = l_norm(x[0]);
#pragma unroll
    for (int k = 1; k < R1; ++k) s[k * S1 + j] = l_norm(l_mul(x[k], l_ldg(tw1 + k * J1 + j)));
  }
  line_sync<WARP>();
  if constexpr (NF == 2) {
#pragma unroll
    for (int m = 0; m < E / R2; ++m) {
      C* x = v + m * R2;
#pragma unroll
      for (int r = 0; r < R2; ++r) x[r] = s[(t + m * T) * S1 + r];
      LineDft<R2, S, HOUT ? 2 : 0, C>::run(x);
    }
  } else {
    const C* tw2 = tw1 + L;
#pragma unroll
    for (int m = 0; m < E / R2; ++m) {
      C* x = v + m * R2;
      const int u = t + m * T, k1 = u % R1, i3 = u / R1, o = k1 * S1 + i3;
#pragma unroll
      for (int r = 0; r < R2; ++r) x[r] = s[o + r * R3];
      LineDft<R2, S, 0, C>::run(x);
      s[o] = l_norm(x[0]);
#pragma unroll
      for (int k = 1; k < R2; ++k) s[o + k * R3] = l_norm(l_mul(x[k], l_ldg(tw2 + k * R3 + i3)));
    }
    line_sync<WARP>();
#pragma unroll
    for (int m = 0; m < E / R3; ++m) {
      C* x = v + m * R3;
      const int u = t + m * T, o = (u % R1) * S1 + (u / R1) * R3;
#pragma unroll
      for (int r = 0; r < R3; ++r) x[r] = s[o + r];
      LineDft<R3, S, HOUT ? 2 : 0, C>::run(x);
    }
  }
}

}  // namespace ls
