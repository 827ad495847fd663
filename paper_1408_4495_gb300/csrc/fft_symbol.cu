// Sec. 2.1: the symbol of the Nystrom table's circulant embedding, by full-length FP64 transforms
// (setup only).  Lines of L entries are held in shared memory and transformed by Stockham autosort
// passes of radix 8, then 4 or 2, then 3 (formulation as in Govindaraju et al., SC'08), whose
// factors come from the per-pass table of fft_plan.h.
#include <atomic>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "fft_plan.h"
#include "kernels.h"
#include "prof.h"

namespace ls {

namespace {

// Line-major without padding; inside each 128-byte row of 8 entries the position is XORed with the
// row index and the line (a bank swizzle), so that the strided stores of the passes spread over
// the banks.
template <int L, int LINES> struct SymLay {
  static constexpr int KC = 8 / LINES > 1 ? 8 / LINES : 1;
  static constexpr int SIZE = LINES * L;
  __device__ static __forceinline__ int off(int line, int i) {
    const int h = ((i / 8) & 7) ^ (line * KC);
    return line * L + (i & ~7) + ((i ^ h) & 7);
  }
};

__device__ __forceinline__ double2 minus_i(double2 a) { return make_double2(a.y, -a.x); }
__device__ __forceinline__ void sym_dft4(double2& a0, double2& a1, double2& a2, double2& a3) {
  const double2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = minus_i(csub(a1, a3));
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1 = cadd(t1, t3);
  a3 = csub(t1, t3);
}
template <int R> __device__ __forceinline__ void sym_dft(double2* v) {
  if constexpr (R == 2) {
    const double2 a = v[0];
    v[0] = cadd(a, v[1]);
    v[1] = csub(a, v[1]);
  } else if constexpr (R == 3) {
    const double2 a = v[0], t = cadd(v[1], v[2]), d = cscale(csub(v[1], v[2]), 0.86602540378443864676);
    const double2 m = csub(a, cscale(t, 0.5)), r = minus_i(d);
    v[0] = cadd(a, t);
    v[1] = cadd(m, r);
    v[2] = csub(m, r);
  } else if constexpr (R == 4) {
    sym_dft4(v[0], v[1], v[2], v[3]);
  } else {
    const double c = 0.70710678118654752440;
    double2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    sym_dft4(e0, e1, e2, e3);
    sym_dft4(o0, o1, o2, o3);
    o1 = make_double2(c * (o1.x + o1.y), c * (o1.y - o1.x));
    o2 = minus_i(o2);
    o3 = make_double2(c * (o3.y - o3.x), -(c * (o3.x + o3.y)));
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
  }
}

// the passes from sub-transforms of length NS to the whole line: butterfly j of a line reads
// entries j + r L/R, multiplies by w^{r k}, w = exp(-2 pi i / (NS R)), k = j mod NS, and writes
// (j / NS) NS R + k + r NS
template <int L, int NS, int LINES, int NT> __device__ __forceinline__ void sym_lines(double2* s, const double2* tw) {
  if constexpr (NS < L) {
    constexpr int R = pass_radix(L, NS), BPL = L / R, BF = LINES * BPL, PER = (BF + NT - 1) / NT;
    using SL = SymLay<L, LINES>;
    double2 v[PER][R];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int b = threadIdx.x + q * NT;
      if (BF % NT == 0 || b < BF) {
        const int line = b / BPL, j = b - line * BPL;
#pragma unroll
        for (int r = 0; r < R; ++r) v[q][r] = s[SL::off(line, j + r * BPL)];
        if constexpr (NS > 1) {
          const double2* w = tw + tw_pass_offset(L, NS) + (j % NS) * R;
#pragma unroll
          for (int r = 1; r < R; ++r) v[q][r] = cmul(v[q][r], __ldg(w + r));
        }
        sym_dft<R>(v[q]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int b = threadIdx.x + q * NT;
      if (BF % NT == 0 || b < BF) {
        const int line = b / BPL, j = b - line * BPL, base = (j / NS) * NS * R + j % NS;
#pragma unroll
        for (int r = 0; r < R; ++r) s[SL::off(line, base + r * NS)] = v[q][r];
      }
    }
    __syncthreads();
    sym_lines<L, NS * R, LINES, NT>(s, tw);
  }
}

// Eight entries a thread.  Short lines in small CTAs, 8 lines and more each (128 bytes of a strided
// line's row): a small grid has few lines, and with 256 threads at every length they filled a few SMs
// only (all passes of 3D n = 16 48.7 -> 36.1 us, n = 24 61.2 -> 38.7, 2D n = 64 40.8 -> 28.5; from 3D n = 64
// and 2D n = 128 on as before, the GPU is full either way).
template <int L> struct SymShape {
  static constexpr int NT = L > 2048 ? L / 8 : L >= 256 ? 256 : L >= 96 ? L : L == 48 ? 96 : 64;
  static constexpr int LINES = NT * 8 / L;
};

// lines of L entries, `inner` of them side by side with element stride es (inner = 1: contiguous
// lines), os apart between outer indices; in place
template <int L> __global__ void __launch_bounds__(SymShape<L>::NT) k_sym_lines(double2* x, long lines, long inner, long os,
                                                                             long es, const double2* __restrict__ tw) {
  constexpr int NT = SymShape<L>::NT, LINES = SymShape<L>::LINES;
  using SL = SymLay<L, LINES>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* s = reinterpret_cast<double2*>(smem_raw);
  const long line0 = (long)blockIdx.x * LINES;
  __shared__ long base[LINES];  // first entry of each of the CTA's lines, -1 past the last
  for (int li = threadIdx.x; li < LINES; li += NT) {
    const long line = line0 + li, o = line / inner;
    base[li] = line < lines ? o * os + (line - o * inner) : -1L;
  }
  __syncthreads();
  const bool rows = inner == 1;
  // contiguous lines: entries first; strided lines: the lines of one entry first
  for (int idx = threadIdx.x; idx < LINES * L; idx += NT) {
    const int li = rows ? idx / L : idx % LINES, e = rows ? idx % L : idx / LINES;
    s[SL::off(li, e)] = base[li] >= 0 ? x[base[li] + e * es] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  sym_lines<L, 1, LINES, NT>(s, tw);
  for (int idx = threadIdx.x; idx < LINES * L; idx += NT) {
    const int li = rows ? idx / L : idx % LINES, e = rows ? idx % L : idx / LINES;
    if (base[li] >= 0) x[base[li] + e * es] = s[SL::off(li, e)];
  }
}

template <int L> void launch_sym(double2* x, long lines, long inner, long os, long es, const double2* tw, cudaStream_t st) {
  constexpr size_t smem = (size_t)SymLay<L, SymShape<L>::LINES>::SIZE * sizeof(double2);
  static std::atomic<bool> attr{false};  // set once per process; repeats are harmless
  if (!attr.load(std::memory_order_acquire)) {
    LS_CUDA(cudaFuncSetAttribute(k_sym_lines<L>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    attr.store(true, std::memory_order_release);
  }
  const long blocks = (lines + SymShape<L>::LINES - 1) / SymShape<L>::LINES;
  LS_LAUNCH("fft_symbol", st,
            k_sym_lines<L><<<(unsigned)blocks, SymShape<L>::NT, smem, st>>>(x, lines, inner, os, es, tw));
}

void sym_pass(int L, double2* x, long lines, long inner, long os, long es, const double2* tw, cudaStream_t st) {
  switch (L) {
#define CASE(LL) \
  case LL: launch_sym<LL>(x, lines, inner, os, es, tw, st); return;
    CASE(16) CASE(32) CASE(48) CASE(64) CASE(96) CASE(128) CASE(256) CASE(512) CASE(1024) CASE(2048) CASE(4096)
#undef CASE
  }
  LS_FAIL(EINVAL_, "unsupported FFT length %d", L);
}

// kpad[k] = k_{t(k)} with t = k for k < n, k - L for k > n, and 0 where any k_a == n.
__global__ void k_kernel_pad(const double2* ktq, double2* kpad, int d, int n) {
  const long L = 2 * n, n1 = n + 1;
  const long total = d == 2 ? L * L : L * L * L;
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    long q = idx, src = 0, mul = 1;
    bool zero = false;
    for (int a = 0; a < d; ++a) {
      const long k = q % L;
      q /= L;
      if (k == n) zero = true;
      const long t = k < n ? k : L - k;
      src += t * mul;
      mul *= n1;
    }
    kpad[idx] = zero ? make_double2(0, 0) : ktq[src];
  }
}

// sym[q] = spectrum[q] / L^d on the quadrant q in [0, n]^d; FP64 and FP32 copies.
__global__ void k_symbol_quadrant(const double2* spec, double2* sym64, float2* sym32, int d, int n) {
  const long L = 2 * n, n1 = n + 1;
  const long total = d == 2 ? n1 * n1 : n1 * n1 * n1;
  const double scale = d == 2 ? 1.0 / (double)(L * L) : 1.0 / (double)(L * L * L);
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)gridDim.x * blockDim.x) {
    long q = idx, dst = 0, mul = 1;
    for (int a = 0; a < d; ++a) {
      const long k = q % n1;
      q /= n1;
      dst += k * mul;
      mul *= L;
    }
    double2 v = spec[dst];
    v.x *= scale;
    v.y *= scale;
    sym64[idx] = v;
    sym32[idx] = make_float2((float)v.x, (float)v.y);
  }
}

}  // namespace

void symbol_twiddles(int L, std::vector<double2>& tw) {
  tw.assign((size_t)tw_table_size(L), make_double2(0.0, 0.0));
  for (int NS = 1; NS < L; NS *= pass_radix(L, NS)) {
    const int R = pass_radix(L, NS);
    if (NS == 1) continue;  // the first pass has no factors
    double2* t = tw.data() + tw_pass_offset(L, NS);
    for (int k = 0; k < NS; ++k)
      for (int r = 0; r < R; ++r) {
        // w^{r k}, w = exp(-2 pi i / (NS R)); the exponent reduced mod NS R
        const long e = ((long)r * k) % ((long)NS * R);
        const double a = -2.0 * M_PI * (double)e / (double)(NS * R);
        t[(size_t)k * R + r] = make_double2(std::cos(a), std::sin(a));
      }
  }
}

// work: L^d entries; tw: the device copy of symbol_twiddles(L)
void build_symbol(int d, int n, const double2* ktq, double2* sym64, float2* sym32, double2* work, const double2* tw,
                  cudaStream_t st) {
  const int L = 2 * n;
  const long L2 = (long)L * L;
  LS_LAUNCH("kernel_pad", st, k_kernel_pad<<<1024, 256, 0, st>>>(ktq, work, d, n));
  sym_pass(L, work, d == 2 ? L : L2, 1, L, 1, tw, st);
  if (d == 2) {
    sym_pass(L, work, L, L, 0, L, tw, st);
  } else {
    sym_pass(L, work, L2, L, L2, L, tw, st);
    sym_pass(L, work, L2, L2, 0, L2, tw, st);
  }
  LS_LAUNCH("symbol", st, k_symbol_quadrant<<<1024, 256, 0, st>>>(work, sym64, sym32, d, n));
}

}  // namespace ls
