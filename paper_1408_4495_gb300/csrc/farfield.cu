// Far-field pattern of the scattered field (exterior evaluation after the solve).
//
// The total field u = u_I + u_s solves u + K(omega^2 m u) = u_I (Sec. 1, eq. ls), so outside
// the domain u_s(x) = -int G(x - y) omega^2 m(y) u(y) dy.  With the large-|x| form of the
// Green's function, G(x - y) ~ c_d e^{i omega r} r^{-(d-1)/2} e^{-i omega theta . y} in the
// direction theta = x / r, the scattered field behaves as e^{i omega r} r^{-(d-1)/2} u_inf:
//   u_inf(theta) = -c_d h^d sum_i e^{-i omega theta . x_i} w_i (u_I(x_i) + u_s,i),
//   w = omega^2 m,  c_2 = e^{i pi/4} / sqrt(8 pi omega),  c_3 = 1 / (4 pi),
// the integral replaced by the Nystrom quadrature of K.
//
// The sum is a contraction: with v_r = w (u_I + u_s) formed once per wave r, every pair of wave
// and direction costs one product per point.  Both exponentials factor over the axes, and the
// grid is symmetric about 1/2 (n even, x_{n-1-j} = 1 - x_j), so along the last axis a pair of
// points gives (v_j + v_{n-1-j}) cos phi_j - i (v_j - v_{n-1-j}) sin phi_j with
// phi_j = omega theta (x_j - 1/2): real times complex, two FP64 FMAs per point and direction.
// Bound by the FP64 pipe (GB300: 2 FMAs per clock and SM).  2D n = 512, 32 waves, 64 directions
// (1.07e9 FMAs, 1.7 ms at 6.3e11 a second; 1.1 ms over the support of the medium): 1.54 ms,
// against 18.1 ms for one block per wave and direction with five complex products a point.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "far_plan.h"
#include "kernels.h"
#include "pdl.cuh"
#include "prof.h"

namespace ls {

namespace {

constexpr int FK = 16;        // point pairs of a line per chunk
constexpr int FTHREADS = 128;  // 8 groups of two lines x 16 direction groups

struct FarTabs {
  const double2* inc;   // [nrhs][d][n]      e^{i omega d_a x_j}
  const double2* outer; // [d - 1][n][nobs]  e^{-i omega theta_a x_j}, a < d - 1
  const double2* cs;    // [n / 2][nobs]     (cos, sin) of omega theta_{d-1} (x_j - 1/2)
};

__global__ void k_far_tables(int d, int n, int nrhs, int nobs, const double* __restrict__ dirs,
                             const double* __restrict__ obs, double omega, double h, double2* __restrict__ inc,
                             double2* __restrict__ outer, double2* __restrict__ cs) {
  const long n0 = (long)nrhs * d * n, n1 = (long)(d - 1) * n * nobs, n2 = (long)(n / 2) * nobs;
  pdl_trigger_small();
  for (long t = blockIdx.x * (long)blockDim.x + threadIdx.x; t < n0 + n1 + n2; t += (long)gridDim.x * blockDim.x) {
    double sn, cn;
    if (t < n0) {
      const long ra = t / n;
      sincos(omega * dirs[ra] * ((double)(t - ra * n + 1) * h), &sn, &cn);
      inc[t] = make_double2(cn, sn);
    } else if (t < n0 + n1) {
      const long u = t - n0, aj = u / nobs;
      const int k = (int)(u - aj * nobs), a = (int)(aj / n), j = (int)(aj - (long)a * n);
      sincos(-omega * obs[(size_t)k * d + a] * ((double)(j + 1) * h), &sn, &cn);
      outer[u] = make_double2(cn, sn);
    } else {
      const long u = t - n0 - n1;
      const int j = (int)(u / nobs), k = (int)(u - (long)j * nobs);
      sincos(omega * obs[(size_t)k * d + d - 1] * ((double)(2 * j + 1 - n) * (0.5 * h)), &sn, &cn);
      cs[u] = make_double2(cn, sn);
    }
  }
}

// One CTA: FL lines of wave r = blockIdx.y against 16 TN directions.  The line pairs of a chunk
// are formed once into shared memory (sum and difference of the two points of a pair) and used
// for all its directions; a thread accumulates two lines x TN directions.  Chunks where the
// medium vanishes are skipped (points with w = 0 do not enter the sum, whatever u_s holds
// there).  partial[(r * tiles + tile) * nobs + k]: the tile's sum for direction k.
template <int D, int TN>
__global__ void __launch_bounds__(FTHREADS) k_far_sum(int n, int nobs, int tiles, const double2* __restrict__ us,
                                                      const double* __restrict__ w, FarTabs tab,
                                                      double2* __restrict__ partial) {
  __shared__ double2 sp[FK][FL + 1], sm[FK][FL + 1];
  __shared__ double2 tc[FK][16 * TN];
  const int tile = blockIdx.x, r = blockIdx.y, k0 = blockIdx.z * 16 * TN;
  const long lines = D == 2 ? n : (long)n * n, l0 = (long)tile * FL;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const double2* u = us + (size_t)r * lines * n;
  const double2* inc = tab.inc + (size_t)r * D * n;
  double2 acc[2][TN];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int q = 0; q < TN; ++q) acc[i][q] = make_double2(0.0, 0.0);
  pdl_enter();
  for (int j0 = 0; j0 < n / 2; j0 += FK) {
    int any = 0;
#pragma unroll
    for (int e = threadIdx.x; e < FK * FL; e += FTHREADS) {
      const int jj = e % FK, li = e / FK, j = j0 + jj;
      const long line = l0 + li;
      double2 a = make_double2(0.0, 0.0), b = a;
      if (j < n / 2 && line < lines) {
        const size_t ia = (size_t)line * n + j, ib = (size_t)line * n + n - 1 - j;
        const double wa = w[ia], wb = w[ib];
        if (wa != 0.0 || wb != 0.0) {
          any = 1;
          double2 p = D == 2 ? inc[line] : cmul(inc[line / n], inc[n + line % n]);
          const double2* il = inc + (size_t)(D - 1) * n;
          if (wa != 0.0) a = cscale(cadd(cmul(p, il[j]), u[ia]), wa);
          if (wb != 0.0) b = cscale(cadd(cmul(p, il[n - 1 - j]), u[ib]), wb);
        }
      }
      sp[jj][li] = cadd(a, b);
      sm[jj][li] = csub(a, b);
    }
    if (!__syncthreads_or(any)) continue;  // (nothing read the tiles: the next chunk overwrites them)
    for (int e = threadIdx.x; e < FK * 16 * TN; e += FTHREADS) {
      const int jj = e / (16 * TN), k = k0 + e % (16 * TN);
      tc[jj][e % (16 * TN)] =
          j0 + jj < n / 2 && k < nobs ? tab.cs[(size_t)(j0 + jj) * nobs + k] : make_double2(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll 4
    for (int jj = 0; jj < FK; ++jj) {
      const double2 s0 = sp[jj][ty], s1 = sp[jj][ty + 8], d0 = sm[jj][ty], d1 = sm[jj][ty + 8];
#pragma unroll
      for (int q = 0; q < TN; ++q) {
        const double2 t = tc[jj][tx + 16 * q];
        acc[0][q].x = fma(d0.y, t.y, fma(s0.x, t.x, acc[0][q].x));
        acc[0][q].y = fma(-d0.x, t.y, fma(s0.y, t.x, acc[0][q].y));
        acc[1][q].x = fma(d1.y, t.y, fma(s1.x, t.x, acc[1][q].x));
        acc[1][q].y = fma(-d1.x, t.y, fma(s1.y, t.x, acc[1][q].y));
      }
    }
    __syncthreads();
  }
  // the factors of the other axes, then the sum over the tile's lines in a fixed order
  double2(*red)[16 * TN] = tc;  // [8][16 TN] of the chunk's [FK][16 TN]
#pragma unroll
  for (int q = 0; q < TN; ++q) {
    const int k = k0 + tx + 16 * q;
    double2 s = make_double2(0.0, 0.0);
    if (k < nobs) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const long line = l0 + ty + 8 * i;
        if (line >= lines) continue;
        const double2 f = D == 2 ? tab.outer[(size_t)line * nobs + k]
                                 : cmul(tab.outer[(size_t)(line / n) * nobs + k],
                                        tab.outer[(size_t)(n + line % n) * nobs + k]);
        s = cadd(s, cmul(f, acc[i][q]));
      }
    }
    red[ty][tx + 16 * q] = s;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < 16 * TN; e += FTHREADS) {
    if (k0 + e >= nobs) continue;
    double2 s = red[0][e];
#pragma unroll
    for (int g = 1; g < 8; ++g) s = cadd(s, red[g][e]);
    partial[((size_t)r * tiles + tile) * nobs + k0 + e] = s;
  }
}

// out[r][k] = -h^d c_d e^{-i omega theta_{d-1} / 2} * sum over the tiles (8 segments, in order)
__global__ void __launch_bounds__(256) k_far_reduce(int d, int nobs, int tiles, const double2* partial,
                                                    const double* __restrict__ obs, double omega, double hd, double2 cd,
                                                    double2* __restrict__ out, int ostride) {
  __shared__ double2 red[8][32];
  const int r = blockIdx.y, lane = threadIdx.x & 31, seg = threadIdx.x >> 5, k = blockIdx.x * 32 + lane;
  const int per = (tiles + 7) / 8, t1 = min(tiles, (seg + 1) * per);
  double2 s = make_double2(0.0, 0.0);
  pdl_wait();
  if (k < nobs)
    for (int t = seg * per; t < t1; ++t) s = cadd(s, partial[((size_t)r * tiles + t) * nobs + k]);
  red[seg][lane] = s;
  __syncthreads();
  if (seg != 0 || k >= nobs) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) s = cadd(s, red[q][lane]);
  double sn, cn;
  sincos(-0.5 * omega * obs[(size_t)k * d + d - 1], &sn, &cn);
  const double2 v = cmul(cmul(cd, make_double2(cn, sn)), s);
  out[(size_t)r * ostride + k] = make_double2(-hd * v.x, -hd * v.y);
}

}  // namespace

template <int D, int TN>
static void launch_far_sum(int n, int nrhs, int nobs, int tiles, const double2* us, const double* w, const FarTabs& tab,
                           double2* partial, cudaStream_t st) {
  LS_LAUNCH("far_field", st,
            launch_pdl(k_far_sum<D, TN>, dim3(tiles, nrhs, (nobs + 16 * TN - 1) / (16 * TN)), FTHREADS, 0, st, n, nobs,
                       tiles, us, w, tab, partial));
}

void far_field(int d, int n, int nrhs, int nobs, const double2* us, const double* dirs, const double* obs,
               const double* w, double omega, double h, double2* out, double2* scratch, cudaStream_t st) {
  const double2 cd = d == 2 ? make_double2(cos(M_PI / 4) / sqrt(8 * M_PI * omega), sin(M_PI / 4) / sqrt(8 * M_PI * omega))
                            : make_double2(1.0 / (4 * M_PI), 0.0);
  const int tiles = far_tiles(d, n), chunk = far_chunk(d, n, nrhs, nobs);
  for (long kc = 0; kc < nobs; kc += chunk) {
    const int ko = (int)std::min<long>(chunk, nobs - kc);
    const double* ob = obs + (size_t)kc * d;
    const size_t n0 = (size_t)nrhs * d * n, n1 = (size_t)(d - 1) * n * ko, n2 = (size_t)(n / 2) * ko;
    double2 *inc = scratch, *outer = inc + n0, *cs = outer + n1, *partial = cs + n2;
    LS_LAUNCH("far_field", st,
              k_far_tables<<<(unsigned)std::min<size_t>((n0 + n1 + n2 + 127) / 128, 152 * 8), 128, 0, st>>>(
                  d, n, nrhs, ko, dirs, ob, omega, h, inc, outer, cs));
    // directions per CTA: 64, or 32 or 16 where that leaves fewer idle (a smaller tile forms v_r
    // more often: about 10 FP64 operations a point against 2 per direction) or SMs without a CTA (one
    // wave, 64 directions: 2D n = 32 61 -> 42 us a call with the overlapped launches below, n = 128 122 ->
    // 65, n = 512 311 -> 140; the single launch of a block per wave and direction took 52, 144, 1485)
    const FarTabs tab{inc, outer, cs};
    const int pad64 = (ko + 63) / 64 * 64, pad32 = (ko + 31) / 32 * 32, pad16 = (ko + 15) / 16 * 16;
    int tn = pad16 < pad32 ? 1 : (pad32 < pad64 ? 2 : 4);
    while (tn > 1 && (long)tiles * nrhs * ((ko + 16 * tn - 1) / (16 * tn)) < 152) tn /= 2;
    auto sum = d == 2 ? (tn == 1 ? launch_far_sum<2, 1> : (tn == 2 ? launch_far_sum<2, 2> : launch_far_sum<2, 4>))
                      : (tn == 1 ? launch_far_sum<3, 1> : (tn == 2 ? launch_far_sum<3, 2> : launch_far_sum<3, 4>));
    sum(n, nrhs, ko, tiles, us, w, tab, partial, st);
    LS_LAUNCH("far_field", st,
              launch_pdl(k_far_reduce, dim3((ko + 31) / 32, nrhs), 256, 0, st, d, ko, tiles, (const double2*)partial, ob,
                         omega, d == 2 ? h * h : h * h * h, cd, out + kc, nobs));
  }
}

}  // namespace ls
