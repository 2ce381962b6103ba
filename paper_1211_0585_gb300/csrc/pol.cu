// Temperature and polarisation (Sect. 4, Conclusion: the method on T and P
// maps together, robust at their higher condition number; the power-spectra
// figure's TT, EE and TE).
//
// A pixel carries (T, Q, U) with a 3 x 3 noise covariance N_p (T independent
// of the Q-U block), separate temperature and polarisation masks (N^-1 = 0 on
// the masked components), and the signal S_l = [[TT, TE, 0], [TE, EE, 0],
// [0, 0, BB]] on (a^T, a^E, a^B). With T = tau 1 over all three components
// (tau = the smallest eigenvalue of N_p over the observed components) one
// iteration is
//   (s_T, s_Q, s_U) = Y s                    T: spin-0 synthesis; Q, U: spin-2 Legendre stage, ring FFTs
//   u_p = A_p (d_p - s_p),  A_p = lambda tau W_p (1 + (lambda - 1) tau W_p)^-1,  W_p = N_p^-1
//                                            Eq. 3, 3 x 3 per pixel
//   t = s + Y^dagger u                       ring FFTs, spin-0 and spin-2 Legendre analyses
//   s_lm = S_l (S_l + lambda tau Omega)^-1 t_lm   Eq. 4, the (T, E) block and B
// with Q +- iU = - sum (a^E +- i a^B) _{+-2}Y_lm: per ring and m,
//   Q_m = - sum_l (F+ a^E + i F- a^B),  U_m = - sum_l (F+ a^B - i F- a^E),
//   a^E = - sum_rings (F+ Q~_m + i F- U~_m),  a^B = - sum_rings (F+ U~_m - i F- Q~_m),
//   F+- = (_2 lambda_lm +- _-2 lambda_lm) / 2
//       F+ = N_l [(2 (m^2 - l) / s^2 - l (l - 1)) lambda_lm + 2 x c_lm lambda_{l-1,m} / s^2]
//       F- = N_l (2 m / s^2) [c_lm lambda_{l-1,m} - (l - 1) x lambda_lm]
// (N_l = ((l-1) l (l+1) (l+2))^-1/2, c_lm = sqrt((2l+1)/(2l-1) (l^2 - m^2)), x = cos theta,
// s^2 = 1 - x^2; zero for l < 2). On the south ring of a pair F+ takes the
// parity (-1)^{l-m} of lambda_lm and F- the opposite.
//
// The T channel, the azimuthal transforms of all three maps and the
// controller are the scalar plan's kernels (its precision). The spin-2
// Legendre stage reads a precomputed table of (F+, F-) per (l, m, ring pair):
// in double-float with compensated dot products on the FP32 pipe for
// WF_PREC_FP64 plans (GB300's FP64 pipe runs at 1/63 of it), in FP64 for
// WF_PREC_FP64_NATIVE plans. Rows below the first l at which lambda_lm(x_k)
// reaches 2^-100 hold zeros and are not read.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "ctl.cuh"
#include "df.cuh"
#include "wf_internal.h"
#include "wf_plan.h"

struct wf_pol_s {
  virtual ~wf_pol_s() = default;
};

namespace wfk {
namespace {

constexpr int kPolThreads = 256;
constexpr int kPixBlocks = 1024;   // pixel kernel: fixed grid, so its chi^2 partials sum in a fixed order
constexpr size_t kSpin2TableMax = size_t(64) << 30;

__device__ __forceinline__ size_t idx_lm(int lmax, int l, int m) { return (size_t)m * (2 * lmax + 1 - m) / 2 + l; }

// (F+, F-) of every (l, m) at the north ring of pair k: one thread per (m, k), the FP64 recurrence
// from the scalar plan's start values (first l with |lambda| >= 2^-100 and the two values there)
__global__ void spin2_table_kernel(const double *xk, const double2 *rec, const int *ls, const double2 *sv, int lmax,
                                   int RP, double2 *tab, int df) {
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= (long long)(lmax + 1) * RP) return;
  const int m = (int)(id / RP), k = (int)(id % RP);
  const double x = xk[k];
  const double s2 = (1.0 - x) * (1.0 + x);
  const size_t base = idx_lm(lmax, m, m);
  const int l0 = ls[id];
  double p1 = 0.0, p2 = 0.0;   // lambda_{l-1}, lambda_{l-2}
  for (int l = m; l <= lmax; ++l) {
    double lam = 0.0;
    if (l >= l0) {
      if (l == l0) lam = sv[id].x;
      else if (l == l0 + 1) lam = sv[id].y;
      else {
        const double2 ab = rec[base + (l - m)];
        lam = ab.x * x * p1 - ab.y * p2;
      }
    }
    double fp = 0.0, fm = 0.0;
    if (l >= 2 && l >= l0) {
      const double dl = l;
      const double nl = 1.0 / sqrt((dl - 1.0) * dl * (dl + 1.0) * (dl + 2.0));
      const double c = sqrt((2.0 * dl + 1.0) / (2.0 * dl - 1.0) * (dl * dl - (double)m * m));
      const double lm1 = l > m ? p1 : 0.0;
      fp = nl * ((2.0 * ((double)m * m - dl) / s2 - dl * (dl - 1.0)) * lam + 2.0 * x * c * lm1 / s2);
      fm = nl * (2.0 * m / s2) * (c * lm1 - (dl - 1.0) * x * lam);
    }
    if (df) {   // (F+ hi, F+ lo, F- hi, F- lo)
      const dfl a = df_from(fp), b = df_from(fm);
      reinterpret_cast<float4 *>(tab)[(base + (l - m)) * RP + k] = make_float4(a.h, a.l, b.h, b.l);
    } else {
      tab[(base + (l - m)) * RP + k] = make_double2(fp, fm);
    }
    p2 = p1;
    p1 = lam;
  }
}

// A launch of the spin-2 analyses takes nk <= kSpin2Pairs ring pairs (64 bytes of shared memory each; 128 KB), from the
// one that tab, ls and the Fourier records point at; RP stays their stride. The launches after the first (Nside 2048) add
// to a^E and a^B.
constexpr int kSpin2Pairs = 2048;

// spin-2 analysis: (a^E, a^B)_lm = - sum over ring pairs of the F+- terms; one CTA per m,
// a warp per l, lanes over ring pairs
__global__ void __launch_bounds__(kPolThreads) spin2_analysis_kernel(const Ctl *gate, const double2 *tab,
                                                                      const double4_32a *FTQ, const double4_32a *FTU,
                                                                      int lmax, int RP, int nk, int add, double2 *aE,
                                                                      double2 *aB) {
  if (gate && gate->done) return;
  extern __shared__ double4_32a pol_sm[];
  double4_32a *q = pol_sm, *u = pol_sm + nk;
  const int m = blockIdx.x;
  for (int k = threadIdx.x; k < nk; k += blockDim.x) {
    q[k] = FTQ[(size_t)m * RP + k];
    u[k] = FTU[(size_t)m * RP + k];
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const size_t base = idx_lm(lmax, m, m);
  for (int l = m + warp; l <= lmax; l += nw) {
    const double p = ((l - m) & 1) ? -1.0 : 1.0;
    double er = 0.0, ei = 0.0, br = 0.0, bi = 0.0;
    const double2 *row = tab + (base + (l - m)) * RP;
    for (int k = lane; k < nk; k += 32) {
      const double2 f = row[k];
      const double4_32a Q = q[k], U = u[k];
      // F+ sees Q_N + p Q_S, U_N + p U_S; F- sees Q_N - p Q_S, U_N - p U_S
      const double qpr = Q.x + p * Q.z, qpi = Q.y + p * Q.w, qmr = Q.x - p * Q.z, qmi = Q.y - p * Q.w;
      const double upr = U.x + p * U.z, upi = U.y + p * U.w, umr = U.x - p * U.z, umi = U.y - p * U.w;
      // a^E = -(F+ Q+ + i F- U-),  a^B = -(F+ U+ - i F- Q-)
      er -= f.x * qpr - f.y * umi;
      ei -= f.x * qpi + f.y * umr;
      br -= f.x * upr + f.y * qmi;
      bi -= f.x * upi - f.y * qmr;
    }
    for (int o = 16; o > 0; o >>= 1) {
      er += __shfl_xor_sync(0xffffffffu, er, o);
      ei += __shfl_xor_sync(0xffffffffu, ei, o);
      br += __shfl_xor_sync(0xffffffffu, br, o);
      bi += __shfl_xor_sync(0xffffffffu, bi, o);
    }
    if (lane == 0) {
      double2 &E = aE[base + (l - m)], &B = aB[base + (l - m)];
      if (add) { er += E.x; ei += E.y; br += B.x; bi += B.y; }
      E = l >= 2 ? make_double2(er, ei) : make_double2(0.0, 0.0);
      B = l >= 2 ? make_double2(br, bi) : make_double2(0.0, 0.0);
    }
  }
}

// spin-2 synthesis: Q_m, U_m on both rings of every pair; one CTA per m, a thread per ring pair
__global__ void __launch_bounds__(kPolThreads) spin2_synthesis_kernel(const Ctl *gate, const double2 *tab,
                                                                       const double2 *aE, const double2 *aB,
                                                                       int lmax, int RP, double4_32a *FSQ,
                                                                       double4_32a *FSU) {
  if (gate && gate->done) return;
  extern __shared__ double2 pol_sa[];
  const int m = blockIdx.x;
  const int Lm = lmax - m + 1;
  double2 *e = pol_sa, *b = pol_sa + Lm;
  const size_t base = idx_lm(lmax, m, m);
  for (int i = threadIdx.x; i < Lm; i += blockDim.x) {
    e[i] = aE[base + i];
    b[i] = aB[base + i];
  }
  __syncthreads();
  for (int k = threadIdx.x; k < RP; k += blockDim.x) {
    double qnr = 0, qni = 0, qsr = 0, qsi = 0, unr = 0, uni = 0, usr = 0, usi = 0;
    for (int i = (m < 2 ? 2 - m : 0); i < Lm; ++i) {
      const double2 f = tab[(base + i) * RP + k];
      const double p = (i & 1) ? -1.0 : 1.0;
      const double2 E = e[i], B = b[i];
      // north: Q = -(F+ E + i F- B), U = -(F+ B - i F- E); south: F+ -> p F+, F- -> -p F-
      const double aqr = f.x * E.x - f.y * B.y, aqi = f.x * E.y + f.y * B.x;   // F+ E + i F- B
      const double bqr = f.x * E.x + f.y * B.y, bqi = f.x * E.y - f.y * B.x;   // F+ E - i F- B
      const double aur = f.x * B.x + f.y * E.y, aui = f.x * B.y - f.y * E.x;   // F+ B - i F- E
      const double bur = f.x * B.x - f.y * E.y, bui = f.x * B.y + f.y * E.x;   // F+ B + i F- E
      qnr -= aqr; qni -= aqi;
      qsr -= p * bqr; qsi -= p * bqi;
      unr -= aur; uni -= aui;
      usr -= p * bur; usi -= p * bui;
    }
    FSQ[(size_t)m * RP + k] = make_double4_32a(qnr, qni, qsr, qsi);
    FSU[(size_t)m * RP + k] = make_double4_32a(unr, uni, usr, usi);
  }
}

// ---- double-float spin-2 Legendre stage
__device__ __forceinline__ float4 cdf(double re, double im) {   // complex double-float (re hi, re lo, im hi, im lo)
  return df_pair(df_from(re), df_from(im));
}
__device__ __forceinline__ float4 zero4() { return make_float4(0.f, 0.f, 0.f, 0.f); }

// (S, C) += (rS, rC), another lane's: error-free in S; FINE, both renormalised and one rounding
template <bool FINE>
__device__ __forceinline__ void lane_add(float &S, float &C, float rS, float rC) {
  if (FINE) {
    const dfl v = df_add2<true>(df_norm(S, C), df_norm(rS, rC));
    S = v.h;
    C = v.l;
  } else {
    comp_add(S, C, rS, rC);
  }
}

// Eight compensated sums over the warp: lane q ends with sum q >> 2 of its 8 (lanes 4 q .. 4 q + 3 hold sum q).
// Halves are exchanged on the way down (4 + 2 + 1 additions, then 2), all in double-float: in FP64, 40 additions
// on a pipe of 1/63 the rate took longer than a short row's products.
template <bool FINE>
__device__ __forceinline__ dfl warp_sum8_df(float (&S)[8], float (&C)[8]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16, n = 4; n >= 1; off >>= 1, n >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const float oS = up ? S[j] : S[j + n], oC = up ? C[j] : C[j + n];   // sent
      const float kS = up ? S[j + n] : S[j], kC = up ? C[j + n] : C[j];   // kept
      const float rS = __shfl_xor_sync(0xffffffffu, oS, off), rC = __shfl_xor_sync(0xffffffffu, oC, off);
      S[j] = kS;
      C[j] = kC;
      lane_add<FINE>(S[j], C[j], rS, rC);
    }
  }
#pragma unroll
  for (int off = 2; off >= 1; off >>= 1)
    lane_add<FINE>(S[0], C[0], __shfl_xor_sync(0xffffffffu, S[0], off), __shfl_xor_sync(0xffffffffu, C[0], off));
  return df_norm(S[0], C[0]);
}

// spin-2 analysis in double-float: a CTA takes lchunk values of l of one m, a
// warp two of them (l - m even, then odd) at a time, lanes over ring pairs.
// Shared memory holds, per ring pair, Q_N + Q_S, Q_N - Q_S, U_N + U_S, U_N - U_S
// (the two parities' combinations of the rings' coefficients).
// Bound by FP32 issue (16 compensated products a ring pair and row pair against
// 32 bytes of table and four shared loads); the table rows of the next two
// tiles of 32 ring pairs are in flight while one is summed. Chunks of l instead
// of a CTA per m keep every SM busy at any lmax. A CTA per m, FP64 sums over the
// warp and one step of loads ahead: 2.28 ms a launch at Nside 512 / lmax 1024 and
// 156 us at Nside 128 / lmax 256; now 1.51 ms and 47 us (1.80 and 54 before the
// loop over tiles was counted, without a search and moves a step).
template <bool FINE>
__global__ void __launch_bounds__(kPolThreads, 3) spin2_analysis_df_kernel(const Ctl *gate, const float4 *tab,
                                                                            const int *ls, const double4_32a *FTQ,
                                                                            const double4_32a *FTU, int lmax, int RP,
                                                                            int nk, int add, int lchunk, double h,
                                                                            double2 *aE, double2 *aB) {
  if (gate && gate->done) return;
  extern __shared__ float4 pol_dsm[];   // [4][nk] combinations, then [nk / 32] first l of each tile
  const int m = blockIdx.x;
  const int lbeg = m + blockIdx.y * lchunk, lend = min(lmax, lbeg + lchunk - 1);
  if (lbeg > lmax) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int ntile = (nk + 31) >> 5;
  int *tmin = reinterpret_cast<int *>(pol_dsm + 4 * nk);
  for (int t = warp; t < ntile; t += nw) {
    const int k = 32 * t + lane;
    const int mn = __reduce_min_sync(0xffffffffu, k < nk ? ls[(size_t)m * RP + k] : 1 << 30);
    if (lane == 0) tmin[t] = mn;
  }
  __syncthreads();
  int tf = 0;                           // the tiles any row of the chunk reads
  while (tf < ntile && tmin[tf] > lend + 1) ++tf;
  for (int k = 32 * tf + threadIdx.x; k < nk; k += blockDim.x) {
    f_parities<FINE>(FTQ[(size_t)m * RP + k], pol_dsm[k], pol_dsm[nk + k]);
    f_parities<FINE>(FTU[(size_t)m * RP + k], pol_dsm[2 * nk + k], pol_dsm[3 * nk + k]);
  }
  __syncthreads();
  const size_t base = idx_lm(lmax, m, m);
  for (int l = lbeg + 2 * warp; l <= lend; l += 2 * nw) {
    const bool has1 = l + 1 <= lmax;
    float S[8], C[8];   // [0..3]: l, [4..7]: l + 1
#pragma unroll
    for (int j = 0; j < 8; ++j) { S[j] = 0.f; C[j] = 0.f; }
    const float4 *row0 = tab + (base + (l - m)) * RP, *row1 = row0 + RP;
    int t0 = 0;                       // the first tile with a term of l or l + 1 (F+- = 0 below a ring pair's first l;
    while (t0 < ntile && tmin[t0] > l + 1) ++t0;   // towards the equator the first l falls)
    auto load = [&](int t, float4 &f0, float4 &f1) {
      const int k = 32 * t + lane;
      f0 = k < nk ? row0[k] : zero4();
      f1 = k < nk && has1 ? row1[k] : zero4();
    };
    auto term = [&](int t, float4 f0, float4 f1) {
      const int k = min(32 * t + lane, nk - 1);   // lanes past nk: zero table values
      const float4 A = pol_dsm[k], Bq = pol_dsm[nk + k], Cu = pol_dsm[2 * nk + k], Du = pol_dsm[3 * nk + k];
      // -a^E = F+ Q+ + i F- U-,  -a^B = F+ U+ - i F- Q-
      {   // l: Q+ = A, Q- = Bq, U+ = Cu, U- = Du
        const dfl fp = {f0.x, f0.y}, fm = {f0.z, f0.w}, fn = df_neg(fm);
        dot2_acc<FINE>(S[0], C[0], fp, dfl{A.x, A.y});
        dot2_acc<FINE>(S[0], C[0], fn, dfl{Du.z, Du.w});
        dot2_acc<FINE>(S[1], C[1], fp, dfl{A.z, A.w});
        dot2_acc<FINE>(S[1], C[1], fm, dfl{Du.x, Du.y});
        dot2_acc<FINE>(S[2], C[2], fp, dfl{Cu.x, Cu.y});
        dot2_acc<FINE>(S[2], C[2], fm, dfl{Bq.z, Bq.w});
        dot2_acc<FINE>(S[3], C[3], fp, dfl{Cu.z, Cu.w});
        dot2_acc<FINE>(S[3], C[3], fn, dfl{Bq.x, Bq.y});
      }
      {   // l + 1: Q+ = Bq, Q- = A, U+ = Du, U- = Cu
        const dfl fp = {f1.x, f1.y}, fm = {f1.z, f1.w}, fn = df_neg(fm);
        dot2_acc<FINE>(S[4], C[4], fp, dfl{Bq.x, Bq.y});
        dot2_acc<FINE>(S[4], C[4], fn, dfl{Cu.z, Cu.w});
        dot2_acc<FINE>(S[5], C[5], fp, dfl{Bq.z, Bq.w});
        dot2_acc<FINE>(S[5], C[5], fm, dfl{Cu.x, Cu.y});
        dot2_acc<FINE>(S[6], C[6], fp, dfl{Du.x, Du.y});
        dot2_acc<FINE>(S[6], C[6], fm, dfl{A.z, A.w});
        dot2_acc<FINE>(S[7], C[7], fp, dfl{Du.z, Du.w});
        dot2_acc<FINE>(S[7], C[7], fn, dfl{A.x, A.y});
      }
    };
    float4 f[2][2];
    if (t0 < ntile) load(t0, f[0][0], f[0][1]);
    if (t0 + 1 < ntile) load(t0 + 1, f[1][0], f[1][1]);
    for (int tb = t0; tb < ntile; tb += 2) {
#pragma unroll
      for (int d = 0; d < 2; ++d) {   // compile-time buffer indices
        const int t = tb + d;
        if (t >= ntile) break;
        term(t, f[d][0], f[d][1]);
        if (t + 2 < ntile) load(t + 2, f[d][0], f[d][1]);
      }
      if (((tb - t0) & 15) == 14) {   // 32 terms a sum (two a tile)
#pragma unroll
        for (int j = 0; j < 8; ++j) dot2_tidy(S[j], C[j]);
      }
    }
    const dfl v = warp_sum8_df<FINE>(S, C);
    if ((lane & 3) == 0) {   // sum lane / 4: E re, im, B re, im of l, then of l + 1
      const int q = lane >> 2, lq = l + (q >> 2);
      if (lq <= lend) {
        double &dst = reinterpret_cast<double *>((((q >> 1) & 1) ? aB : aE) + base + (lq - m))[q & 1];
        const double a = -h * df_to(v);   // h: LegArgs::fomega
        dst = lq >= 2 ? (add ? dst + a : a) : 0.0;
      }
    }
  }
}

// spin-2 synthesis in double-float: a CTA takes one m and blockDim.x ring pairs, a thread one of them.
// The eight products F+ E.re, F- B.im, F+ E.im, F- B.re, F+ B.re, F- E.im,
// F+ B.im, F- E.re are summed separately over even (S0) and odd (S1) l - m;
// the north ring takes even + odd, the south ring (parity (-1)^(l-m) for F+,
// the opposite for F-) even - odd.
// Bound by FP32 issue (80 instructions a row). Each lane copies its own table
// column into a shared ring of kSynDepth rows ahead with cp.async (no barrier:
// nobody else reads it), which holds the loads of a DRAM latency without the
// registers that a third CTA per SM needs. Four rows loaded at a time, a CTA per
// m: 1.65 ms a launch at Nside 512 / lmax 1024, 78 us at Nside 128 / lmax 256; now
// 1.41 ms and 46 us.
constexpr int kSynDepth = 8;   // rows in flight, even
__device__ __forceinline__ void cp_async16(float4 *dst, const float4 *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <bool FINE>
__global__ void __launch_bounds__(kPolThreads, 3) spin2_synthesis_df_kernel(const Ctl *gate, const float4 *tab,
                                                                             const int *ls, const double2 *aE,
                                                                             const double2 *aB, int lmax, int RP,
                                                                             double4_32a *FSQ, double4_32a *FSU) {
  if (gate && gate->done) return;
  extern __shared__ float4 pol_dsa[];   // [kSynDepth][blockDim.x] ring of rows, then [Lm + 1][2]: E, B as complex double-float
  const int m = blockIdx.x;
  const int Lm = lmax - m + 1;
  const size_t base = idx_lm(lmax, m, m);
  const int k = blockIdx.y * blockDim.x + threadIdx.x;
  float4 *ring = pol_dsa + threadIdx.x, *coef = pol_dsa + (size_t)kSynDepth * blockDim.x;
  const int nt = blockDim.x;
  // the warp's first row (its ring pairs' first l, at least l = 2), made even
  const int lw = __reduce_min_sync(0xffffffffu, k < RP ? ls[(size_t)m * RP + k] : 1 << 30);
  const int i0 = max(m < 2 ? 2 - m : 0, lw - m) & ~1;
  const float4 *col = tab + base * RP + min(k, RP - 1);
  auto fetch = [&](int i, int j) {   // rows i and i + 1 into places j, j + 1 (one group, also when there is none left)
    if (i < Lm) cp_async16(ring + (size_t)j * nt, col + (size_t)i * RP);
    if (i + 1 < Lm) cp_async16(ring + (size_t)(j + 1) * nt, col + (size_t)(i + 1) * RP);
    cp_commit();
  };
#pragma unroll
  for (int j = 0; j < kSynDepth; j += 2) fetch(i0 + j, j);
  for (int i = threadIdx.x; i < Lm; i += nt) {
    coef[2 * i] = cdf(aE[base + i].x, aE[base + i].y);
    coef[2 * i + 1] = cdf(aB[base + i].x, aB[base + i].y);
  }
  __syncthreads();
  float S0[8], C0[8], S1[8], C1[8];   // compile-time indices: the sums stay in registers
#pragma unroll
  for (int j = 0; j < 8; ++j) { S0[j] = 0.f; C0[j] = 0.f; S1[j] = 0.f; C1[j] = 0.f; }
  auto accum = [&](int i, float4 f, float(&Sa)[8], float(&Ca)[8]) {
    const dfl fp = {f.x, f.y}, fm = {f.z, f.w};
    const float4 E = coef[2 * i], Bv = coef[2 * i + 1];
    const dfl er = {E.x, E.y}, ei = {E.z, E.w}, br = {Bv.x, Bv.y}, bi = {Bv.z, Bv.w};
    dot2_acc<FINE>(Sa[0], Ca[0], fp, er);
    dot2_acc<FINE>(Sa[1], Ca[1], fm, bi);
    dot2_acc<FINE>(Sa[2], Ca[2], fp, ei);
    dot2_acc<FINE>(Sa[3], Ca[3], fm, br);
    dot2_acc<FINE>(Sa[4], Ca[4], fp, br);
    dot2_acc<FINE>(Sa[5], Ca[5], fm, ei);
    dot2_acc<FINE>(Sa[6], Ca[6], fp, bi);
    dot2_acc<FINE>(Sa[7], Ca[7], fm, er);
  };
  const int istart = m < 2 ? 2 - m : 0;   // rows of l < 2 hold zeros; their coefficients may be anything
  for (int ib = i0; ib < Lm; ib += kSynDepth) {
#pragma unroll
    for (int j = 0; j < kSynDepth; j += 2) {   // compile-time places in the ring
      const int i = ib + j;
      if (i >= Lm) break;
      cp_wait<kSynDepth / 2 - 1>();
      const float4 f0 = ring[(size_t)j * nt], f1 = ring[(size_t)(j + 1) * nt];
      if (i >= istart) accum(i, f0, S0, C0);
      if (i + 1 < Lm && i + 1 >= istart) accum(i + 1, f1, S1, C1);
      fetch(i + kSynDepth, j);          // into the places just used
    }
    if (((ib - i0) & 31) == 24) {   // 16 terms a sum
#pragma unroll
      for (int j = 0; j < 8; ++j) { dot2_tidy(S0[j], C0[j]); dot2_tidy(S1[j], C1[j]); }
    }
  }
  cp_wait<0>();
  if (k >= RP) return;
  dfl e[8], o[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    e[j] = df_norm(S0[j], C0[j]);
    o[j] = df_norm(S1[j], C1[j]);
  }
  // sums over both parities (p) and their difference (d)
  auto p = [&](int j) { return df_add2<FINE>(e[j], o[j]); };
  auto d = [&](int j) { return df_add2<FINE>(e[j], df_neg(o[j])); };
  auto put = [](dfl x, dfl y) { return df_pack(df_neg(df_add2<FINE>(x, y))); };
  // north: Q = -(F+ E + i F- B), U = -(F+ B - i F- E); south: F+ -> p F+, F- -> -p F-
  FSQ[(size_t)m * RP + k] = make_double4_32a(put(p(0), df_neg(p(1))), put(p(2), p(3)), put(d(0), d(1)),
                                             put(d(2), df_neg(d(3))));
  FSU[(size_t)m * RP + k] = make_double4_32a(put(p(4), p(5)), put(p(6), df_neg(p(7))), put(d(4), df_neg(d(5))),
                                             put(d(6), d(7)));
}

// Eq. 3 per pixel with the 3 x 3 messenger and the chi^2 partials (sum r^T W r and r^T (N + (lambda-1) tau)^-1 r).
// The gains (N + (lambda - 1) tau)^-1 depend on lambda only: each block keeps those of its pixels (the grid
// is fixed, so a block always owns the same pixels) with the lambda they belong to, and recomputes them,
// divisions on the FP64 pipe, only when lambda changes. Bound by that pipe: 22 instructions a pixel with both
// products W r and G r formed once (37 with every term of the sums by itself: 23 us at Nside 128).
__global__ void __launch_bounds__(kPolThreads) pol_pixel_kernel(const Ctl *ctl, long long npix, double tau,
                                                                 const double *s, const double *d, const double4_32a *w,
                                                                 double4_32a *gain, double *gainlam, double *u,
                                                                 double *part) {
  __shared__ double red[2][kPolThreads / 32];
  if (ctl->done) return;
  const double lam = ctl->lambda, c = (lam - 1.0) * tau, lt = lam * tau;
  const bool fresh = gainlam[blockIdx.x] == lam;   // this block's gains are already at this lambda
  double c2n = 0.0, c2l = 0.0;
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < npix; p += (long long)gridDim.x * blockDim.x) {
    const double4_32a W = w[p];   // (w_T, w_QQ, w_QU, w_UU)
    const double rt = d[p] - s[p], rq = d[npix + p] - s[npix + p], ru = d[2 * npix + p] - s[2 * npix + p];
    double gt, g11, g12, g22;
    if (fresh) {
      const double4_32a G = gain[p];
      gt = G.x; g11 = G.y; g12 = G.z; g22 = G.w;
    } else {
      gt = W.x / (1.0 + c * W.x);
      const double a11 = 1.0 + c * W.y, a12 = c * W.z, a22 = 1.0 + c * W.w;
      const double det = a11 * a22 - a12 * a12;
      const double i11 = a22 / det, i12 = -a12 / det, i22 = a11 / det;
      g11 = W.y * i11 + W.z * i12;
      g12 = W.y * i12 + W.z * i22;
      g22 = W.z * i12 + W.w * i22;
      gain[p] = make_double4_32a(gt, g11, g12, g22);
    }
    // G r and W r once each: the update is lambda tau G r, the partial sums r.(W r) and r.(G r)
    const double at = gt * rt, aq = fma(g12, ru, g11 * rq), au = fma(g22, ru, g12 * rq);
    const double bt = W.x * rt, bq = fma(W.z, ru, W.y * rq), bu = fma(W.w, ru, W.z * rq);
    u[p] = lt * at;
    u[npix + p] = lt * aq;
    u[2 * npix + p] = lt * au;
    c2n = fma(rt, bt, fma(rq, bq, fma(ru, bu, c2n)));
    c2l = fma(rt, at, fma(rq, aq, fma(ru, au, c2l)));
  }
  for (int o = 16; o > 0; o >>= 1) {
    c2n += __shfl_xor_sync(0xffffffffu, c2n, o);
    c2l += __shfl_xor_sync(0xffffffffu, c2l, o);
  }
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = c2n; red[1][threadIdx.x >> 5] = c2l; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0;
    for (int i = 0; i < kPolThreads / 32; ++i) { a += red[0][i]; b += red[1][i]; }
    part[2 * blockIdx.x] = a;
    part[2 * blockIdx.x + 1] = b;
    if (!fresh) gainlam[blockIdx.x] = lam;   // after the barrier: every gain of the block is written
  }
}

// Eq. 4 with the (T, E) block and B, the prior chi^2 of the input state, increment and norm per m. Bound by the FP64
// pipe, so one division for the block's four elements. A product with 1 / det rounds once more than a quotient, which an
// iteration at high signal to noise takes up 1 / (1 - m11) times (T 1.45 times less exact at Nside 8): the elements next
// to 1 are formed from their difference to it. Every element a quotient: 3 % of the T + P solve at Nside 128
__global__ void __launch_bounds__(128) pol_eq4_kernel(const Ctl *ctl, int lmax, long long nalm, double tau,
                                                       double omega, const double *cls, const double2 *ta,
                                                       double2 *s, double *m_part) {
  __shared__ double red[3][4];
  if (ctl->done) return;
  const int m = blockIdx.x;
  const double k = ctl->lambda * tau * omega;
  const double wgt = (m == 0) ? 1.0 : 2.0;
  const double *TT = cls, *EE = cls + (lmax + 1), *BB = cls + 2 * (lmax + 1), *TE = cls + 3 * (lmax + 1);
  double c2 = 0.0, inc = 0.0, nrm = 0.0;
  for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
    const size_t q = idx_lm(lmax, l, m);
    const double2 sT = s[q], sE = s[nalm + q], sB = s[2 * nalm + q];
    const double2 tT = make_double2(sT.x + ta[q].x, sT.y + ta[q].y);
    const double2 tE = make_double2(sE.x + ta[nalm + q].x, sE.y + ta[nalm + q].y);
    const double2 tB = make_double2(sB.x + ta[2 * nalm + q].x, sB.y + ta[2 * nalm + q].y);
    const double tt = TT[l], ee = EE[l], bb = BB[l], te = TE[l];
    // S (S + k)^-1 on (T, E)
    const double a11 = tt + k, a12 = te, a22 = ee + k, det = a11 * a22 - a12 * a12;
    double m11, m12, m21, m22;
    if (has_reciprocal(det)) {   // S (S + k)^-1 = 1 - k (S + k)^-1
      const double rd = 1.0 / det, c = k * rd, x11 = c * a22, x22 = c * a11;
      m12 = m21 = c * te;
      m11 = x11 < 0.5 ? 1.0 - x11 : (tt * a22 - te * te) * rd;
      m22 = x22 < 0.5 ? 1.0 - x22 : (ee * a11 - te * te) * rd;
    } else {
      m11 = (tt * a22 - te * a12) / det;
      m12 = (-tt * a12 + te * a11) / det;
      m21 = (te * a22 - ee * a12) / det;
      m22 = (-te * a12 + ee * a11) / det;
    }
    const double fb = bb > 0.0 ? bb / (bb + k) : 0.0;
    const double2 nT = make_double2(m11 * tT.x + m12 * tE.x, m11 * tT.y + m12 * tE.y);
    const double2 nE = make_double2(m21 * tT.x + m22 * tE.x, m21 * tT.y + m22 * tE.y);
    const double2 nB = make_double2(fb * tB.x, fb * tB.y);
    // prior chi^2 of the input state
    const double sdet = tt * ee - te * te;
    double qf = 0.0;
    if (sdet > 0.0) {
      qf = (ee * (sT.x * sT.x + sT.y * sT.y) - 2.0 * te * (sT.x * sE.x + sT.y * sE.y) +
            tt * (sE.x * sE.x + sE.y * sE.y)) / sdet;
    } else if (tt > 0.0) {
      qf = (sT.x * sT.x + sT.y * sT.y) / tt;
    }
    if (bb > 0.0) qf += (sB.x * sB.x + sB.y * sB.y) / bb;
    c2 += wgt * qf;
    const double d1x = nT.x - sT.x, d1y = nT.y - sT.y, d2x = nE.x - sE.x, d2y = nE.y - sE.y;
    const double d3x = nB.x - sB.x, d3y = nB.y - sB.y;
    inc += wgt * (d1x * d1x + d1y * d1y + d2x * d2x + d2y * d2y + d3x * d3x + d3y * d3y);
    nrm += wgt * (nT.x * nT.x + nT.y * nT.y + nE.x * nE.x + nE.y * nE.y + nB.x * nB.x + nB.y * nB.y);
    s[q] = nT;
    s[nalm + q] = nE;
    s[2 * nalm + q] = nB;
  }
  for (int o = 16; o > 0; o >>= 1) {
    c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    inc += __shfl_xor_sync(0xffffffffu, inc, o);
    nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
  }
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = c2; red[1][threadIdx.x >> 5] = inc; red[2][threadIdx.x >> 5] = nrm; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0.0, b = 0.0, e = 0.0;
    for (int i = 0; i < 4; ++i) { a += red[0][i]; b += red[1][i]; e += red[2][i]; }
    m_part[3 * m] = a;
    m_part[3 * m + 1] = b;
    m_part[3 * m + 2] = e;
  }
}

struct Pol : wf_pol_s {
  Plan *P = nullptr;   // scalar plan: geometry, tables, the T channel's Fourier buffers and stream
  int nside = 0, lmax = 0, RP = 0;
  long long npix = 0, nalm = 0, n_obs = 0;
  double tau = 0.0, omega = 0.0;
  wf_options opt{};
  std::vector<double> h_tt;
  double2 *d_tab = nullptr;                       // (F+, F-) [nalm][RP]: double2, or float4 double-float when df
  bool df = false;                                // double-float spin-2 stage (WF_PREC_FP64 plans)
  double *d_cls = nullptr;                        // [4][lmax+1] TT, EE, BB, TE
  double4_32a *d_w = nullptr;                         // [npix] (w_T, w_QQ, w_QU, w_UU)
  double4_32a *d_gain = nullptr;                      // [npix] cached 3 x 3 gains (g_T, g_QQ, g_QU, g_UU)
  double *d_gainlam = nullptr;                    // [kPixBlocks] lambda of each block's cached gains
  double *d_d = nullptr, *d_map = nullptr, *d_u = nullptr;   // [3][npix]
  double2 *d_s = nullptr, *d_ta = nullptr;        // [3][nalm]
  double4_32a *d_FSQ = nullptr, *d_FSU = nullptr, *d_FTQ = nullptr, *d_FTU = nullptr;
  double *d_part = nullptr, *d_m_part = nullptr;
  Ctl *d_ctl = nullptr, *h_ctl = nullptr;
  wf_iter_record *d_hist = nullptr;
  int hist_cap = 0;
  cudaGraphExec_t graph = nullptr;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  std::vector<void *> allocs;

  ~Pol() override {
    if (graph) cudaGraphExecDestroy(graph);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
    if (h_ctl) cudaFreeHost(h_ctl);
    for (void *p : allocs) cudaFree(p);
    if (P) wf_plan_destroy(P);
  }
  wf_status dalloc(void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) { *p = nullptr; return cuda_status(e, "cudaMalloc (polarisation)"); }
    allocs.push_back(*p);
    return WF_OK;
  }
  cudaStream_t stream() const { return P->run_stream(); }
  // (T, E, B) a_lm -> (T, Q, U) maps, and back (the adjoint), on the plan's kernels and the spin-2 stage
  void synth(cudaStream_t s, const double2 *alm, double *map, const Ctl *gate) const;
  void analysis(cudaStream_t s, const double *map, double2 *alm, const Ctl *gate) const;
  void enqueue_iteration(cudaStream_t s);
};

void Pol::synth(cudaStream_t s, const double2 *alm, double *map, const Ctl *gate) const {
  LegArgs la = P->leg_args();
  la.lsht = lmax;
  la.alm_in = alm;
  la.gate = gate;
  P->launch_leg(la, s, LEG_SYNTH);                                    // T -> the plan's FS
  if (df) {
    auto kernel = fine_steps(RP) ? spin2_synthesis_df_kernel<true> : spin2_synthesis_df_kernel<false>;
    raise_smem_cap(reinterpret_cast<const void *>(kernel));
    // half of the ring pairs a CTA up to 256 of them: enough CTAs where few values of m do not fill the chip,
    // and the coefficients (whose conversion is FP64 work) read by few
    const int nt = std::min(kPolThreads, std::max(32, (RP / 2 + 31) / 32 * 32));
    const dim3 grid(lmax + 1, (RP + nt - 1) / nt);
    kernel<<<grid, nt, sizeof(float4) * (kSynDepth * nt + 2 * (size_t)(lmax + 1)), s>>>(
        gate, reinterpret_cast<const float4 *>(d_tab), P->d_ls, alm + nalm, alm + 2 * nalm, lmax, RP, d_FSQ, d_FSU);
  } else {
    raise_smem_cap(reinterpret_cast<const void *>(spin2_synthesis_kernel));
    spin2_synthesis_kernel<<<lmax + 1, kPolThreads, sizeof(double2) * 2 * (lmax + 1), s>>>(
        gate, d_tab, alm + nalm, alm + 2 * nalm, lmax, RP, d_FSQ, d_FSU);
  }
  const double4_32a *fs[3] = {P->d_FS, d_FSQ, d_FSU};
  RingArgs ra[3];
  RingDfArgs rd[3];
  for (int c = 0; c < 3; ++c) {
    ra[c] = P->ring_args();
    ra[c].lsht = lmax;
    ra[c].FS = fs[c];
    ra[c].map_out = map + (size_t)c * npix;
    ra[c].gate = gate;
    rd[c] = P->ringdf_args();
  }
  P->launch_rng_maps(ra, rd, 3, s, RING_SYNTH);
}

void Pol::analysis(cudaStream_t s, const double *map, double2 *alm, const Ctl *gate) const {
  double4_32a *ft[3] = {P->d_FT, d_FTQ, d_FTU};
  RingArgs ra[3];
  RingDfArgs rd[3];
  for (int c = 0; c < 3; ++c) {
    ra[c] = P->ring_args();
    ra[c].lsht = lmax;
    ra[c].FT = ft[c];
    ra[c].map_in = map + (size_t)c * npix;
    ra[c].gate = gate;
    rd[c] = P->ringdf_args();
  }
  P->launch_rng_maps(ra, rd, 3, s, RING_ANALYSIS);
  LegArgs la = P->leg_args();
  la.lsht = lmax;
  la.alm = alm;
  la.gate = gate;
  P->launch_leg(la, s, LEG_ANALYSIS);                                 // T
  for (int k0 = 0; k0 < RP; k0 += kSpin2Pairs) {
    const int nk = std::min(kSpin2Pairs, RP - k0), add = k0 > 0;
    if (df) {
      auto kernel = fine_steps(RP) ? spin2_analysis_df_kernel<true> : spin2_analysis_df_kernel<false>;
      raise_smem_cap(reinterpret_cast<const void *>(kernel));
      // 64 values of l a CTA (four row pairs a warp), 16 where lmax leaves few chunks
      const int lchunk = lmax >= 256 ? 64 : 16;
      const dim3 grid(lmax + 1, (lmax + lchunk) / lchunk);
      kernel<<<grid, kPolThreads, sizeof(float4) * 4 * nk + sizeof(int) * ((nk + 31) / 32), s>>>(
          gate, reinterpret_cast<const float4 *>(d_tab) + k0, P->d_ls + k0, d_FTQ + k0, d_FTU + k0, lmax, RP, nk, add,
          lchunk, la.fomega, alm + nalm, alm + 2 * nalm);
    } else {
      raise_smem_cap(reinterpret_cast<const void *>(spin2_analysis_kernel));
      spin2_analysis_kernel<<<lmax + 1, kPolThreads, sizeof(double4_32a) * 2 * nk, s>>>(
          gate, d_tab + k0, d_FTQ + k0, d_FTU + k0, lmax, RP, nk, add, alm + nalm, alm + 2 * nalm);
    }
  }
}

void Pol::enqueue_iteration(cudaStream_t s) {
  synth(s, d_s, d_map, d_ctl);
  pol_pixel_kernel<<<kPixBlocks, kPolThreads, 0, s>>>(d_ctl, npix, tau, d_map, d_d, d_w, d_gain, d_gainlam, d_u,
                                                       d_part);
  analysis(s, d_u, d_ta, d_ctl);
  pol_eq4_kernel<<<lmax + 1, 128, 0, s>>>(d_ctl, lmax, nalm, tau, omega, d_cls, d_ta, d_s, d_m_part);
  const CtlMap c{d_ctl, d_part, d_m_part, P->d_cl, d_hist, hist_cap};
  launch_control(&c, 1, kPixBlocks, lmax, s);
}

}  // namespace
}  // namespace wfk

using namespace wfk;

#define PO_CUDA(call)                                      \
  do {                                                     \
    cudaError_t e_ = (call);                               \
    if (e_ != cudaSuccess) return cuda_status(e_, #call);  \
  } while (0)

extern "C" {

wf_status wf_pol_create(int nside, int lmax, const double *cls, const double *noise, const uint8_t *mask_t,
                        const uint8_t *mask_p, const wf_options *opt, wf_pol_t *out) {
  if (!out || !cls || !noise) { set_error("wf_pol_create: NULL argument"); return WF_EINVAL; }
  *out = nullptr;
  wf_options o;
  if (opt) o = *opt;
  else wf_options_default(&o);
  if (o.precision == WF_PREC_MIXED) {
    set_error("wf_pol_create: polarisation runs on the FP64 paths (WF_PREC_FP64, WF_PREC_FP64_NATIVE)");
    return WF_EINVAL;
  }
  o.band_limit = 0;
  if (nside < 1 || nside > 2048 || (nside & (nside - 1)) || lmax < 0 || lmax > 4 * nside) {
    set_error("wf_pol_create: nside must be a power of two in [1, 2048] and 0 <= lmax <= 4 nside");
    return WF_EINVAL;
  }
  const long long npix = 12LL * nside * nside;
  const size_t nalm = (size_t)(lmax + 1) * (lmax + 2) / 2;
  const size_t tab_bytes = nalm * (size_t)(2 * nside) * sizeof(double2);
  if (tab_bytes > kSpin2TableMax) {
    set_error("wf_pol_create: the spin-2 table would take " + std::to_string(tab_bytes) + " bytes (limit 64 GiB)");
    return WF_EINVAL;
  }
  for (int c = 0; c < 3; ++c)
    for (int l = 0; l <= lmax; ++l)
      if (!std::isfinite(cls[c * (lmax + 1) + l]) || cls[c * (lmax + 1) + l] < 0.0) {
        set_error("wf_pol_create: C_TT, C_EE, C_BB must be finite and >= 0");
        return WF_EINVAL;
      }
  for (int l = 0; l <= lmax; ++l) {
    const double tt = cls[l], ee = cls[lmax + 1 + l], te = cls[3 * (lmax + 1) + l];
    if (!std::isfinite(te) || te * te > tt * ee * (1.0 + 1e-12)) {
      set_error("wf_pol_create: C_TE must satisfy C_TE^2 <= C_TT C_EE");
      return WF_EINVAL;
    }
  }
  // inverse noise per pixel and the messenger covariance
  std::vector<double4_32a> w(npix);
  double tau = INFINITY;
  long long n_obs = 0;
  for (long long p = 0; p < npix; ++p) {
    const double nt = noise[4 * p], nqq = noise[4 * p + 1], nqu = noise[4 * p + 2], nuu = noise[4 * p + 3];
    double4_32a v = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    if (!mask_t || mask_t[p]) {
      if (!std::isfinite(nt) || !(nt > 0.0)) { set_error("wf_pol_create: T noise must be > 0 where observed"); return WF_EINVAL; }
      v.x = 1.0 / nt;
      tau = std::min(tau, nt);
      ++n_obs;
    }
    if (!mask_p || mask_p[p]) {
      const double det = nqq * nuu - nqu * nqu;
      if (!std::isfinite(det) || !(nqq > 0.0) || !(det > 0.0)) {
        set_error("wf_pol_create: the Q-U noise block must be positive definite where observed");
        return WF_EINVAL;
      }
      v.y = nuu / det;
      v.z = -nqu / det;
      v.w = nqq / det;
      tau = std::min(tau, 0.5 * (nqq + nuu) - std::sqrt(0.25 * (nqq - nuu) * (nqq - nuu) + nqu * nqu));
      n_obs += 2;
    }
    w[p] = v;
  }
  if (n_obs == 0) { set_error("wf_pol_create: no observed component"); return WF_EINVAL; }
  Pol *Q = new (std::nothrow) Pol();
  if (!Q) { set_error("out of host memory"); return WF_ENOMEM; }
  Q->opt = o;
  std::vector<double> unit(npix, 1.0);
  wf_plan_t p = nullptr;
  wf_status st = wf_plan_create(nside, lmax, cls, unit.data(), nullptr, &o, &p);   // geometry, tables, T channel
  if (st) { delete Q; return st; }
  Q->P = static_cast<Plan *>(p);
  Q->nside = nside;
  Q->lmax = lmax;
  Q->RP = Q->P->RP;
  Q->npix = npix;
  Q->nalm = (long long)nalm;
  Q->tau = tau;
  Q->omega = Q->P->omega;
  Q->n_obs = n_obs;
  Q->df = o.precision == WF_PREC_FP64;
  const size_t nF = (size_t)(lmax + 1) * Q->RP;
  if ((st = Q->dalloc((void **)&Q->d_tab, tab_bytes)) || (st = Q->dalloc((void **)&Q->d_cls, sizeof(double) * 4 * (lmax + 1))) ||
      (st = Q->dalloc((void **)&Q->d_w, sizeof(double4_32a) * npix)) ||
      (st = Q->dalloc((void **)&Q->d_gain, sizeof(double4_32a) * npix)) ||
      (st = Q->dalloc((void **)&Q->d_gainlam, sizeof(double) * kPixBlocks)) ||
      (st = Q->dalloc((void **)&Q->d_d, sizeof(double) * 3 * npix)) ||
      (st = Q->dalloc((void **)&Q->d_map, sizeof(double) * 3 * npix)) ||
      (st = Q->dalloc((void **)&Q->d_u, sizeof(double) * 3 * npix)) ||
      (st = Q->dalloc((void **)&Q->d_s, sizeof(double2) * 3 * nalm)) ||
      (st = Q->dalloc((void **)&Q->d_ta, sizeof(double2) * 3 * nalm)) ||
      (st = Q->dalloc((void **)&Q->d_FSQ, sizeof(double4_32a) * nF)) || (st = Q->dalloc((void **)&Q->d_FSU, sizeof(double4_32a) * nF)) ||
      (st = Q->dalloc((void **)&Q->d_FTQ, sizeof(double4_32a) * nF)) || (st = Q->dalloc((void **)&Q->d_FTU, sizeof(double4_32a) * nF)) ||
      (st = Q->dalloc((void **)&Q->d_part, sizeof(double) * 2 * kPixBlocks)) ||
      (st = Q->dalloc((void **)&Q->d_m_part, sizeof(double) * 3 * (lmax + 1))) ||
      (st = Q->dalloc((void **)&Q->d_ctl, sizeof(Ctl))) ||
      (st = Q->dalloc((void **)&Q->d_hist, sizeof(wf_iter_record) * (size_t)(o.max_iter + 1)))) {
    delete Q;
    return st;
  }
  Q->hist_cap = o.max_iter + 1;
  cudaStream_t s = Q->stream();
  cudaError_t e = cudaMemcpyAsync(Q->d_cls, cls, sizeof(double) * 4 * (lmax + 1), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(Q->d_w, w.data(), sizeof(double4_32a) * npix, cudaMemcpyHostToDevice, s);
  const std::vector<double> no_gains(kPixBlocks, -1.0);   // no gains cached yet: lambda >= 1 never equals -1
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(Q->d_gainlam, no_gains.data(), sizeof(double) * kPixBlocks, cudaMemcpyHostToDevice, s);
  // the ring stage never writes the equator pair's south slot: it must read as zero
  if (e == cudaSuccess) e = cudaMemsetAsync(Q->d_FTQ, 0, sizeof(double4_32a) * nF, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(Q->d_FTU, 0, sizeof(double4_32a) * nF, s);
  if (e == cudaSuccess) {
    const long long n = (long long)(lmax + 1) * Q->RP;
    spin2_table_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(Q->P->d_x, Q->P->d_rec, Q->P->d_ls, Q->P->d_sv,
                                                                  lmax, Q->RP, Q->d_tab, Q->df ? 1 : 0);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMallocHost((void **)&Q->h_ctl, sizeof(Ctl));
  if (e == cudaSuccess) e = cudaEventCreate(&Q->ev0);
  if (e == cudaSuccess) e = cudaEventCreate(&Q->ev1);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) { st = cuda_status(e, "wf_pol_create setup"); delete Q; return st; }
  *out = Q;
  return WF_OK;
}

wf_status wf_pol_destroy(wf_pol_t pol) {
  if (!pol) return WF_OK;
  Pol *Q = static_cast<Pol *>(pol);
  cudaStreamSynchronize(Q->stream());
  delete Q;
  return WF_OK;
}

wf_status wf_pol_alm2map(wf_pol_t pol, const double *alm_dev, double *map_dev) {
  if (!pol || !alm_dev || !map_dev) { set_error("wf_pol_alm2map: NULL argument"); return WF_EINVAL; }
  Pol *Q = static_cast<Pol *>(pol);
  Q->synth(Q->stream(), reinterpret_cast<const double2 *>(alm_dev), map_dev, nullptr);
  PO_CUDA(cudaGetLastError());
  return WF_OK;
}

wf_status wf_pol_map2alm(wf_pol_t pol, const double *map_dev, double *alm_dev) {
  if (!pol || !alm_dev || !map_dev) { set_error("wf_pol_map2alm: NULL argument"); return WF_EINVAL; }
  Pol *Q = static_cast<Pol *>(pol);
  Q->analysis(Q->stream(), map_dev, reinterpret_cast<double2 *>(alm_dev), nullptr);
  PO_CUDA(cudaGetLastError());
  return WF_OK;
}

wf_status wf_pol_solve(wf_pol_t pol, const double *d, int d_on_device, double *alm_out, int alm_on_device,
                       wf_stats *stats, wf_iter_record *records, int max_records, int *n_records) {
  if (!pol || !d || !alm_out) { set_error("wf_pol_solve: NULL argument"); return WF_EINVAL; }
  Pol *Q = static_cast<Pol *>(pol);
  Plan *P = Q->P;
  cudaStream_t s = Q->stream();
  PO_CUDA(cudaEventRecord(Q->ev0, s));
  PO_CUDA(cudaMemcpyAsync(Q->d_d, d, sizeof(double) * 3 * Q->npix,
                          d_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  PO_CUDA(cudaMemsetAsync(Q->d_s, 0, sizeof(double2) * 3 * Q->nalm, s));
  // lambda from the ratio C_TT / (tau Omega) at l_iter (Sect. 3 names C_TT), clamped to >= 1
  const double lam0 = (Q->opt.cooling && Q->opt.l_iter0 <= Q->lmax)
                          ? std::max(1.0, P->h_cl[Q->opt.l_iter0] / (Q->tau * Q->omega)) : 1.0;
  Ctl c = P->make_ctl(1, lam0, Q->lmax, 0);
  c.band_limit = 0;
  c.tau = Q->tau;
  c.sigma_chi2 = std::sqrt(2.0 * (double)Q->n_obs);
  *Q->h_ctl = c;
  PO_CUDA(cudaMemcpyAsync(Q->d_ctl, Q->h_ctl, sizeof(Ctl), cudaMemcpyHostToDevice, s));
  const int gi = Q->opt.graph_iters;
  if (!Q->graph) {
    const wf_status gs = capture_graph(s, gi, &Q->graph, "graph of the polarised solve",
                                       [&] { Q->enqueue_iteration(s); });
    if (gs) return gs;
  }
  const int max_launch = (Q->opt.max_iter + gi - 1) / gi + 1;
  for (int it = 0; it < max_launch; ++it) {
    PO_CUDA(cudaGraphLaunch(Q->graph, s));
    PO_CUDA(cudaMemcpyAsync(Q->h_ctl, Q->d_ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
    PO_CUDA(cudaStreamSynchronize(s));
    if (Q->h_ctl->done) break;
  }
  PO_CUDA(cudaMemcpyAsync(alm_out, Q->d_s, sizeof(double2) * 3 * Q->nalm,
                          alm_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
  PO_CUDA(cudaEventRecord(Q->ev1, s));
  const Ctl fin = *Q->h_ctl;
  wf_iter_record last{};
  if (fin.iter > 0)
    PO_CUDA(cudaMemcpyAsync(&last, Q->d_hist + (fin.iter - 1), sizeof(last), cudaMemcpyDeviceToHost, s));
  int nrec = 0;
  if (records && max_records > 0) {
    nrec = fin.iter < max_records ? fin.iter : max_records;
    if (nrec > 0)
      PO_CUDA(cudaMemcpyAsync(records, Q->d_hist, sizeof(wf_iter_record) * nrec, cudaMemcpyDeviceToHost, s));
  }
  PO_CUDA(cudaStreamSynchronize(s));
  if (n_records) *n_records = nrec;
  P->fs_valid = false;
  if (stats) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, Q->ev0, Q->ev1);
    *stats = wf_stats{};
    stats->iters = fin.iter;
    stats->converged = fin.converged;
    stats->levels = fin.level + 1;
    stats->lmax_sht_final = fin.lsht;
    stats->lambda_final = fin.lambda;
    stats->chi2_prior = last.chi2_prior;
    stats->chi2_noise = last.chi2_noise;
    stats->chi2 = last.chi2_prior + last.chi2_noise;
    stats->chi2_per_dof = stats->chi2 / (double)Q->n_obs;
    stats->rel_increment = fin.last_rel;
    stats->ms_device = ms;
    stats->rel_posterior_grad = -1.0;
  }
  if (fin.numeric) { set_error("wf_pol_solve: chi^2 is not finite"); return WF_ENUMERIC; }
  if (!fin.converged) { set_error("wf_pol_solve: max_iter reached before the stop rule"); return WF_ENOTCONVERGED; }
  return WF_OK;
}

}  // extern "C"
