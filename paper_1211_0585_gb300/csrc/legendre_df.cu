// Legendre stage in double-float arithmetic: FP64-accurate results from the
// FP32 pipe.
//
// GB300 runs FP64 FMAs at 1/63 of the FP32 rate, and the FP64 Legendre kernel
// (legendre.cu) is bound by that pipe. Here every value of the inner loops is
// an unevaluated sum of two floats (hi + lo, 48 significant bits) and every
// operation is built from error-free transformations:
//   two_prod(a, b)  p = a b, e = fma(a, b, -p)           (exact)
//   two_sum(a, b)   s = a + b, e = (a - (s - bb)) + (b - bb), bb = s - a  (exact)
// Sums over rings and over l use the compensated dot product of Ogita, Rump
// and Oishi ("Accurate sum and dot product", SIAM J. Sci. Comput. 26, 2005):
// the running sum in a float S with its exact rounding errors collected in a
// float C, which is as accurate as a dot product in twice the working
// precision.
//
// The recurrence is rescaled so that it needs one double-float product and one
// double-float subtraction per step: with lambda_l = g_l mu_l, g_m = g_{m+1} = 1,
// g_l = b_l g_{l-2},
//     mu_l = A_l x mu_{l-1} - mu_{l-2},   A_l = a_l g_{l-1} / g_l,
// (g_l stays within [2^-2.6, 2^0.2] for lmax <= 4096, so mu has lambda's range).
// The factor g_l is applied in double after the cross-ring reduction (analysis)
// and folded into the harmonic coefficients before synthesis.
//
// Terms with |lambda_lm(x)| < 2^-60 (the evanescent region near the poles) are
// not evaluated; they lie below the 48-bit precision of any sum they enter.
//
// Where the plan holds lambda_lm(x_k) precomputed, legendre_tab.cu reads it
// instead; the table is built here (FP64 recurrence, stored as double-float).
#include <cuda_runtime.h>

#include "df.cuh"
#include "start_values.cuh"
#include "wf_internal.h"

namespace wfk {

constexpr int kNoStartD = 1 << 30;
// ring pairs whose analysis state is held in shared memory at once: four a thread
template <int NT> constexpr int kAnaChunk = 4 * NT;

__device__ __forceinline__ size_t alm_idx_d(int lmax, int l, int m) {
  return (size_t)m * (2 * lmax + 1 - m) / 2 + l;
}

// Sixteen compensated sums over the warp's lanes by exchanging halves: lanes 2 q and 2 q + 1 end with sum q
__device__ __forceinline__ void warp_sums16(float (&S)[16], float (&C)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int off = 16, n = 8; n >= 1; off >>= 1, n >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const float oS = up ? S[j] : S[j + n], oC = up ? C[j] : C[j + n];
      S[j] = up ? S[j + n] : S[j];
      C[j] = up ? C[j + n] : C[j];
      comp_add(S[j], C[j], __shfl_xor_sync(0xffffffffu, oS, off), __shfl_xor_sync(0xffffffffu, oC, off));
    }
  }
  comp_add(S[0], C[0], __shfl_xor_sync(0xffffffffu, S[0], 1), __shfl_xor_sync(0xffffffffu, C[0], 1));
}

constexpr int kDB = 8;   // l per block of the analysis

// kDB recurrence steps of one ring pair from l0, accumulating mu * (E or O)
// into the 2 kDB compensated sums; INJECT places the table start values.
template <bool INJECT, bool FINE>
__device__ __forceinline__ void analysis_block(int l0, const float2 *sA, dfl x, dfl &p1, dfl &p2, int ls, float4 v,
                                               float4 e, float4 o, float (&S)[16], float (&C)[16]) {
#pragma unroll
  for (int j = 0; j < kDB; ++j) {
    const int l = l0 + j;
    const float2 a2 = sA[j];
    dfl mu = df_step<FINE>(dfl{a2.x, a2.y}, x, p1, p2);
    if (INJECT) {
      if (l == ls) mu = dfl{v.x, v.y};
      if (l == ls + 1) mu = dfl{v.z, v.w};
    }
    p2 = p1;
    p1 = mu;
    const float4 f = (j & 1) ? o : e;
    dot2_acc<FINE>(S[2 * j], C[2 * j], mu, dfl{f.x, f.y});
    dot2_acc<FINE>(S[2 * j + 1], C[2 * j + 1], mu, dfl{f.z, f.w});
  }
}

// Start values for the double-float recurrence: first l with |lambda| >= 2^-60,
// and mu at that l and the next (mu = lambda / g), one thread per (m, k).
__global__ void __launch_bounds__(256) start_values_df_kernel(const double *xk, const double2 *rec, const double *g,
                                                              int lmax, int RP, int *ls_out, float4 *sv_out) {
  extern __shared__ double croot[];   // [m + 1] sqrt((2i + 1) / 2i)
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nid = (long long)(lmax + 1) * RP;
  lambda_mm_factors(croot, (int)(min(id - threadIdx.x + blockDim.x, nid) - 1) / RP);
  if (id >= nid) return;
  const int m = (int)(id / RP), k = (int)(id % RP);
  const double x = xk[k];
  const double st = sqrt((1.0 - x) * (1.0 + x));
  int ls = kNoStartD;
  double v0 = 0.0, v1 = 0.0;
  if (m == 0 || st > 0.0) {
    int e = 0;
    const double v = lambda_mm_scaled(croot, m, st, e);
    ls = walk_to_cut(rec + alm_idx_d(lmax, m, m), x, v, e, m, lmax, -60, kNoStartD, v0, v1);
  }
  float4 out = make_float4(0.f, 0.f, 0.f, 0.f);
  if (ls != kNoStartD) {
    const size_t base = alm_idx_d(lmax, m, m);
    const dfl a = df_from(v0 / g[base + (ls - m)]);
    const dfl b = (ls + 1 <= lmax) ? df_from(v1 / g[base + (ls + 1 - m)]) : dfl{0.f, 0.f};
    out = make_float4(a.h, a.l, b.h, b.l);
  }
  ls_out[id] = ls;
  sv_out[id] = out;
}

// g_l and A_l of the rescaled recurrence, one CTA per m (serial in l).
__global__ void rescale_coeffs_kernel(const double2 *rec, int lmax, double *g, float2 *A) {
  const int m = blockIdx.x;
  if (threadIdx.x != 0) return;
  const size_t base = alm_idx_d(lmax, m, m);
  double g2 = 1.0, g1 = 1.0;  // g_{l-2}, g_{l-1}
  for (int l = m; l <= lmax; ++l) {
    const double2 ab = rec[base + (l - m)];
    double gl, Al;
    if (l <= m + 1) {
      gl = 1.0;
      Al = ab.x;  // a_{m+1} (a_m = 0)
    } else {
      gl = ab.y * g2;
      Al = ab.x * g1 / gl;
    }
    g[base + (l - m)] = gl;
    const dfl d = df_from(Al);
    A[base + (l - m)] = make_float2(d.h, d.l);
    g2 = g1;
    g1 = gl;
  }
}

// The table: one thread per (m, k) runs the FP64 recurrence from the start
// values of the FP64 kernel and stores lambda as (hi, lo) from the first l of
// the 2^-60 cut on, zeros below it.
__global__ void lam_table_kernel(const double *xk, const double2 *rec, const int *ls64, const double2 *sv64,
                                 const int *ls_df, const long long *poff, int lmax, int RP, float4 *tab) {
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= (long long)(lmax + 1) * RP) return;
  const int m = (int)(id / RP), k = (int)(id % RP);
  const int npr = tab_rows(lmax, m);
  float4 *col = tab + ((size_t)poff[m] * ((RP + 31) >> 5) + (size_t)(k >> 5) * npr) * 32 + (k & 31);
  const int l64 = ls64[id], ldf = ls_df[id];
  const double x = xk[k];
  const size_t base = alm_idx_d(lmax, m, m);
  double p2 = 0.0, p1 = 0.0;  // lambda_{l-2}, lambda_{l-1}
  dfl row[4];                 // the pair of rows at hand: even and odd parts of the first, of the second
  for (int l = m; l < m + 2 * npr; ++l) {
    double lam = 0.0;
    if (l <= lmax && l >= l64) {
      if (l == l64) lam = sv64[id].x;
      else if (l == l64 + 1) lam = sv64[id].y;
      else {
        const double2 ab = rec[base + (l - m)];
        lam = ab.x * x * p1 - ab.y * p2;
      }
      p2 = p1;
      p1 = lam;
    }
    const dfl d = (l >= ldf && l <= lmax) ? df_from(lam) : dfl{0.f, 0.f};
    row[(l - m) & 3] = d;
    if (((l - m) & 3) == 3) {
      float4 *at = col + (size_t)(((l - m) >> 2) * 2) * 32;
      at[0] = df_pair(row[0], row[2]);
      at[32] = df_pair(row[1], row[3]);
    } else if ((l - m) == 2 * npr - 1) {   // the last row of an odd count, by itself
      col[(size_t)(npr - 1) * 32] = df_pair(row[0], row[1]);
    }
  }
}

// NT threads a CTA. At Nside 2048 / lmax 4096 the sums, coefficients and ring-pair
// state of one m take most of an SM's shared memory, so that one CTA fits however
// small it is: 256 threads there left 8 warps an SM to hide the recurrences'
// chains. With 512 threads, 1024 for the synthesis alone, an iteration's launch
// went from 102 to 94 ms and a synthesis from 36 to 31; blocks of 8 l with one
// barrier each (16 l, two barriers and sums in double before) and one form of the
// recurrence block a warp took the iteration to 78 ms. FP32 issue bounds both
// (37 instructions a term: 25 ms a pass).
template <int MODE, int NT, bool FINE>
__global__ void __launch_bounds__(NT, NT == 256 ? 2 : 1) legendre_df_kernel(const LegArgs A, const LegDfArgs D) {
  extern __shared__ double2 dsm[];
  __shared__ float2 red[2][NT / 32][16];
  __shared__ double mred[NT / 32][3];
  const int m = blockIdx.x;
  const int lmax = A.lmax, RP = A.RP;
  int L = A.lsht;
  double lam = 1.0;
  if (MODE != LEG_ITER && A.gate && A.gate->done) return;
  if (MODE == LEG_ITER) {
    if (A.ctl->done) return;
    L = A.ctl->lsht;
    lam = A.ctl->lambda;
  }
  const size_t base = alm_idx_d(lmax, m, m);
  if (m > L) {
    if (MODE == LEG_ITER || MODE == LEG_ANALYSIS) {
      double c2 = 0.0, inc = 0.0;
      for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
        const double2 so = A.alm[base + (l - m)];
        const double wgt = (m == 0) ? 1.0 : 2.0;
        const double a2 = so.x * so.x + so.y * so.y;
        if (MODE == LEG_ITER) {
          if (A.cl[l] > 0.0) c2 += wgt * a2 / A.cl[l];
          inc += wgt * a2;
        }
        A.alm[base + (l - m)] = make_double2(0.0, 0.0);
      }
      if (MODE == LEG_ITER) {
        for (int o = 16; o > 0; o >>= 1) {
          c2 += __shfl_xor_sync(0xffffffffu, c2, o);
          inc += __shfl_xor_sync(0xffffffffu, inc, o);
        }
        if ((threadIdx.x & 31) == 0) { mred[threadIdx.x >> 5][0] = c2; mred[threadIdx.x >> 5][1] = inc; }
        __syncthreads();
        if (threadIdx.x == 0) {
          double a = 0.0, b = 0.0;
          for (int w = 0; w < NT / 32; ++w) { a += mred[w][0]; b += mred[w][1]; }
          A.m_part[3 * m] = a;
          A.m_part[3 * m + 1] = b;
          A.m_part[3 * m + 2] = 0.0;
        }
      }
    }
    if (MODE == LEG_ITER || MODE == LEG_SYNTH) {
      for (int k = threadIdx.x; k < RP; k += blockDim.x)
        A.FS[(size_t)m * RP + k] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    }
    return;
  }
  const int Lm = L - m + 1;
  const int Lp = Lm + kLB;
  // shared: tl [Lp] double2 | sA [Lp] float2 | ss [Lp] float4 (synthesis coefficients g_l s_lm)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double2 *tl = dsm;
  float2 *sA = reinterpret_cast<float2 *>(dsm + Lp);
  float4 *ss = reinterpret_cast<float4 *>(sA + Lp + (Lp & 1));
  for (int i = threadIdx.x; i < Lp; i += blockDim.x) {
    sA[i] = (i < Lm) ? D.A[base + i] : make_float2(0.f, 0.f);
    tl[i] = make_double2(0.0, 0.0);
  }
  __syncthreads();

  if (MODE == LEG_ANALYSIS || MODE == LEG_ITER) {
    // per ring pair state in shared memory: the thread's sums then cover all of
    // its ring pairs of a chunk before one reduction per block of kDB values of
    // l; chunks of kAnaChunk ring pairs run one after another, each adding its
    // share to t_l
    for (int k0 = 0; k0 < RP; k0 += kAnaChunk<NT>) {
      const int nk = min(kAnaChunk<NT>, RP - k0);
      const int np = (nk + 31) & ~31;              // whole warps: a lane past the last ring pair has a state of its own
      float4 *stE = ss;                            // (Er, Ei) as hi/lo
      float4 *stO = stE + np;                      // (Or, Oi)
      float4 *stP = stO + np;                      // (p1, p2)
      float2 *stX = reinterpret_cast<float2 *>(stP + np);  // x as double-float
      for (int kk = threadIdx.x; kk < np; kk += blockDim.x) {
        double4_32a t = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        dfl xk{0.f, 0.f};
        if (kk < nk) {
          t = A.FT[(size_t)m * RP + k0 + kk];
          xk = df_from(A.x[k0 + kk]);
        }
        f_parities<FINE>(t, stE[kk], stO[kk]);
        stP[kk] = make_float4(0.f, 0.f, 0.f, 0.f);
        stX[kk] = make_float2(xk.h, xk.l);
      }
      __syncthreads();
      int lsr[4];                                  // first l of the thread's ring pairs
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int kk = threadIdx.x + i * NT;
        lsr[i] = kk < nk ? D.ls[(size_t)m * RP + k0 + kk] : kNoStartD;
      }
      int buf = 0;
      for (int l0 = m; l0 <= L; l0 += kDB, buf ^= 1) {
        float S[16], C[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) { S[j] = 0.f; C[j] = 0.f; }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          // the whole warp runs the same block: lanes without a term yet carry zeros, and one with a start value in
          // it takes the others through the injecting form (as per-lane branches the two forms ran one after the other)
          const int ls = lsr[i], kk = threadIdx.x + i * NT;
          const bool begun = ls < l0 + kDB;
          if (!__any_sync(0xffffffffu, begun)) continue;
          const bool starts = begun && ls + 1 >= l0;
          const float2 x2 = stX[kk];
          const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 e4 = begun ? stE[kk] : z, o4 = begun ? stO[kk] : z, q4 = stP[kk];
          dfl p1 = dfl{q4.x, q4.y}, p2 = dfl{q4.z, q4.w};
          if (__any_sync(0xffffffffu, starts))
            analysis_block<true, FINE>(l0, sA + (l0 - m), dfl{x2.x, x2.y}, p1, p2, ls,
                                 starts ? D.sv[(size_t)m * RP + k0 + kk] : z, e4, o4, S, C);
          else
            analysis_block<false, FINE>(l0, sA + (l0 - m), dfl{x2.x, x2.y}, p1, p2, ls, z, e4, o4, S, C);
          if (begun) stP[kk] = make_float4(p1.h, p1.l, p2.h, p2.l);
        }
        warp_sums16(S, C);
        if (!(lane & 1)) red[buf][warp][lane >> 1] = make_float2(S[0], C[0]);
        __syncthreads();                           // one a block: the other buffer is the next one's
        if (threadIdx.x < 16) {
          float tS = 0.f, tC = 0.f;
          for (int w = 0; w < NT / 32; ++w) {
            const float2 v = red[buf][w][threadIdx.x];
            const float n = tS + v.x, bb = n - tS;
            tC += v.y + ((tS - (n - bb)) + (v.x - bb));
            tS = n;
          }
          double *dst = reinterpret_cast<double *>(&tl[l0 - m + (threadIdx.x >> 1)]);
          dst[threadIdx.x & 1] += (double)tS + (double)tC;
        }
      }
      __syncthreads();
    }
    // undo the rescaling: lambda = g mu
    for (int l = m + threadIdx.x; l <= L; l += blockDim.x) {
      const double gl = A.fomega * D.g[base + (l - m)];
      tl[l - m].x *= gl;
      tl[l - m].y *= gl;
    }
    __syncthreads();
  }

  if (MODE == LEG_ANALYSIS) {
    for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x)
      A.alm[base + (l - m)] = (l <= L) ? tl[l - m] : make_double2(0.0, 0.0);
    return;
  }

  if (MODE == LEG_ITER) {
    double c2 = 0.0, inc = 0.0, nrm = 0.0;
    const double wgt = (m == 0) ? 1.0 : 2.0;
    const double lto = lam * A.tau * A.omega;
    for (int l = m + threadIdx.x; l <= lmax; l += blockDim.x) {
      const double2 so = A.alm[base + (l - m)];
      const double c = A.cl[l];
      double2 sn = make_double2(0.0, 0.0);
      if (l <= L && c > 0.0) {
        const double f = c / (c + lto);
        const double2 t = tl[l - m];
        sn = make_double2(f * (so.x + t.x), f * (so.y + t.y));
      }
      if (c > 0.0) c2 += wgt * (so.x * so.x + so.y * so.y) / c;
      const double dx = sn.x - so.x, dy = sn.y - so.y;
      inc += wgt * (dx * dx + dy * dy);
      nrm += wgt * (sn.x * sn.x + sn.y * sn.y);
      A.alm[base + (l - m)] = sn;
      if (l <= L) {
        const double gl = D.g[base + (l - m)];
        const dfl re = df_from(gl * sn.x), im = df_from(gl * sn.y);
        ss[l - m] = make_float4(re.h, re.l, im.h, im.l);
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      c2 += __shfl_xor_sync(0xffffffffu, c2, o);
      inc += __shfl_xor_sync(0xffffffffu, inc, o);
      nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    }
    if (lane == 0) { mred[warp][0] = c2; mred[warp][1] = inc; mred[warp][2] = nrm; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0, b = 0.0, c = 0.0;
      for (int w = 0; w < NT / 32; ++w) { a += mred[w][0]; b += mred[w][1]; c += mred[w][2]; }
      A.m_part[3 * m] = a;
      A.m_part[3 * m + 1] = b;
      A.m_part[3 * m + 2] = c;
    }
  } else {  // LEG_SYNTH
    for (int l = m + threadIdx.x; l <= L; l += blockDim.x) {
      const double gl = D.g[base + (l - m)];
      const double2 s = A.alm_in[base + (l - m)];
      const dfl re = df_from(gl * s.x), im = df_from(gl * s.y);
      ss[l - m] = make_float4(re.h, re.l, im.h, im.l);
    }
    __syncthreads();
  }

  // ---- synthesis onto every ring pair (one ring pair per thread at a time)
  for (int k = threadIdx.x; k < RP; k += blockDim.x) {
    const size_t mk = (size_t)m * RP + k;
    const int ls = D.ls[mk];
    float ERs = 0.f, ERc = 0.f, EIs = 0.f, EIc = 0.f, ORs = 0.f, ORc = 0.f, OIs = 0.f, OIc = 0.f;
    if (ls <= L) {
      const dfl x = df_from(A.x[k]);
      const float4 s4 = D.sv[mk];
      dfl p2 = dfl{s4.x, s4.y};
      dfl p1 = dfl{s4.z, s4.w};
      int l = ls;
      {
        const float4 c = ss[l - m];
        if (((l - m) & 1) == 0) { dot2_acc<FINE>(ERs, ERc, p2, dfl{c.x, c.y}); dot2_acc<FINE>(EIs, EIc, p2, dfl{c.z, c.w}); }
        else { dot2_acc<FINE>(ORs, ORc, p2, dfl{c.x, c.y}); dot2_acc<FINE>(OIs, OIc, p2, dfl{c.z, c.w}); }
      }
      if (l + 1 <= L) {
        const float4 c = ss[l + 1 - m];
        if (((l + 1 - m) & 1) == 0) { dot2_acc<FINE>(ERs, ERc, p1, dfl{c.x, c.y}); dot2_acc<FINE>(EIs, EIc, p1, dfl{c.z, c.w}); }
        else { dot2_acc<FINE>(ORs, ORc, p1, dfl{c.x, c.y}); dot2_acc<FINE>(OIs, OIc, p1, dfl{c.z, c.w}); }
      }
      l += 2;
      if (((l - m) & 1) == 1 && l <= L) {
        const float2 a2 = sA[l - m];
        const dfl mu = df_step<FINE>(dfl{a2.x, a2.y}, x, p1, p2);
        p2 = p1; p1 = mu;
        const float4 c = ss[l - m];
        dot2_acc<FINE>(ORs, ORc, mu, dfl{c.x, c.y});
        dot2_acc<FINE>(OIs, OIc, mu, dfl{c.z, c.w});
        ++l;
      }
      for (; l + 1 <= L; l += 2) {
        const float2 a0 = sA[l - m], a1 = sA[l + 1 - m];
        const dfl me = df_step<FINE>(dfl{a0.x, a0.y}, x, p1, p2);
        const dfl mo = df_step<FINE>(dfl{a1.x, a1.y}, x, me, p1);
        p2 = me; p1 = mo;
        const float4 ce = ss[l - m], co = ss[l + 1 - m];
        dot2_acc<FINE>(ERs, ERc, me, dfl{ce.x, ce.y});
        dot2_acc<FINE>(EIs, EIc, me, dfl{ce.z, ce.w});
        dot2_acc<FINE>(ORs, ORc, mo, dfl{co.x, co.y});
        dot2_acc<FINE>(OIs, OIc, mo, dfl{co.z, co.w});
      }
      if (l <= L) {
        const float2 a0 = sA[l - m];
        const dfl me = df_step<FINE>(dfl{a0.x, a0.y}, x, p1, p2);
        const float4 ce = ss[l - m];
        dot2_acc<FINE>(ERs, ERc, me, dfl{ce.x, ce.y});
        dot2_acc<FINE>(EIs, EIc, me, dfl{ce.z, ce.w});
      }
    }
    A.FS[mk] = f_rings<FINE>(df_norm(ERs, ERc), df_norm(EIs, EIc), df_norm(ORs, ORc), df_norm(OIs, OIc));
  }
}

// tl [Lp] double2 | sA [Lp (+1)] float2 | max(Lp, 3.5 chunk) float4 (synthesis
// coefficients, or the per-ring-pair analysis state of one chunk)
static size_t leg_df_smem(int lmax, int RP, int chunk) {
  const size_t Lp = (size_t)lmax + 1 + kLB;
  const size_t np = ((RP < chunk ? (size_t)RP : (size_t)chunk) + 31) / 32 * 32;
  const size_t st = 3 * np + np / 2;
  const size_t q = Lp > st ? Lp : st;
  return Lp * sizeof(double2) + (Lp + 1) * sizeof(float2) + q * sizeof(float4) + 16;
}

template <int MODE, int NT, bool FINE = false>
static void launch_df(const LegArgs &a, const LegDfArgs &d, cudaStream_t s) {
  raise_smem_cap(reinterpret_cast<const void *>(legendre_df_kernel<MODE, NT, FINE>));
  // the synthesis alone holds no ring-pair state
  const size_t sm = leg_df_smem(a.lmax, a.RP, MODE == LEG_SYNTH ? 0 : kAnaChunk<NT>);
  legendre_df_kernel<MODE, NT, FINE><<<a.lmax + 1, NT, sm, s>>>(a, d);
}

void launch_legendre_df(const LegArgs &a, const LegDfArgs &d, cudaStream_t s, int mode) {
  if (d.tab) {
    LegBatchMaps bm{};
    bm.n = 1;
    bm.FT[0] = a.FT;
    bm.FS[0] = a.FS;
    bm.alm[0] = mode == LEG_SYNTH ? const_cast<double2 *>(a.alm_in) : a.alm;   // read only by the synthesis
    bm.ctl[0] = mode == LEG_ITER ? a.ctl : a.gate;
    bm.m_part[0] = a.m_part;
    bm.part[0] = a.part;
    bm.coef[0] = a.coef;
    bm.cl[0] = a.cl;
    bm.tau[0] = a.tau;
    launch_legendre_tab(a, d, bm, 1, s, mode);
    return;
  }
  // four ring pairs a thread keep the larger CTAs' sums over lanes as cheap a term as the smaller ones'
  const bool wide = a.RP >= 2048;
  const bool fine = fine_steps(a.RP);
  switch (mode) {
    case LEG_SYNTH:
      if (wide) launch_df<LEG_SYNTH, 1024>(a, d, s);
      else if (fine) launch_df<LEG_SYNTH, 256, true>(a, d, s);
      else launch_df<LEG_SYNTH, 256>(a, d, s);
      break;
    case LEG_ANALYSIS:
      if (wide) launch_df<LEG_ANALYSIS, 512>(a, d, s);
      else if (fine) launch_df<LEG_ANALYSIS, 256, true>(a, d, s);
      else launch_df<LEG_ANALYSIS, 256>(a, d, s);
      break;
    default:
      if (wide) launch_df<LEG_ITER, 512>(a, d, s);
      else if (fine) launch_df<LEG_ITER, 256, true>(a, d, s);
      else launch_df<LEG_ITER, 256>(a, d, s);
      break;
  }
}

size_t lam_table_rows(int lmax) {
  size_t rows = 0;
  for (int m = 0; m <= lmax; ++m) rows += (size_t)tab_rows(lmax, m);
  return rows;
}

void launch_lam_table(const double *x, const double2 *rec, const int *ls64, const double2 *sv64, const int *ls_df,
                      const long long *poff, int lmax, int RP, float4 *tab, cudaStream_t s) {
  const long long n = (long long)(lmax + 1) * RP;
  lam_table_kernel<<<(int)((n + 127) / 128), 128, 0, s>>>(x, rec, ls64, sv64, ls_df, poff, lmax, RP, tab);
}

void launch_df_tables(const double *x, const double2 *rec, int lmax, int RP, double *g, float2 *A, int *ls,
                      float4 *sv, cudaStream_t s) {
  rescale_coeffs_kernel<<<lmax + 1, 32, 0, s>>>(rec, lmax, g, A);
  const long long n = (long long)(lmax + 1) * RP;
  const int nt = start_value_threads(n);
  start_values_df_kernel<<<(int)((n + nt - 1) / nt), nt, (size_t)(lmax + 1) * sizeof(double), s>>>(x, rec, g, lmax, RP, ls, sv);
}

}  // namespace wfk
