// Double-float arithmetic helpers shared by the FP64-accurate kernels: a value
// is the unevaluated sum hi + lo of two floats (48 significant bits), and
// every operation is built from error-free transformations (two_sum,
// two_prod via fma).
#pragma once

#include <cuda_runtime.h>

namespace wfk {

struct dfl { float h, l; };

__device__ __forceinline__ dfl df_from(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ double df_to(dfl a) { return (double)a.h + (double)a.l; }

// A double-float in the 8 bytes of a double: the Fourier records F of the
// double-float stages hold (hi, lo) pairs where those of the native stages hold
// doubles, so that no stage pays the FP64 pipe (1/63 of FP32) for conversions.
__device__ __forceinline__ double df_pack(dfl a) { return __hiloint2double(__float_as_int(a.h), __float_as_int(a.l)); }
__device__ __forceinline__ dfl df_unpack(double v) {
  return {__int_as_float(__double2hiint(v)), __int_as_float(__double2loint(v))};
}

__device__ __forceinline__ dfl df_neg(dfl a) { return {-a.h, -a.l}; }
__device__ __forceinline__ float4 df_pair(dfl a, dfl b) { return make_float4(a.h, a.l, b.h, b.l); }

// (S, C) += (rS, rC), another thread's compensated sum: error-free in S
__device__ __forceinline__ void comp_add(float &S, float &C, float rS, float rC) {
  const float s = S + rS;
  const float bb = s - S;
  C = C + rC + ((S - (s - bb)) + (rS - bb));
  S = s;
}

// S + C of a compensated sum as a double-float
__device__ __forceinline__ dfl df_norm(float S, float C) {
  const float s = S + C, bb = s - S;
  return {s, (S - (s - bb)) + (C - bb)};
}

// a + b (two_sum of the high parts, low parts added, renormalised)
__device__ __forceinline__ dfl df_add(dfl a, dfl b) {
  const float s = a.h + b.h;
  const float bb = s - a.h;
  float e = (a.h - (s - bb)) + (b.h - bb);
  e += a.l + b.l;
  const float r = s + e;
  return {r, e - (r - s)};
}

// a + b with the low parts' sum error-free too (accurate double-word addition, Joldes, Muller and Popescu, ACM TOMS 44,
// 2017): where a few sums stand between long chains of products, as the Fourier records' do. FINE: that of the errors
// too, one rounding in all (24 instructions instead of 20)
template <bool FINE>
__device__ __forceinline__ dfl df_add2(dfl a, dfl b) {
  const float s = a.h + b.h, bb = s - a.h;
  const float e = (a.h - (s - bb)) + (b.h - bb);
  const float t = a.l + b.l, bt = t - a.l;
  const float f = (a.l - (t - bt)) + (b.l - bt);
  const float c = e + t;
  const float v = s + c;
  float w = f;
  if (FINE) {
    const float bc = c - e;
    w += (e - (c - bc)) + (t - bc);
  }
  w += c - (v - s);
  const float r = v + w;
  return {r, w - (r - v)};
}

// a * b (two_prod of the high parts plus the cross terms, renormalised)
__device__ __forceinline__ dfl df_mul(dfl a, dfl b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
  const float r = p + e;
  return {r, e - (r - p)};
}

// S + C += a * b: compensated dot-product step (Ogita, Rump and Oishi,
// "Accurate sum and dot product", SIAM J. Sci. Comput. 26, 2005). The loops over
// l and over ring pairs are made of this step, and FP32 issue bounds them once
// their table reads are hidden: in 13 instructions 2.8e12 products/s measured.
// FINE, 13 instructions: every error term exact but for the two cross terms,
// as in the sum of Ogita et al., and the product of the low parts. Else 10: two_sum(S, p) splits into the parts of S
// and of p that the rounded sum lost, the part of p is formed from the exact
// product (one fma instead of two_prod's error term and a subtraction) and the
// cross terms are added to it. Those three round at the sum's own ulp, which
// short sums feel (7 % more error over 16 terms, 1 % over 128: fine_steps);
// long ones are bound by the rounding of C, which dot2_tidy keeps small.
template <bool FINE = false>
__device__ __forceinline__ void dot2_acc(float &S, float &C, dfl a, dfl b) {
  const float p = __fmul_rn(a.h, b.h);
  const float s = __fadd_rn(S, p);
  const float bb = s - S;
  const float d = S - (s - bb);
  if (FINE) {
    float v = fmaf(a.h, b.h, -p);
    v = fmaf(a.l, b.l, v);
    v = fmaf(a.l, b.h, v);
    v = fmaf(a.h, b.l, v);
    C += (d + (p - bb)) + v;
  } else {
    float v = fmaf(a.h, b.h, -bb);
    v = fmaf(a.l, b.h, v);
    v = fmaf(a.h, b.l, v);
    C += d + v;
  }
  S = s;
}

// The collected errors of a long compensated sum moved into its leading part: the next ones round at a small C's ulp
// again (every 32 terms or so the error of a sum of 512 falls by two). two_sum, exact also where the terms cancelled
// and |C| > |S|: folding a sum that has ended once more, as a launch for a longer one beside it does, changes nothing.
__device__ __forceinline__ void dot2_tidy(float &S, float &C) {
  const float s = S + C, bb = s - S;
  C = (S - (s - bb)) + (C - bb);
  S = s;
}

// mu_l = (A x) mu1 - mu2 in double-float: one step of the rescaled Legendre
// recurrence mu_l = A_l x mu_{l-1} - mu_{l-2}. 17 FP32 instructions, the sum's
// error from the exact product as in dot2_acc; FINE, 19: the product's error by
// itself, which rounds at the product's ulp and not at the sum's
template <bool FINE = false>
__device__ __forceinline__ dfl df_step(dfl A, dfl x, dfl mu1, dfl mu2) {
  const float ch = __fmul_rn(A.h, x.h);
  float ce = fmaf(A.h, x.h, -ch);
  ce = fmaf(A.h, x.l, fmaf(A.l, x.h, ce));
  const float qh = __fmul_rn(ch, mu1.h);
  const float sh = __fadd_rn(qh, -mu2.h);
  float e;
  if (FINE) {
    float qe = fmaf(ch, mu1.h, -qh);
    qe = fmaf(ch, mu1.l, fmaf(ce, mu1.h, qe));
    const float bb = sh - qh;
    e = (qh - (sh - bb)) + (-mu2.h - bb);
    e += qe - mu2.l;
  } else {
    const float bb = sh + mu2.h;          // the part of the product in sh
    const float d = -mu2.h - (sh - bb);
    float v = fmaf(ch, mu1.h, -bb);
    v = fmaf(ch, mu1.l, fmaf(ce, mu1.h, v));
    e = d + (v - mu2.l);
  }
  const float rh = sh + e;
  return {rh, e - (rh - sh)};
}

// A Fourier record (north re, im, south re, im; df_pack'ed) as the sums of its two rings for even l - m, E = N + S,
// and for odd, O = N - S, each (re hi, re lo, im hi, im lo); and the record of E and O.
template <bool FINE>
__device__ __forceinline__ void f_parities(const double4_32a &t, float4 &E, float4 &O) {
  const dfl nr = df_unpack(t.x), ni = df_unpack(t.y), sr = df_unpack(t.z), si = df_unpack(t.w);
  E = df_pair(df_add2<FINE>(nr, sr), df_add2<FINE>(ni, si));
  O = df_pair(df_add2<FINE>(nr, df_neg(sr)), df_add2<FINE>(ni, df_neg(si)));
}
template <bool FINE>
__device__ __forceinline__ double4_32a f_rings(dfl er, dfl ei, dfl orr, dfl oi) {
  return make_double4_32a(df_pack(df_add2<FINE>(er, orr)), df_pack(df_add2<FINE>(ei, oi)), df_pack(df_add2<FINE>(er, df_neg(orr))),
                          df_pack(df_add2<FINE>(ei, df_neg(oi))));
}

}  // namespace wfk
