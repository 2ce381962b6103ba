// Folding of a ring's azimuthal Fourier coefficients onto the residues of its
// DFT (m-aliasing): for a ring of n pixels,
//   G_q = sum_{j >= 0} s^j F_{q + n j} + sum_{j >= 1} s^j conj(F_{n j - q}),
// m <= L, with s = -1 on rings whose first pixel sits half a pixel off
// (the phase e^{i m phi0} changes sign with each alias) and s = 1 otherwise.
// On rings shorter than the thread block, each residue's alias series is split
// over several threads and their partial sums are added in a fixed order.
#pragma once

#include <cuda_runtime.h>

#include "df.cuh"
#include "wf_internal.h"

namespace wfk {

// The share j = j0, j0 + dj, ... of residue q's series, from F stored as
// double4_32a (north re, north im, south re, south im) at [m RP + k].
__device__ __forceinline__ double2 fold_alias_sum(const double4_32a *FS, int RP, int k, int slot, int shifted,
                                                  int n, int q, int L, int j0, int dj) {
  double ar = 0.0, ai = 0.0;
  for (int j = j0, m = q + n * j0; m <= L; j += dj, m += n * dj) {
    const double4_32a f4 = FS[(size_t)m * RP + k];
    double fr = slot ? f4.z : f4.x, fi = slot ? f4.w : f4.y;
    if (shifted && (j & 1)) { fr = -fr; fi = -fi; }
    ar += fr; ai += fi;
  }
  for (int j = 1 + j0, m = n * (1 + j0) - q; m <= L; j += dj, m += n * dj) {
    const double4_32a f4 = FS[(size_t)m * RP + k];
    double fr = slot ? f4.z : f4.x, fi = slot ? -f4.w : -f4.y;
    if (shifted && (j & 1)) { fr = -fr; fi = -fi; }
    ar += fr; ai += fi;
  }
  return make_double2(ar, ai);
}

// Both slots' shares at once in double-float (records of df_pack'ed values),
// north and south each as (re hi, re lo, im hi, im lo), each record read once.
struct FoldPair { float4 n, s; };
__device__ __forceinline__ FoldPair fold_record(const double4_32a *FS, size_t at, float sg, float cj) {
  const double4_32a f = FS[at];
  const dfl nr = df_unpack(f.x), ni = df_unpack(f.y), sr = df_unpack(f.z), si = df_unpack(f.w);
  const float ci = sg * cj;
  return {make_float4(sg * nr.h, sg * nr.l, ci * ni.h, ci * ni.l),
          make_float4(sg * sr.h, sg * sr.l, ci * si.h, ci * si.l)};
}
template <bool FINE>
__device__ __forceinline__ float4 fold_add(float4 a, float4 b) {
  return df_pair(df_add2<FINE>(dfl{a.x, a.y}, dfl{b.x, b.y}), df_add2<FINE>(dfl{a.z, a.w}, dfl{b.z, b.w}));
}
template <bool FINE>
__device__ __forceinline__ FoldPair fold_alias_sum2(const double4_32a *FS, int RP, int k, int shifted, int n, int q,
                                                    int L, int j0, int dj) {
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  FoldPair a{z, z};
  bool first = true;
  auto take = [&](FoldPair r) {
    if (first) a = r;
    else { a.n = fold_add<FINE>(a.n, r.n); a.s = fold_add<FINE>(a.s, r.s); }
    first = false;
  };
  for (int j = j0, m = q + n * j0; m <= L; j += dj, m += n * dj)
    take(fold_record(FS, (size_t)m * RP + k, (shifted && (j & 1)) ? -1.f : 1.f, 1.f));
  for (int j = 1 + j0, m = n * (1 + j0) - q; m <= L; j += dj, m += n * dj)
    take(fold_record(FS, (size_t)m * RP + k, (shifted && (j & 1)) ? -1.f : 1.f, -1.f));
  return a;
}

// fold_ring for both rings of a pair: store(q, G_q north, G_q south), in
// double-float. part: shared scratch of blockDim.x FoldPair. A residue's series
// of at most L / n + 1 aliases is split over as many threads as it has terms
// and the block has room for (over blockDim.x / n threads whatever the series'
// length, the sum over them walked up to 64 empty parts on the smallest rings).
template <bool FINE, class Store>
__device__ __forceinline__ void fold_ring2(const double4_32a *FS, int RP, int k, int shifted, int n, int L,
                                           FoldPair *part, Store store) {
  const int nt = blockDim.x;
  const int nj = min(nt / n, L / n + 1);
  if (nj <= 1) {
    for (int q = threadIdx.x; q < n; q += nt) {
      const FoldPair g = fold_alias_sum2<FINE>(FS, RP, k, shifted, n, q, L, 0, 1);
      store(q, g.n, g.s);
    }
    return;
  }
  const int t = threadIdx.x;
  if (t < n * nj) part[t] = fold_alias_sum2<FINE>(FS, RP, k, shifted, n, t % n, L, t / n, nj);
  __syncthreads();
  if (t < n) {
    FoldPair g = part[t];
    for (int jg = 1; jg < nj; ++jg) {
      const FoldPair p = part[jg * n + t];
      g.n = fold_add<FINE>(g.n, p.n);
      g.s = fold_add<FINE>(g.s, p.s);
    }
    store(t, g.n, g.s);
  }
}

// G_q for every residue, passed to store(q, G_q) by one thread each.
// part: shared scratch of blockDim.x double2. Contains a __syncthreads when
// the ring is shorter than the block (uniform over the CTA).
template <class Store>
__device__ __forceinline__ void fold_ring(const double4_32a *FS, int RP, int k, int slot, int shifted, int n, int L,
                                          double2 *part, Store store) {
  const int nt = blockDim.x;
  if (n >= nt) {
    for (int q = threadIdx.x; q < n; q += nt) store(q, fold_alias_sum(FS, RP, k, slot, shifted, n, q, L, 0, 1));
    return;
  }
  const int nj = nt / n, t = threadIdx.x;
  if (t < n * nj) part[t] = fold_alias_sum(FS, RP, k, slot, shifted, n, t % n, L, t / n, nj);
  __syncthreads();
  if (t < n) {
    double2 g = make_double2(0.0, 0.0);
    for (int jg = 0; jg < nj; ++jg) {
      g.x += part[jg * n + t].x;
      g.y += part[jg * n + t].y;
    }
    store(t, g);
  }
}

}  // namespace wfk
