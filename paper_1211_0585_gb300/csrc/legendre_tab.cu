// Legendre stage over the precomputed lambda table (double-float,
// FP64-accurate), for one map or two that share the shape.
//
// Row r of m is the pair l = m + 2r, m + 2r + 1 (the even and odd parity parts).
// The table holds lambda_lm(x_k) as double-floats by pairs of rows, over the
// ring pairs in tiles of 32 of them: [m][tile][r][32] float4, at even r the even
// parts of rows r and r + 1 (lambda_{m+2r} hi, lo, lambda_{m+2r+2} hi, lo), at
// r + 1 their odd parts, so that an analysis lane of one parity takes two rows in
// one load; the last row of an odd count holds its even and its odd part.
// Entries below the 2^-60 cut (and the columns past RP of a partial tile) are
// zero. One iteration is two launches:
//   analysis   CTA (m, kTabRows rows): t_l of its rows over every ring pair,
//              then Eq. 4 of those l -- complete in the CTA --, the new state, its
//              double-float coefficients for the synthesis and the partial sums;
//   synthesis  CTA (m, up to 8 tiles): the coefficients' rows onto its ring pairs.
// The standalone transforms are the same kernels without Eq. 4. Every map's
// arithmetic and order are those of a launch for it alone, so a map's iterates
// do not depend on what shares its launches.
//
// Why two launches of many small CTAs: as one CTA per m doing both passes, a
// launch lasted as long as the CTA of m = 0 (its rows are twice the average and
// only its own 8 warps work on them): 249 us an iteration at Nside 256 / lmax
// 512, where the table's two passes are 119 us of HBM time; now 160 us, and 261
// instead of 302 us for two maps (Nside 512: 1029 against 1008 us for one map,
// where HBM bounds both forms, 1457 against 1835 for two).
#include <cuda_runtime.h>

#include <algorithm>

#include "df.cuh"
#include "pdl.cuh"
#include "wf_internal.h"

namespace wfk {

namespace {

constexpr int kTabChunk = 1024;   // ring pairs whose Fourier sums are staged in shared memory at once
constexpr int kAhead = 2;         // tiles (analysis) or row batches (synthesis) in flight in registers
constexpr int kSynRows = 4;       // synthesis: rows per load batch
constexpr int kWarpsT = kThreads / 32;
constexpr int kNoStartT = 1 << 30;

__device__ __forceinline__ size_t aidx_t(int lmax, int l, int m) { return (size_t)m * (2 * lmax + 1 - m) / 2 + l; }

// the maps of a launch: which run, and their band limits
template <int NB, bool ITER>
struct MapSet {
  bool on[NB];
  int Lb[NB];
  int L = -1;
  __device__ __forceinline__ MapSet(const LegArgs &A, const LegBatchMaps &Bm) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      on[b] = b < Bm.n && !(Bm.ctl[b] && Bm.ctl[b]->done);
      Lb[b] = on[b] ? (ITER ? Bm.ctl[b]->lsht : A.lsht) : -1;
      L = max(L, Lb[b]);
    }
  }
};

// Analysis. A warp takes groups of 4 rows, streamed over all tiles of 32 ring
// pairs; lane (rho, sigma, p) sums rows 2 rho and 2 rho + 1 of the group, parity
// p, over the columns sigma + 8 j: one 16-byte table value and one 16-byte
// Fourier sum from shared memory for four products (a lane per row with both
// parities took three, and its shared-memory wavefronts, 12 a column step, were
// more than the SM's FP32 issue slots). The sigma lanes combine by exchanging
// halves. Bound by HBM at Nside 512 (540 us a launch at lmax 1024, 0.87 of the
// copy rate; 595 us with one tile in flight, 643 us with groups of 8 rows, whose
// registers leave two CTAs per SM), by latency at the two CTAs an SM that two maps'
// registers leave (833 us for both) and by FP32 issue and HBM below Nside 512 (0.54 of the issue slots at Nside 256). 96 rows a CTA: 91 us at Nside 256 / lmax 512 and 816
// at Nside 512 for two maps, against 97 and 855 with 64 and 98 and 968 with 32.
template <int NB, bool ITER, bool FINE>
__global__ void __launch_bounds__(kThreads, NB == 1 ? 3 : 2) tab_analysis_kernel(const LegArgs A, const LegDfArgs D,
                                                                                 const LegBatchMaps Bm) {
  extern __shared__ float4 fsm[];   // [NB][parity][chunk] Fourier sums E = N + S, O = N - S
  __shared__ int tmin[kTabChunk / 32];
  __shared__ double2 tl[NB][2 * kTabRows];
  __shared__ double mred[kWarpsT][3];
  const int m = blockIdx.x, r0 = blockIdx.y * kTabRows;
  const int lmax = A.lmax, RP = A.RP;
  pdl_wait();
  pdl_next();
  if (m + 2 * r0 > lmax) return;
  const MapSet<NB, ITER> S(A, Bm);
  if (S.L < 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int npr = tab_rows(lmax, m);                                // table rows of m
  const int rows = min(kTabRows, npr - r0);
  const int rend = S.L >= m ? min(r0 + rows - 1, (S.L - m) >> 1) : -1;   // last row any map needs
  const size_t base = aidx_t(lmax, m, m);
  for (int i = threadIdx.x; i < 2 * kTabRows; i += kThreads)
#pragma unroll
    for (int b = 0; b < NB; ++b) tl[b][i] = make_double2(0.0, 0.0);

  const int p = lane & 1, sig = (lane >> 1) & 7, rho = lane >> 4;
  const int nkc = min(RP, kTabChunk);
  for (int k0 = 0; k0 < RP && rend >= r0; k0 += kTabChunk) {
    const int nk = min(kTabChunk, RP - k0), ntile = (nk + 31) >> 5;
    if (k0) __syncthreads();
    for (int t = warp; t < ntile; t += kWarpsT) {
      const int kk = 32 * t + lane;
      const int mn = __reduce_min_sync(0xffffffffu, kk < nk ? D.ls[(size_t)m * RP + k0 + kk] : kNoStartT);
      if (lane == 0) tmin[t] = mn;
    }
    __syncthreads();
    // tiles from the first with a term on (towards the equator the first l falls)
    auto first_tile = [&](int l) {
      int t = 0;
      while (t < ntile && tmin[t] > l) ++t;
      return t;
    };
    // a group of rows is taken from the tile of its own last l, whatever band limits share the launch: where its sums are
    // folded back (dot2_tidy) then depends on the map alone
    auto first_of_group = [&](int rg) { return first_tile(m + 2 * (r0 + 4 * rg) + 7); };
    for (int kk = 32 * first_of_group((rend - r0) >> 2) + threadIdx.x; kk < nk; kk += kThreads) {
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        float4 e = make_float4(0.f, 0.f, 0.f, 0.f), o = e;
        if (S.Lb[b] >= m) f_parities<FINE>(Bm.FT[b][(size_t)m * RP + k0 + kk], e, o);
        fsm[(size_t)(2 * b) * nkc + kk] = e;
        fsm[(size_t)(2 * b + 1) * nkc + kk] = o;
      }
    }
    __syncthreads();
    const float4 *tc = D.tab + ((size_t)D.poff[m] * ((RP + 31) >> 5) + (size_t)(k0 >> 5) * npr) * 32;
    for (int rg = warp; r0 + 4 * rg <= rend; rg += kWarpsT) {
      const int ra = r0 + 4 * rg + 2 * rho;            // this lane's rows: ra, ra + 1
      const bool use = ra <= rend, last = ra == npr - 1;   // last: a row by itself
      auto load = [&](int t, float4 (&v)[4]) {
        const float4 *src = tc + ((size_t)t * npr + ra + (last ? 0 : p)) * 32 + sig;
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = use ? __ldcs(src + 8 * j) : make_float4(0.f, 0.f, 0.f, 0.f);
      };
      float aS[NB][4], aC[NB][4];                      // row ra re, im, row ra + 1 re, im
#pragma unroll
      for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int q = 0; q < 4; ++q) { aS[b][q] = 0.f; aC[b][q] = 0.f; }
      float4 v[kAhead][4];                             // tiles in flight
      const int t0 = first_of_group(rg);
#pragma unroll
      for (int d = 0; d < kAhead; ++d)
        if (t0 + d < ntile) load(t0 + d, v[d]);
      for (int tb = t0; tb < ntile; tb += kAhead) {
#pragma unroll
        for (int d = 0; d < kAhead; ++d) {             // compile-time buffer indices
          const int t = tb + d;
          if (t >= ntile) break;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int kk = min(32 * t + sig + 8 * j, nk - 1);   // columns past RP: zero table values
            const dfl la{v[d][j].x, v[d][j].y}, lb{v[d][j].z, v[d][j].w};
#pragma unroll
            for (int b = 0; b < NB; ++b) {
              const float4 f = fsm[(size_t)(2 * b + p) * nkc + kk];
              dot2_acc<FINE>(aS[b][0], aC[b][0], la, dfl{f.x, f.y});
              dot2_acc<FINE>(aS[b][1], aC[b][1], la, dfl{f.z, f.w});
              dot2_acc<FINE>(aS[b][2], aC[b][2], lb, dfl{f.x, f.y});
              dot2_acc<FINE>(aS[b][3], aC[b][3], lb, dfl{f.z, f.w});
            }
          }
          if (t + kAhead < ntile) load(t + kAhead, v[d]);
        }
        if (((tb - t0) & 7) == 6) {                    // 32 terms a sum
#pragma unroll
          for (int b = 0; b < NB; ++b)
#pragma unroll
            for (int q = 0; q < 4; ++q) dot2_tidy(aS[b][q], aC[b][q]);
        }
      }
      // lane bits 1, 2 keep the row, re or im; bit 3 is summed over
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        float(&s)[4] = aS[b];
        float(&c)[4] = aC[b];
#pragma unroll
        for (int off = 2, n = 2; n >= 1; off <<= 1, n >>= 1) {
          const bool up = (lane & off) != 0;
#pragma unroll
          for (int q = 0; q < n; ++q) {
            const float oS = up ? s[q] : s[q + n], oC = up ? c[q] : c[q + n];
            s[q] = up ? s[q + n] : s[q];
            c[q] = up ? c[q + n] : c[q];
            comp_add(s[q], c[q], __shfl_xor_sync(0xffffffffu, oS, off), __shfl_xor_sync(0xffffffffu, oC, off));
          }
        }
        comp_add(s[0], c[0], __shfl_xor_sync(0xffffffffu, s[0], 8), __shfl_xor_sync(0xffffffffu, c[0], 8));
        // (a row by itself: its odd part went where an odd lane's second row goes)
        const int second = (lane >> 1) & 1, row = last ? ra : ra + second;
        if (!(lane & 8) && (last ? second == p && use : row <= rend))
          reinterpret_cast<double *>(&tl[b][2 * (row - r0) + p])[(lane >> 2) & 1] += (double)s[0] + (double)c[0];
      }
    }
  }
  __syncthreads();

  // the chunk's l: Eq. 4, or the t_l themselves
  const double wgt = (m == 0) ? 1.0 : 2.0, h = A.fomega;
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    if (!S.on[b]) continue;
    double2 *alm = Bm.alm[b] + base;
    double c2 = 0.0, inc = 0.0, nrm = 0.0;
    const double lto = ITER ? Bm.ctl[b]->lambda * Bm.tau[b] * A.omega : 0.0;
    for (int i = threadIdx.x; i < 2 * rows; i += kThreads) {
      const int l = m + 2 * r0 + i;
      if (l > lmax) break;
      const double2 t = tl[b][i];
      if (!ITER) {
        alm[l - m] = l <= S.Lb[b] ? make_double2(h * t.x, h * t.y) : make_double2(0.0, 0.0);
        continue;
      }
      const double2 so = alm[l - m];
      const double c = Bm.cl[b][l];
      double2 sn = make_double2(0.0, 0.0);
      if (l <= S.Lb[b] && c > 0.0) {
        const double f = c / (c + lto);
        sn = make_double2(f * fma(h, t.x, so.x), f * fma(h, t.y, so.y));
      }
      if (c > 0.0) c2 += wgt * (so.x * so.x + so.y * so.y) / c;
      const double dx = sn.x - so.x, dy = sn.y - so.y;
      inc += wgt * (dx * dx + dy * dy);
      nrm += wgt * (sn.x * sn.x + sn.y * sn.y);
      alm[l - m] = sn;
      Bm.coef[b][base + (l - m)] = df_pair(df_from(sn.x), df_from(sn.y));
    }
    if (!ITER) continue;
    constexpr int nw = (2 * kTabRows + 31) / 32;       // warps with an l
    if (warp < nw) {
      for (int o = 16; o > 0; o >>= 1) {
        c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        inc += __shfl_xor_sync(0xffffffffu, inc, o);
        nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
      }
      if (lane == 0) { mred[warp][0] = c2; mred[warp][1] = inc; mred[warp][2] = nrm; }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
      double a = 0.0;
      for (int x = 0; x < nw; ++x) a += mred[x][threadIdx.x];
      Bm.part[b][((size_t)m * gridDim.y + blockIdx.y) * 3 + threadIdx.x] = a;
    }
    __syncthreads();
  }
}

// Synthesis. A warp takes a tile of 32 ring pairs (lane = ring pair) and walks
// the rows from the first any of them needs, two batches of kSynRows in flight
// in registers. Bound by HBM at Nside 512 (489 us a launch at lmax 1024, 0.96 of
// the copy rate; 624 us for two maps), 69 us at Nside 256 / lmax 512.
template <int NB, bool ITER, bool FINE>
__global__ void __launch_bounds__(kThreads, 3) tab_synthesis_kernel(const LegArgs A, const LegDfArgs D,
                                                                                  const LegBatchMaps Bm, int nchunk) {
  extern __shared__ float4 csm[];   // [NB][nc] coefficients (re hi, re lo, im hi, im lo)
  const int m = blockIdx.x;
  const int lmax = A.lmax, RP = A.RP;
  pdl_wait();
  pdl_next();
  const MapSet<NB, ITER> S(A, Bm);
  if (S.L < 0) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t base = aidx_t(lmax, m, m);
  if (ITER && blockIdx.y == 0 && threadIdx.x < 3) {   // the partial sums of m, in the order of its chunks
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      if (!S.on[b]) continue;
      double a = 0.0;
      for (int x = 0; x < nchunk && m + 2 * x * kTabRows <= lmax; ++x)
        a += Bm.part[b][((size_t)m * nchunk + x) * 3 + threadIdx.x];
      Bm.m_part[b][3 * m + threadIdx.x] = a;
    }
  }
  const int k = 32 * (blockIdx.y * (blockDim.x >> 5) + warp) + lane;
  if (m > S.L) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (S.on[b] && k < RP) Bm.FS[b][(size_t)m * RP + k] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
    return;
  }
  const int npr = tab_rows(lmax, m), rneed = (S.L - m) >> 1;
  const bool single = rneed == npr - 1 && (npr & 1);       // a row by itself at the end
  const int rlast = single ? npr - 2 : rneed | 1;          // last of the rows in pairs
  const int nc = 2 * ((rneed | 1) + 1);
  for (int i = threadIdx.x; i < nc; i += blockDim.x) {
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
      if (m + i <= S.Lb[b]) {
        if (ITER) {
          c = Bm.coef[b][base + i];
        } else {
          const double2 v = Bm.alm[b][base + i];
          c = df_pair(df_from(v.x), df_from(v.y));
        }
      }
      csm[(size_t)b * nc + i] = c;
    }
  }
  __syncthreads();
  const int lw = __reduce_min_sync(0xffffffffu, k < RP ? D.ls[(size_t)m * RP + k] : kNoStartT);
  float acc[NB][8];
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int q = 0; q < 8; ++q) acc[b][q] = 0.f;
  if (lw <= S.L) {
    const float4 *src = D.tab + ((size_t)D.poff[m] * ((RP + 31) >> 5) + (size_t)(k >> 5) * npr) * 32 + lane;
    auto load = [&](int r, float4 (&v)[kSynRows]) {    // r even: rows r .. of pairs (even l - m, odd l - m)
#pragma unroll
      for (int i = 0; i < kSynRows; ++i)
        v[i] = (r + i <= rlast) ? __ldcs(src + (size_t)(r + i) * 32) : make_float4(0.f, 0.f, 0.f, 0.f);
    };
    float4 buf[kAhead + 1][kSynRows];
    const int rfirst = ((lw - m) >> 1) & ~1;
#pragma unroll
    for (int d = 0; d <= kAhead; ++d)
      if (d < kAhead) load(rfirst + d * kSynRows, buf[d]);
    for (int r0 = rfirst; r0 <= rlast; r0 += (kAhead + 1) * kSynRows) {
#pragma unroll
      for (int d = 0; d <= kAhead; ++d) {              // compile-time buffer indices
        const int r = r0 + d * kSynRows;
        if (r > rlast) break;
        load(r + kAhead * kSynRows, buf[(d + kAhead) % (kAhead + 1)]);
#pragma unroll
        for (int i = 0; i < kSynRows; i += 2) {
          if (r + i > rlast) break;
          const float4 e = buf[d][i], o = buf[d][i + 1];   // rows r + i and r + i + 1: even parts, odd parts
#pragma unroll
          for (int b = 0; b < NB; ++b) {
            const float4 *c = csm + (size_t)b * nc + 2 * (r + i);
            dot2_acc<FINE>(acc[b][0], acc[b][1], dfl{e.x, e.y}, dfl{c[0].x, c[0].y});
            dot2_acc<FINE>(acc[b][2], acc[b][3], dfl{e.x, e.y}, dfl{c[0].z, c[0].w});
            dot2_acc<FINE>(acc[b][4], acc[b][5], dfl{o.x, o.y}, dfl{c[1].x, c[1].y});
            dot2_acc<FINE>(acc[b][6], acc[b][7], dfl{o.x, o.y}, dfl{c[1].z, c[1].w});
            dot2_acc<FINE>(acc[b][0], acc[b][1], dfl{e.z, e.w}, dfl{c[2].x, c[2].y});
            dot2_acc<FINE>(acc[b][2], acc[b][3], dfl{e.z, e.w}, dfl{c[2].z, c[2].w});
            dot2_acc<FINE>(acc[b][4], acc[b][5], dfl{o.z, o.w}, dfl{c[3].x, c[3].y});
            dot2_acc<FINE>(acc[b][6], acc[b][7], dfl{o.z, o.w}, dfl{c[3].z, c[3].w});
          }
        }
      }
      if ((r0 - rfirst) % (2 * (kAhead + 1) * kSynRows)) {   // every 24 rows
#pragma unroll
        for (int b = 0; b < NB; ++b)
#pragma unroll
          for (int q = 0; q < 8; q += 2) dot2_tidy(acc[b][q], acc[b][q + 1]);
      }
    }
  }
  if (single && lw <= S.L) {
    const float4 x = D.tab[((size_t)D.poff[m] * ((RP + 31) >> 5) + (size_t)(k >> 5) * npr + npr - 1) * 32 + lane];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const float4 *c = csm + (size_t)b * nc + 2 * (npr - 1);
      dot2_acc<FINE>(acc[b][0], acc[b][1], dfl{x.x, x.y}, dfl{c[0].x, c[0].y});
      dot2_acc<FINE>(acc[b][2], acc[b][3], dfl{x.x, x.y}, dfl{c[0].z, c[0].w});
      dot2_acc<FINE>(acc[b][4], acc[b][5], dfl{x.z, x.w}, dfl{c[1].x, c[1].y});
      dot2_acc<FINE>(acc[b][6], acc[b][7], dfl{x.z, x.w}, dfl{c[1].z, c[1].w});
    }
  }
  if (k < RP) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
      if (S.on[b])
        Bm.FS[b][(size_t)m * RP + k] = f_rings<FINE>(df_norm(acc[b][0], acc[b][1]), df_norm(acc[b][2], acc[b][3]),
                                               df_norm(acc[b][4], acc[b][5]), df_norm(acc[b][6], acc[b][7]));
  }
}

size_t ana_smem(int nb, int RP) { return (size_t)nb * 2 * std::min(RP, kTabChunk) * sizeof(float4); }
size_t syn_smem(int nb, int lmax) { return (size_t)nb * 2 * (tab_rows(lmax, 0) + 1) * sizeof(float4); }

template <int NB, bool FINE>
void launch_tab(const LegArgs &a, const LegDfArgs &d, const LegBatchMaps &bm, cudaStream_t s, int mode) {
  const int nchunk = tab_chunks(a.lmax), ntile = (a.RP + 31) / 32;
  const int nw = std::min(8, ntile);
  const dim3 ga(a.lmax + 1, nchunk), gs(a.lmax + 1, (ntile + nw - 1) / nw);
  const size_t sa = ana_smem(NB, a.RP), ss = syn_smem(NB, a.lmax);
  auto ana = [&](auto kernel) {
    raise_smem_cap(reinterpret_cast<const void *>(kernel));
    launch_pdl(kernel, ga, kThreads, sa, s, a, d, bm);
  };
  auto syn = [&](auto kernel) {
    raise_smem_cap(reinterpret_cast<const void *>(kernel));
    launch_pdl(kernel, gs, 32 * nw, ss, s, a, d, bm, nchunk);
  };
  if (mode == LEG_SYNTH) syn(tab_synthesis_kernel<NB, false, FINE>);
  else if (mode == LEG_ANALYSIS) ana(tab_analysis_kernel<NB, false, FINE>);
  else {
    ana(tab_analysis_kernel<NB, true, FINE>);
    syn(tab_synthesis_kernel<NB, true, FINE>);
  }
}

}  // namespace

int tab_chunks(int lmax) { return (tab_rows(lmax, 0) + kTabRows - 1) / kTabRows; }

size_t leg_tab_smem(int lmax, int RP) { return std::max(ana_smem(1, RP), syn_smem(1, lmax)); }

void launch_legendre_tab(const LegArgs &a, const LegDfArgs &d, const LegBatchMaps &bm, int nb, cudaStream_t s,
                         int mode) {
  const bool fine = fine_steps(a.RP);
  if (nb == 1) fine ? launch_tab<1, true>(a, d, bm, s, mode) : launch_tab<1, false>(a, d, bm, s, mode);
  else fine ? launch_tab<2, true>(a, d, bm, s, mode) : launch_tab<2, false>(a, d, bm, s, mode);
}

}  // namespace wfk
