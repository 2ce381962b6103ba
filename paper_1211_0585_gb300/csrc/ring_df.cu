// Ring stage in double-float arithmetic (FP64-accurate FFTs on the FP32 pipe).
//
// Same algorithm and data flow as ring.cu (fold F_m onto residues with the
// half-pixel shift, inverse DFT, Eq. 3 per pixel with the chi^2 partials,
// forward DFT, unfold), but every FFT value is a pair of floats per real
// component and every butterfly is built from error-free transformations
// (two_sum, two_prod), because GB300's FP64 pipe is 1/63 of its FP32 pipe. So
// are the Fourier records on both sides, the fold, the unfold, the per-pixel
// Eq. 3 update and the chi^2 sums up to the warp's; the FP64 pipe sees the
// sums over warps and the gains of a new lambda. Tables (twiddles, half-shift, chirp, Bluestein
// filter) are stored as double-float pairs, converted once from the double
// tables when the plan is built.
#include <cuda_runtime.h>

#include "df.cuh"
#include "fft.cuh"
#include "fold.cuh"
#include "pdl.cuh"
#include "wf_internal.h"

namespace wfk {

namespace {

// complex double-float held as float4 (re.h, re.l, im.h, im.l)
__device__ __forceinline__ dfl RE(float4 v) { return {v.x, v.y}; }
__device__ __forceinline__ dfl IM(float4 v) { return {v.z, v.w}; }
__device__ __forceinline__ float4 cconj(float4 a) { return make_float4(a.x, a.y, -a.z, -a.w); }
__device__ __forceinline__ float4 cneg(float4 a) { return make_float4(-a.x, -a.y, -a.z, -a.w); }

// the compensated sum (S, C) over the warp's lanes, on every lane
__device__ __forceinline__ void warp_sum_df(float &S, float &C) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    comp_add(S, C, __shfl_xor_sync(0xffffffffu, S, o), __shfl_xor_sync(0xffffffffu, C, o));
}

}  // namespace

// One CTA per ring pair and map (grid.y: maps of one shape share the launch,
// since the pairs of one map leave a second wave of CTAs nearly empty below
// Nside 512: two maps 103 -> 89 us and three 205 -> 159 us at Nside 256, three
// transforms 40 -> 27 us at Nside 128): the two rings of a pair have the same length,
// half-pixel shift and tables, and real pixel values, so they share one
// complex transform (Sect. 2 basis change, both directions):
//   synthesis  IDFT(G_N + i G_S) = f_N + i f_S
//   analysis   Z = DFT(u_N + i u_S): U_N(q) = (Z_q + conj Z_{n-q}) / 2,
//                                    U_S(q) = (Z_q - conj Z_{n-q}) / (2 i)
// which halves the FFT work against one transform per ring. The equator is a
// pair of one ring (its south half stays zero). Eq. 3 runs in place on the
// inverse transform's output, which is the forward transform's input order.
// 256 threads and three CTAs per SM (up to 64 KB of FFT buffer each at Nside
// 512), so that one pair's barriers and global loads overlap another's work.
// With the records, the fold and the sums in double, the FP64 pipe was as busy
// as the FP32 one (37 %) and the kernel took 250 us at Nside 512, 65 us at 256;
// in double-float throughout 203 and 52 us, with the twiddles by stage
// (fft.cuh) 184 us at Nside 512.
constexpr int kRingDfThreads = 256;
template <int MODE, bool FINE>
__global__ void __launch_bounds__(kRingDfThreads, 3) ring_df_kernel(const RingArgs A, const RingDfArgs T,
                                                                     const __grid_constant__ RingMaps Maps) {
  using O = OpsDF<FINE>;
  extern __shared__ float4 rsm[];
  const RingMap &Q = Maps.m[blockIdx.y];
  const int2 pr = A.porder[A.first + blockIdx.x];  // (north ring, south ring or -1)
  const RingDev rg = A.rings[pr.x];
  const bool two = pr.y >= 0;
  const long long offS = two ? A.rings[pr.y].off : 0;
  const int n = rg.n;
  const int M = 1 << rg.logM;
  const int Mp = M;
  // [Mp] (swizzled, px): shared memory, or this CTA's part of the global scratch
  float4 *buf = A.scratch ? reinterpret_cast<float4 *>(A.scratch) + (size_t)blockIdx.x * M : rsm;
  __shared__ float2 red[kRingDfThreads / 32][4];
  __shared__ FoldPair fold_part[kRingDfThreads];

  if (M <= 512) {   // short rings: their tables into L1 while the kernel before ends (a miss each, one after another)
    auto touch = [&](const float4 *p, int bytes) {
      for (int i = threadIdx.x * 128; i < bytes; i += 128 * kRingDfThreads) {
        float x;
        asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(x) : "l"(reinterpret_cast<const char *>(p) + i));
      }
    };
    touch(T.tw, 16 * 3 * (M / 2 - 1));
    if (rg.shifted) touch(T.hs + rg.hs_off, 16 * n);
    if (rg.blue) {
      touch(T.chirp + rg.ch_off, 16 * n);
      touch(T.B + rg.B_off, 16 * M);
    }
  }
  pdl_wait();
  pdl_next();
  int L = A.lsht;
  double lam = 1.0;
  if (MODE != RING_ITER && Q.gate && Q.gate->done) return;
  if (MODE == RING_ITER) {
    if (Q.ctl->done) return;
    L = Q.ctl->lsht;
    lam = Q.ctl->lambda;
  }
  const float4 *hs = T.hs + rg.hs_off;
  const float4 *ch = T.chirp + rg.ch_off;
  const float4 *Bf = T.B + rg.B_off;
  const int k = rg.pair;

  if (MODE == RING_SYNTH || MODE == RING_ITER) {
    // Z = G_N + i G_S
    fold_ring2<FINE>(Q.FS, A.RP, k, rg.shifted, n, L, fold_part, [&](int q, float4 gN, float4 gS) {
      float4 acc = df_pair(df_add2<FINE>(RE(gN), df_neg(IM(gS))), df_add2<FINE>(IM(gN), RE(gS)));
      if (rg.shifted) acc = O::mul(acc, hs[q]);
      buf[px<O>(q)] = rg.blue ? O::mul(cconj(acc), ch[q]) : acc;
    });
    if (rg.blue) {
      for (int q = n + threadIdx.x; q < M; q += blockDim.x) buf[px<O>(q)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    if (rg.blue) bluestein4<O, 1>(buf, Mp, M, rg.logM, Bf, T.tw, A.logMmax);
    else fft_dif4<O, 1>(buf, Mp, M, rg.logM, +1, T.tw, A.logMmax);
  }
  // pixel p of both rings: z = f_N + i f_S at buf[loc(p)] (Bluestein: conj of ch[p] buf[p])
  auto loc = [&](int p) { return rg.blue ? px<O>(p) : px<O>(digitrev(p, rg.logM)); };
  auto pixel = [&](int p) {
    const float4 v = buf[loc(p)];
    return rg.blue ? cconj(O::mul(ch[p], v)) : v;
  };
  if (MODE == RING_SYNTH) {
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
      const float4 z = pixel(p);
      Q.map_out[rg.off + p] = df_to(RE(z));
      if (two) Q.map_out[offS + p] = df_to(IM(z));
    }
    return;
  }
  if (MODE == RING_ITER) {
    // Eq. 3 and the chi^2 partials in double-float (the FP64 pipe is 1/63 of the
    // FP32 one): compensated sums per thread and warp, the sum over warps in double
    float cs[4] = {0.f, 0.f, 0.f, 0.f}, cc[4] = {0.f, 0.f, 0.f, 0.f};   // north chi2, chi2_lambda, south
    const bool fresh = Q.gainlam[pr.x] == lam;   // gains of this pair already at this lambda
    const dfl ltd = df_from(lam * Q.tau);
    const double l1t = (lam - 1.0) * Q.tau;
    auto update = [&](long long at, dfl s, int half) {  // Eq. 3, returns u
      const float2 d2 = Q.d[at], w2 = Q.w[at];
      const dfl dv{d2.x, d2.y}, wv{w2.x, w2.y};
      dfl g;
      if (fresh) {
        const float2 g2 = Q.gain[at];
        g = dfl{g2.x, g2.y};
      } else {  // the first pass at a new lambda: the gain from w in double
        const double w = Q.w64[at];
        g = df_from(w / (1.0 + l1t * w));
        Q.gain[at] = make_float2(g.h, g.l);
      }
      const dfl res = df_add(dv, df_neg(s));
      const dfl r2 = df_mul(res, res);
      dot2_acc<true>(cs[2 * half], cc[2 * half], wv, r2);
      dot2_acc<true>(cs[2 * half + 1], cc[2 * half + 1], g, r2);
      return df_mul(df_mul(ltd, g), res);
    };
    for (int p = threadIdx.x; p < n; p += blockDim.x) {
      const float4 z = pixel(p);
      const dfl uN = update(rg.off + p, RE(z), 0);
      const dfl uS = two ? update(offS + p, IM(z), 1) : dfl{0.f, 0.f};
      const float4 u = df_pair(uN, uS);
      buf[loc(p)] = rg.blue ? O::mul(u, ch[p]) : u;
    }
    if (rg.blue) {
      for (int q = n + threadIdx.x; q < M; q += blockDim.x) buf[px<O>(q)] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    {
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        warp_sum_df(cs[i], cc[i]);
        if (lane == 0) red[warp][i] = make_float2(cs[i], cc[i]);
      }
      __syncthreads();   // also orders the pixel pass before the forward transform
      if (threadIdx.x < (two ? 4 : 2)) {
        double v = 0.0;
        for (int w = 0; w < kRingDfThreads / 32; ++w) {
          const float2 r = red[w][threadIdx.x];
          v += (double)r.x + (double)r.y;
        }
        Q.ring_part[2 * (threadIdx.x < 2 ? pr.x : pr.y) + (threadIdx.x & 1)] = v;
      }
      if (threadIdx.x == 0 && !fresh) {  // after the barrier: every gain of the pair is written
        Q.gainlam[pr.x] = lam;
        if (two) Q.gainlam[pr.y] = lam;
      }
    }
  } else {  // RING_ANALYSIS: u = the input maps
    for (int p = threadIdx.x; p < M; p += blockDim.x) {
      if (p < n) {
        const float4 u = df_pair(df_from(Q.map_in[rg.off + p]), df_from(two ? Q.map_in[offS + p] : 0.0));
        buf[loc(p)] = rg.blue ? O::mul(u, ch[p]) : u;
      } else if (rg.blue) {
        buf[px<O>(p)] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    __syncthreads();
  }

  if (rg.blue) bluestein4<O, 1>(buf, Mp, M, rg.logM, Bf, T.tw, A.logMmax);
  else fft_dit4<O, 1>(buf, Mp, M, rg.logM, -1, T.tw, A.logMmax);
  for (int m = threadIdx.x; m <= L; m += blockDim.x) {
    const int q = m % n, j = m / n, qn = q ? n - q : 0;
    const float4 Zq = rg.blue ? O::mul(ch[q], buf[px<O>(q)]) : buf[px<O>(q)];
    const float4 Zn = rg.blue ? O::mul(ch[qn], buf[px<O>(qn)]) : buf[px<O>(qn)];
    // U_N = (Z_q + conj Z_{n-q}) / 2, U_S = (Z_q - conj Z_{n-q}) / (2 i); the records hold 2 U times a power of two
    // next to Omega / 2, and the analysis' sums are multiplied by the rest in double: a rounding less than here
    auto add = [](dfl x, dfl y) { return FINE ? df_add2<true>(x, y) : df_add(x, y); };
    float4 UN = df_pair(add(RE(Zq), RE(Zn)), add(IM(Zq), df_neg(IM(Zn))));
    float4 US = df_pair(add(IM(Zq), IM(Zn)), add(RE(Zn), df_neg(RE(Zq))));
    if (rg.shifted) {
      UN = O::mul(UN, cconj(hs[q]));
      US = O::mul(US, cconj(hs[q]));
      if (j & 1) { UN = cneg(UN); US = cneg(US); }
    }
    auto put = [&](dfl v) { return df_pack(dfl{A.fscale * v.h, A.fscale * v.l}); };
    Q.FT[(size_t)m * A.RP + k] =
        make_double4_32a(put(RE(UN)), put(IM(UN)), two ? put(RE(US)) : 0.0, two ? put(IM(US)) : 0.0);
  }
}

// double -> double-float (hi, lo) per element
__global__ void to_df2_kernel(const double *src, float2 *dst, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const dfl v = df_from(src[i]);
    dst[i] = make_float2(v.h, v.l);
  }
}

void launch_to_df2(const double *src, float2 *dst, long long n, cudaStream_t s) {
  if (n <= 0) return;
  long long blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  to_df2_kernel<<<(int)blocks, 256, 0, s>>>(src, dst, n);
}

// double -> double-float table conversion
__global__ void to_df_kernel(const double2 *src, float4 *dst, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = src[i];
    dst[i] = df_pair(df_from(v.x), df_from(v.y));
  }
}

void launch_to_df(const double2 *src, float4 *dst, long long n, cudaStream_t s) {
  if (n <= 0) return;
  long long blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  to_df_kernel<<<(int)blocks, 256, 0, s>>>(src, dst, n);
}

__global__ void pack_twiddles_kernel(const double2 *tw, int logMmax, float4 *df, float2 *f32) {
  const int id = blockIdx.x * blockDim.x + threadIdx.x;
  auto get = [&](int s, int i, int c) {   // e^{-2 pi i (i c) / 2^s}; sizes above the longest only at i = 0
    const double2 v = tw[s <= logMmax ? (i * c) << (logMmax - s) : 0];
    return df_pair(df_from(v.x), df_from(v.y));
  };
  if (df && id < (1 << logMmax) / 2 - 1) {            // (s, i) at 2^(s-2) - 1 + i
    const int qsh = 31 - __clz(id + 1), Q = 1 << qsh, i = id + 1 - Q;
    for (int c = 1; c < 4; ++c) df[3 * (Q - 1) + (c - 1) * Q + i] = get(qsh + 2, i, c);
  }
  if (f32 && id < (1 << (logMmax < 4 ? 4 : logMmax)) / 8 - 1) {
    const int qsh = 31 - __clz(id + 1), Q = 1 << qsh, i = id + 1 - Q;
    for (int c = 1; c < 4; ++c) {
      const float4 a = get(qsh + 4, i, c), b = get(qsh + 2, i, c);
      f32[6 * (Q - 1) + (c - 1) * Q + i] = make_float2(a.x, a.z);
      f32[6 * (Q - 1) + (2 + c) * Q + i] = make_float2(b.x, b.z);
    }
  }
}

void launch_pack_twiddles(const double2 *tw, int logMmax, float4 *df, float2 *f32, cudaStream_t s) {
  const int n = 1 << (logMmax < 4 ? 4 : logMmax);
  pack_twiddles_kernel<<<(n + 255) / 256, 256, 0, s>>>(tw, logMmax, df, f32);
}

template <int MODE, bool FINE>
static void launch_ring_df_form(const RingArgs *a, const RingDfArgs *t, int nmaps, const RingClass *cls, int ncls,
                                cudaStream_t s) {
  auto smem = [](const RingClass &c) { return c.global ? (size_t)16 : ((size_t)1 << c.logM) * sizeof(float4); };
  raise_smem_cap(reinterpret_cast<const void *>(ring_df_kernel<MODE, FINE>));
  for (int c = 0; c < ncls; ++c) {
    if (cls[c].count <= 0) continue;
    const size_t sm = smem(cls[c]);
    RingArgs ac = a[0];
    ac.first = cls[c].first;
    ac.scratch = cls[c].global ? a[0].scratch : nullptr;
    const int most = cls[c].global ? 1 : kRingMapsMax;   // the scratch array holds one map's rings
    for (int i0 = 0; i0 < nmaps; i0 += most) {
      const int n = nmaps - i0 < most ? nmaps - i0 : most;
      RingMaps q{};
      for (int i = 0; i < n; ++i) {
        const RingArgs &x = a[i0 + i];
        const RingDfArgs &y = t[i0 + i];
        q.m[i] = RingMap{x.FS, x.FT, x.map_in, x.map_out, y.d, y.w, x.w, y.gain, y.gainlam, x.ring_part, x.ctl,
                         x.gate, x.tau};
      }
      launch_pdl(ring_df_kernel<MODE, FINE>, dim3(cls[c].count, n), kRingDfThreads, sm, s, ac, t[0], q);
    }
  }
}

template <int MODE>
static void launch_ring_df_mode(const RingArgs *a, const RingDfArgs *t, int nmaps, const RingClass *cls, int ncls,
                                cudaStream_t s) {
  if (fine_steps(a[0].RP)) launch_ring_df_form<MODE, true>(a, t, nmaps, cls, ncls, s);
  else launch_ring_df_form<MODE, false>(a, t, nmaps, cls, ncls, s);
}

void launch_ring_df(const RingArgs *a, const RingDfArgs *t, int nmaps, const RingClass *cls, int ncls,
                    cudaStream_t s, int mode) {
  switch (mode) {
    case RING_SYNTH: launch_ring_df_mode<RING_SYNTH>(a, t, nmaps, cls, ncls, s); break;
    case RING_ANALYSIS: launch_ring_df_mode<RING_ANALYSIS>(a, t, nmaps, cls, ncls, s); break;
    default: launch_ring_df_mode<RING_ITER>(a, t, nmaps, cls, ncls, s); break;
  }
}

}  // namespace wfk
